// Internal definitions shared by the library's translation units: job state,
// per-point and per-trial payloads of the three fold modes, the folds
// themselves (Eq. 3 of arXiv:2006.06866) and the fixed-point entropy table
// (Eq. 4).  Nothing here is part of the C ABI.
#pragma once

#include <cstddef>
#include <cstdint>
#include <cuda_runtime.h>

#include "../../include/gce.h"

namespace gce {

// ------------------------------------------------------------------ job state

// Device-side state of one call: reductions of the scan kernel, input-check
// flags and the persistent kernel's work counter.  Zeroed (pmin set to +inf)
// by k_init at the start of every call.
struct JobState {
    unsigned long long tau_max_bits;    // max |t - t0| as binary64 bits
    unsigned long long pmin_bits;       // min period as binary64 bits
    unsigned long long pdot_max_bits;   // max |Pdot| as binary64 bits
    unsigned long long work;            // next work item (persistent kernel)
    // (err, wide and epoch in one 16-byte load: a load of its own for each puts half a
    // microsecond more before the first work of a small call's kernels)
    unsigned int err;                   // ERR_* bits
    // FP64 and FIXED32 jobs prepared for the coarse fold: 1 when the job's range is
    // beyond it, so that the mode's own fold runs on every point (set by k_trials,
    // read by the kernels after it)
    unsigned int wide;
    unsigned int epoch;                 // 1 when some point has tau = 0
    unsigned int pad;
};
static_assert(offsetof(JobState, err) == 32 && sizeof(JobState) == 48, "job_flags' layout");
// {err, wide, epoch, 0}; the state's buffer is aligned
__device__ __forceinline__ uint4 job_flags(const JobState *st) {
    return *reinterpret_cast<const uint4 *>(&st->err);
}

enum : unsigned int {
    ERR_TIME = 1u,      // non-finite time or magnitude
    ERR_PERIOD = 2u,    // non-finite or non-positive period
    ERR_PDOT = 4u,      // non-finite period derivative
    ERR_RANGE = 8u,     // trial range beyond what the chosen fold represents
    ERR_BAND = 16u,     // filter index outside [0, n_bands)
    ERR_SLOT = 32u,     // checked builds only: a counter slot outside the trial's kept range
};

// The CE kernel's modes of GCE_PHASE_FP64 and GCE_PHASE_FIXED32 jobs (not part of
// the ABI): a coarser fixed-point fold with every point's distance to the phase-bin
// edges checked against the folds' error bounds, and the mode's own fold for the
// points within them.
enum { kJobFp64 = 3, kJobFixed32 = 4 };
__host__ __device__ constexpr bool coarse_mode(int mode) {
    return mode == kJobFp64 || mode == kJobFixed32;
}

// Whether a job's maxima lie inside the FIXED32 fold's range: F < 2^63, and the
// Pdot cross term small enough for its FP32 path.
__host__ __device__ inline bool fixed_range_ok(double fmax, double amax, int e_tau) {
    return !(ldexp(fmax, e_tau) >= 536870912.0 || ldexp(amax, 2 * e_tau) >= 262144.0);
}

// Fixed-point scaling of the FIXED32 fold, derived from the job's maxima.
// tau_max < 2^e_tau.  T = tau 2^s (|T| < 2^62), F = f 2^r with s + r = 96, so
// T F / 2^64 = tau f 2^32; U = tau^2 2^u (U < 2^62), A = a 2^v with
// u + v = 96, so U A / 2^64 = a tau^2 2^32.
struct FixedScale {
    int e_tau;
    int s, r, u, v;
};

__host__ __device__ inline FixedScale fixed_scale_from(double tau_max) {
    FixedScale fs;
    int e = 0;
    if (tau_max > 0.0) {
        int ex;
        frexp(tau_max, &ex);   // tau_max = m 2^ex, m in [0.5, 1)  =>  tau_max < 2^ex
        e = ex;
    }
    fs.e_tau = e;
    fs.s = 62 - e;
    fs.r = 96 - fs.s;
    fs.u = 62 - 2 * e;
    fs.v = 96 - fs.u;
    return fs;
}

// ------------------------------------------------------------------ payloads

// Per point, sorted by magnitude bin, in the layout of the fold mode.
//   FP64:    double tau                                        (8 bytes)
//   SPLIT32: float4 {tau_hi, tau_lo, tau2_hi, tau2_lo}          (16 bytes)
//   FIXED32: uint4  {T1 (int32), t0f, U1, u0f}                  (16 bytes)
//            T = tau 2^s = T1 2^32 + T0; U = tau^2 2^u = U1 2^32 + U0 (U0
//            balanced); t0f, u0f are the bit patterns of the floats
//            2^23 + (T0 >> 9) and 2^23 + ((U0 + 2^31) >> 9).
// Per flat trial:
//   FP64:    double2 {f, a}
//   SPLIT32: float4  {f_hi, f_lo, a_hi, a_lo}
//   FIXED32: FixedTrial, see fold_fixed.
struct FixedTrial {
    uint4 i;   // {F1, F0 (int32, balanced), A1 (int32), A0}: F = f 2^r, A = -a 2^v
    float4 f;  // {G0, G2, K, k as bits}: the FP32 cross terms' scales and offset
};
template <int MODE> struct ModeTraits;
// half_t: the first two words of a point, all a fold without a Pdot term reads
// (SPLIT32 {tau_hi, tau_lo}, FIXED32 {T1, t0f}); FP64 points are one word.
template <> struct ModeTraits<GCE_PHASE_FP64> {
    typedef double point_t;
    typedef double half_t;
    typedef double2 trial_t;
    __device__ static point_t widen(half_t h) { return h; }
};
template <> struct ModeTraits<GCE_PHASE_SPLIT32> {
    typedef float4 point_t;
    typedef float2 half_t;
    typedef float4 trial_t;
    __device__ static point_t widen(half_t h) { return make_float4(h.x, h.y, 0.0f, 0.0f); }
};
template <> struct ModeTraits<GCE_PHASE_FIXED32> {
    typedef uint4 point_t;
    typedef uint2 half_t;
    typedef FixedTrial trial_t;
    __device__ static point_t widen(half_t h) { return make_uint4(h.x, h.y, 0u, 0u); }
};

// The coarse fold's points and trials (see coarse_margin); the binary64 tau of each
// point is kept beside them (MainArgs::tau) for the points near an edge.
struct CoarsePoint {
    unsigned int T1;
    float T1f, b;
    unsigned int U1;
    float U1f, ub;
};
struct __align__(16) CoarseTrial {
    unsigned int F1;
    float F0, F1f;
    unsigned int A1;
    float A0, A1f;
    unsigned int margin;
    unsigned int zero;  // FIXED32 jobs: its own fold's phase at tau = 0 (FP64's is 0)
};
// A segment word of a coarse job: the segment's start (below 2^16), and in the high half
// how many of its points have tau = 0.  Those come last in the segment.  They lie on an
// edge in every trial, so the coarse fold could decide them in none; but a trial puts all
// of them in one bin (zero), which is counted once per segment.  (300 curves x 600 points
// x 2e4 periods, FIXED32, every curve with a point at t0: 4.74 ms with the undecided
// points' walk, lane after lane, 1.87 with the lanes together.)
__host__ __device__ inline unsigned int segment_word(int start, int zeros) {
    return (unsigned int)start | (unsigned int)zeros << 16;
}
__host__ __device__ inline int segment_start(unsigned int w) { return (int)(w & 0xffffu); }
__host__ __device__ inline int segment_zeros(unsigned int w) { return (int)(w >> 16); }
template <> struct ModeTraits<kJobFp64> {
    typedef CoarsePoint point_t;
    typedef CoarsePoint half_t;
    typedef CoarseTrial trial_t;
};
template <> struct ModeTraits<kJobFixed32> : ModeTraits<kJobFp64> {};

// Balanced split of a 64-bit value: x = hi 2^32 + lo with lo a signed 32-bit
// value in [-2^31, 2^31), so that signed multiply-high works on it.
__host__ __device__ inline void split_balanced(long long x, int *hi, int *lo) {
    long long h = x >> 32;  // arithmetic
    unsigned int l = (unsigned int)(x & 0xffffffffll);
    if (l >= 0x80000000u) h += 1;
    *hi = (int)h;
    *lo = (int)l;  // two's complement reinterpretation: l - 2^32 when l >= 2^31
}

// ------------------------------------------------------------------ folds

// Eq. 3 in binary64 with the pinned operation sequence (see gce.h); returns the
// phase bin.  With pdot == false, a is known to be +-0 and x = s exactly.  The
// period part s = tau f is split out so that trials sharing the period can
// share it (fold_fp64_from completes the fold from it).
__device__ __forceinline__ double fold_fp64_fpart(double tau, double f) { return __dmul_rn(tau, f); }

template <bool PDOT>
__device__ __forceinline__ int fold_fp64_from(double s, double tau, double a, double nphi,
                                              int n_phase) {
    double x = s;
    if (PDOT) {
        double b = __dmul_rn(a, tau);
        x = __fma_rn(-b, tau, s);
    }
    double phi = __dsub_rn(x, floor(x));
    int j = __double2int_rd(__dmul_rn(phi, nphi));
    return min(j, n_phase - 1);
}

template <bool PDOT>
__device__ __forceinline__ int fold_fp64(double tau, double f, double a, double nphi,
                                         int n_phase) {
    return fold_fp64_from<PDOT>(fold_fp64_fpart(tau, f), tau, a, nphi, n_phase);
}

// Eq. 3 in FP32 double-float.  tau = th + tl and f = fh + fl (float pairs),
// tau^2 = t2h + t2l and a = ah + al with the a pair stored negated.  The
// integer cycles of th fh are removed by an FMA against the rounding constant
// M = 1.5 2^23: t = fma(th, fh, M) holds rint(th fh) + M (|th fh| < 2^21 cycles,
// checked per job), and r = fma(th, fh, -(t - M)) is the exact product minus
// that integer, rounded once (|r| <= 1/2).  The cross terms tl fh and th fl
// (tl fl is below 2^-48 relative) are added by FMA.  The Pdot term -a tau^2 is
// reduced the same way and the sum reduced once more.  x then lies in
// (-1, 1), and one round-down FMA against the same constant gives
// n_phase + floor(x n_phase) in [0, 2 n_phase): the returned slot, where slots
// j and j + n_phase both stand for phase bin j (so no modulo is needed here).
// Phase error about 1e-7 cycles (a few 2^-25 roundings).
constexpr float kRound = 12582912.0f;  // 1.5 * 2^23

// The period part of the fold, shared by trials of the same period: th fh with
// its integer cycles removed, plus the cross terms (the whole residual x when
// Pdot = 0).
__device__ __forceinline__ float fold_split_fpart(float4 pt, float4 tr) {
    const float th = pt.x, tl = pt.y;
    const float fh = tr.x, fl = tr.y;
    const float t = __fmaf_rn(th, fh, kRound);
    const float r = __fmaf_rn(th, fh, __fsub_rn(kRound, t));
    return __fmaf_rn(th, fl, __fmaf_rn(tl, fh, r));
}

// The rest of the fold from the period part c: the Pdot term -a tau^2 reduced
// the same way, the sum reduced once more, then the slot.  REDUCE (without
// Pdot): the residual is reduced once more as well, to |x| <= 1/2, for folds that
// must stay in the narrow slot range (see slot_range).
template <bool PDOT, bool REDUCE = false>
__device__ __forceinline__ int fold_split_from(float c, float4 pt, float4 tr, float nphi,
                                               float zoff) {
    float x = c;
    if (!PDOT && REDUCE) x = __fsub_rn(c, __fsub_rn(__fadd_rn(c, kRound), kRound));
    if (PDOT) {
        const float t2h = pt.z, t2l = pt.w;
        const float nah = tr.z, nal = tr.w;  // -a split
        const float t2 = __fmaf_rn(nah, t2h, kRound);
        const float r2 = __fmaf_rn(nah, t2h, __fsub_rn(kRound, t2));
        c = __fmaf_rn(nah, t2l, c);
        c = __fmaf_rn(nal, t2h, c);
        const float y = __fadd_rn(c, r2);
        x = __fsub_rn(y, __fsub_rn(__fadd_rn(y, kRound), kRound));
    }
    const float z = __fmaf_rd(x, nphi, zoff);  // zoff = 1.5 2^23 + n_phase
    return __float_as_int(z) - __float_as_int(kRound);
}

template <bool PDOT>
__device__ __forceinline__ int fold_split(float4 pt, float4 tr, float nphi, float zoff) {
    return fold_split_from<PDOT>(fold_split_fpart(pt, tr), pt, tr, nphi, zoff);
}

// Two points of one trial at once (fma.rn.f32x2: each half is the scalar
// operation, rounded alone, so the slots are those of fold_split).  The CE
// kernel's hot loop is bound by instruction issue, and a packed instruction
// takes one issue slot for two FMAs; the pairing is over points and not over
// trials because the staged points can be laid out as pairs once per curve
// (no register moves in the loop), where a trial pair would need every point
// value duplicated.
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pack2(float a, float b) {
    f32x2 d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(a), "f"(b));
    return d;
}
__device__ __forceinline__ f32x2 dup2(float a) { return pack2(a, a); }
__device__ __forceinline__ void unpack2(f32x2 v, float &a, float &b) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ float lo2(f32x2 v) {
    float a, b;
    unpack2(v, a, b);
    return a;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
    f32x2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ f32x2 fma2_rd(f32x2 a, f32x2 b, f32x2 c) {
    f32x2 d;
    asm("fma.rm.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
    f32x2 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

// A SPLIT32 trial in the registers of the packed fold: every constant twice.
struct SplitPrep {
    f32x2 fh, fl, nah, nal;
};
__device__ __forceinline__ SplitPrep split_prep(float4 t) {
    return SplitPrep{dup2(t.x), dup2(t.y), dup2(t.z), dup2(t.w)};
}
__device__ __forceinline__ float4 split_trial(const SplitPrep &t) {
    return make_float4(lo2(t.fh), lo2(t.fl), lo2(t.nah), lo2(t.nal));
}
// Two points: {tau_hi, tau_hi'}, {tau_lo, tau_lo'} and the same of tau^2.
struct SplitPair {
    f32x2 th, tl, t2h, t2l;
};

// fold_split_fpart of two points (a - b is written fma(b, -1, a): exact the
// same value, and no negated operand is needed).
__device__ __forceinline__ f32x2 fold_split_fpart2(const SplitPair &p, const SplitPrep &tr) {
    const f32x2 m = dup2(kRound), neg = dup2(-1.0f);
    const f32x2 t = fma2(p.th, tr.fh, m);
    const f32x2 r = fma2(p.th, tr.fh, fma2(t, neg, m));
    return fma2(p.th, tr.fl, fma2(p.tl, tr.fh, r));
}

// fold_split_from of two points; returns the bit patterns of the two rounding
// FMAs (slot + bits of kRound).
template <bool PDOT, bool REDUCE>
__device__ __forceinline__ void fold_split_from2(f32x2 c, const SplitPair &p, const SplitPrep &tr,
                                                 float nphi, float zoff, unsigned int &z0,
                                                 unsigned int &z1) {
    const f32x2 m = dup2(kRound), nm = dup2(-kRound), neg = dup2(-1.0f);
    f32x2 x = c;
    if (PDOT) {
        const f32x2 t2 = fma2(tr.nah, p.t2h, m);
        const f32x2 r2 = fma2(tr.nah, p.t2h, fma2(t2, neg, m));
        c = fma2(tr.nah, p.t2l, c);
        c = fma2(tr.nal, p.t2h, c);
        x = add2(c, r2);
    }
    if (PDOT || REDUCE) x = fma2(add2(add2(x, m), nm), neg, x);
    float a, b;
    unpack2(fma2_rd(x, dup2(nphi), dup2(zoff)), a, b);
    z0 = __float_as_uint(a);
    z1 = __float_as_uint(b);
}

// Eq. 3 in 32-bit-limb fixed point, the phase in units of 2^-32 cycles so that
// the integer cycles wrap out of a 32-bit word.  With T = T1 2^32 + T0 and
// F = F1 2^32 + F0, bits 64..95 of T F are
//   lo32(T1 F1) + hi32(T1 F0) + T0 F1 / 2^32            (+ dropped carries).
// The first two are exact integer products (IMAD, IMAD.HI).  The third is
// below g1 = F1 units and is computed on the FP32 pipe: t0f = 2^23 + (T0 >> 9)
// times G0 = F1 2^(-23-k), added to an offset K that removes the 2^23 G0
// term and carries the 1.5 2^23 rounding constant, so the FMA result's bit
// pattern holds the term rounded to 2^k units (k per trial, the smallest with
// F1 < 2^(22+k)); it joins the accumulator shifted left by k, and the integer
// offset C = -(bits(1.5 2^23) << k) cancels the constant's bits.  The Pdot term
// -a tau^2 is the same construction for U and A = -a 2^v: lo32(U1 A1) and
// hi32(A0 U1) exact, hi32(A1 U0) through u0f and G2 in the same FMA chain.
// Error: dropped carries (-1..+2 units), T0 >> 9 truncation (<= F1 2^-23),
// FP32 roundings (<= 3 2^(k-1)), so a few 2^-32 cycles for k <= 2.
// The phase bin is floor(phase n_phase / 2^32) = hi32(phase n_phase).
__device__ __forceinline__ unsigned int mad_lo_u32(unsigned int a, unsigned int b,
                                                   unsigned int c) {
    unsigned int d;
    asm("mad.lo.u32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
    return d;
}
__device__ __forceinline__ unsigned int mad_hi_s32(int a, int b, unsigned int c) {
    int d;
    asm("mad.hi.s32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"((int)c));
    return (unsigned int)d;
}
__device__ __forceinline__ unsigned int mad_hi_u32(unsigned int a, unsigned int b,
                                                   unsigned int c) {
    unsigned int d;
    asm("mad.hi.u32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
    return d;
}

// Per-trial values of the FIXED32 fold that stay in registers.
struct FixedPrep {
    unsigned int F1, A1, A0, C, k;
    int F0;
    float G0, G2, K;
};

__device__ __forceinline__ FixedPrep fixed_prep(const FixedTrial &t) {
    FixedPrep p;
    p.F1 = t.i.x;
    p.F0 = (int)t.i.y;
    p.A1 = t.i.z;
    p.A0 = t.i.w;
    p.G0 = t.f.x;
    p.G2 = t.f.y;
    p.K = t.f.z;
    p.k = __float_as_uint(t.f.w);
    p.C = 0u - (0x4B400000u << p.k);
    return p;
}

// The period part of the fixed-point fold, shared by trials of the same period:
// the exact integer products of T and F, with the offset C.
__device__ __forceinline__ unsigned int fold_fixed_fpart(uint4 pt, const FixedPrep &t) {
    const int T1 = (int)pt.x;
    const unsigned int acc = mad_lo_u32((unsigned int)T1, t.F1, t.C);
    return mad_hi_s32(T1, t.F0, acc);
}

// The rest of the fold from the period part acc: the Pdot products, the FP32
// cross terms and, for the bin, the multiply-high by n_phase.  K0: the shift
// by k is zero (every trial of the tile has F1 < 2^22).
template <bool PDOT, bool K0>
__device__ __forceinline__ unsigned int fold_fixed_phase_from(unsigned int acc, uint4 pt,
                                                              const FixedPrep &t) {
    float zin = t.K;
    if (PDOT) {
        const unsigned int U1 = pt.z;
        acc = mad_lo_u32(U1, t.A1, acc);
        acc = mad_hi_u32(t.A0, U1, acc);
        zin = __fmaf_rn(__uint_as_float(pt.w), t.G2, zin);
    }
    const unsigned int zb = __float_as_uint(__fmaf_rn(__uint_as_float(pt.y), t.G0, zin));
    return acc + (K0 ? zb : __funnelshift_l(0u, zb, t.k));
}

template <bool PDOT>
__device__ __forceinline__ int fold_fixed(uint4 pt, const FixedPrep &t, unsigned int n_phase) {
    return (int)__umulhi(fold_fixed_phase_from<PDOT, false>(fold_fixed_fpart(pt, t), pt, t),
                         n_phase);
}

template <bool PDOT, bool K0>
__device__ __forceinline__ unsigned int fold_fixed_bin_from(unsigned int acc, uint4 pt,
                                                            const FixedPrep &t,
                                                            unsigned int n_phase) {
    return __umulhi(fold_fixed_phase_from<PDOT, K0>(acc, pt, t), n_phase);
}

// x 2^e as ldexp rounds it: one multiplication where 2^e is a normal number.
__device__ __forceinline__ double scale2(double x, int e) {
    if (e < -1022 || e > 1023) return ldexp(x, e);
    return __dmul_rn(x, __longlong_as_double((long long)(e + 1023) << 52));
}

// A point and a trial in the FIXED32 formats (the preparation of plain and
// out-of-range jobs, and the CE kernel for the points the coarse fold leaves to it).
__device__ inline uint4 fixed_point(double tau, const FixedScale &fs) {
    // T = round(tau 2^s), |T| < 2^62; U = floor(T^2 / 2^62) = tau^2 2^u computed
    // exactly from T in 128-bit integer arithmetic.
    const long long T = __double2ll_rn(scale2(tau, fs.s));
    const unsigned long long aT = (unsigned long long)(T < 0 ? -T : T);
    const unsigned long long hi = __umul64hi(aT, aT), lw = aT * aT;
    const long long U = (long long)((hi << 2) | (lw >> 62));
    int u1, u0;
    split_balanced(U, &u1, &u0);
    const unsigned int t0 = (unsigned int)(T & 0xffffffffll);
    return make_uint4((unsigned int)(int)(T >> 32), 0x4B000000u | (t0 >> 9),  // 2^23 + (T0 >> 9)
                      (unsigned int)u1,
                      0x4B000000u | (((unsigned int)u0 ^ 0x80000000u) >> 9));  // 2^23 + ((U0+2^31) >> 9)
}
__device__ inline FixedTrial fixed_trial(double f, double aa, const FixedScale &fs) {
    FixedTrial v;
    // Out-of-range values are flagged by the range check; clamp so the conversions stay defined.
    const double F = fmin(scale2(f, fs.r), 9.2e18);
    int f1, f0;
    split_balanced(__double2ll_rn(F), &f1, &f0);
    long long an = 0;
    if (aa != 0.0) an = -__double2ll_rn(fmax(fmin(scale2(aa, fs.v), 9.2e18), -9.2e18));
    const int a1 = (int)(an >> 32);
    const unsigned int a0 = (unsigned int)(an & 0xffffffffll);
    // k: the smallest shift with F1 < 2^(22+k)
    const unsigned int uf1 = (unsigned int)f1;
    const int bits = 32 - __clz(uf1);
    const int k = bits > 22 ? bits - 22 : 0;
    const float scale = __uint_as_float((unsigned int)(104 - k) << 23);  // 2^(-23-k)
    const float g0 = __uint2float_rn(uf1) * scale;
    const float g2 = __int2float_rn(a1) * scale;
    // rounded once: the binary64 terms are exact, and so is 2^23 g0
    float kk = __fsub_rn(12582912.0f, 8388608.0f * g0);
    if (a1 != 0)
        kk = __double2float_rn(12582912.0 - 8388608.0 * (double)g0 - 8388608.0 * (double)g2 -
                               scale2((double)a1, -1 - k));
    v.i = make_uint4(uf1, (unsigned int)f0, (unsigned int)a1, a0);
    v.f = make_float4(g0, g2, kk, __uint_as_float((unsigned int)k));
    return v;
}

// The coarse fold (FP64 and FIXED32 jobs).  FIXED32's construction with fewer integer
// multiplies: with T = tau 2^(58-e) = T1 2^32 + T0 and F = f 2^(38+e) = F1 2^32 + F0,
// both balanced, the phase in units of 2^-32 cycles is
//   lo32(T1 F1) + (T1 F0 + T0 F1) / 2^32   (+ T0 F0 / 2^64),
// the first an exact integer product, the rest two FP32 FMAs into 1.5 2^29, whose
// result's bit pattern counts 64 units per step and joins by one shift-add.  -a tau^2
// is the same with U = tau^2 2^(58-2e) and A = -a 2^(38+2e).  The high-half multiplies
// that bound FIXED32 (a quarter of the FMA rate) are left only in the bin.
//   Range: cycles < 2^21 (F1 < 2^28) and Pdot cycles < 2^18 (A1 < 2^26), so that the
//   FMA results stay within 2^28 of the constant.
//   Error, in units: T1 and F0 as floats 2, T0 and F1 8, two FMA roundings 64, the
//   dropped product and the limbs' own rounding 1: 75; with Pdot U1 and A0 2, U0 and
//   A1 2, two more roundings 64, dropped and rounded 1: 69 more.
//   The mode's own fold: binary64 2^-53 (2 cycles + 2 Pdot cycles + 3) of a cycle: 3;
//   FIXED32 5 + 5 2^k (its limbs, floors, truncations and roundings), and |A1| / 4 +
//   2^k more where its two FP32 terms could carry the sum past 2^24 (its A1).
// coarse_margin is 5/4 of the sum and 8.  With w = (phase + margin) n_phase, the bin
// is hi32(w), and it is the own fold's too unless lo32(w) < 2 margin n_phase.
constexpr float kCoarseRound = 805306368.0f;  // 1.5 2^29
constexpr unsigned int kCoarseOffset = 0u - (0x4E400000u << 6);  // cancels its bits
__device__ inline CoarsePoint coarse_point(double tau, int e) {
    CoarsePoint p;
    int hi, lo;
    const long long T = __double2ll_rn(scale2(tau, 58 - e));
    split_balanced(T, &hi, &lo);
    p.T1 = (unsigned int)hi;
    p.T1f = (float)hi;
    p.b = (float)lo * 2.3283064365386963e-10f;  // 2^-32
    // U = floor(T^2 / 2^58) in integers: tau^2 itself may be beyond binary64's range
    const unsigned long long aT = (unsigned long long)(T < 0 ? -T : T);
    split_balanced((long long)((__umul64hi(aT, aT) << 6) | ((aT * aT) >> 58)), &hi, &lo);
    p.U1 = (unsigned int)hi;
    p.U1f = (float)hi;
    p.ub = (float)lo * 2.3283064365386963e-10f;
    return p;
}
__device__ inline CoarseTrial coarse_trial(double f, double aa, const FixedScale &fs, bool own_fixed,
                                           bool epoch) {
    CoarseTrial t;
    const int e = fs.e_tau;
    int hi, lo;
    split_balanced(__double2ll_rn(scale2(f, 38 + e)), &hi, &lo);
    t.F1 = (unsigned int)hi;
    t.F1f = (float)hi;
    t.F0 = (float)lo * 2.3283064365386963e-10f;
    hi = lo = 0;
    if (aa != 0.0) split_balanced(-__double2ll_rn(scale2(aa, 38 + 2 * e)), &hi, &lo);
    t.A1 = (unsigned int)hi;
    t.A1f = (float)hi;
    t.A0 = (float)lo * 2.3283064365386963e-10f;
    unsigned int err = 75u + (aa != 0.0 ? 69u : 0u) + 3u;
    if (own_fixed) {
        // FIXED32's F1 and A1 are these over 16
        const unsigned int f1 = (t.F1 >> 4) + 1u;
        const unsigned int a1 = (unsigned int)((hi < 0 ? -hi : hi) >> 4) + 1u;
        const int bits = 32 - __clz(f1);
        const unsigned int k = bits > 22 ? (unsigned int)bits - 22u : 0u;
        err += 5u + (5u << k);
        if (f1 + a1 / 2u + (8u << k) >= (1u << (22u + k))) err += a1 / 4u + (1u << k);
    }
    t.margin = err + err / 4u + 8u;
    t.zero = 0u;  // (without Pdot, FIXED32's fold rounds to it exactly)
    if (own_fixed && epoch && aa != 0.0) {
        const FixedPrep p = fixed_prep(fixed_trial(f, aa, fs));
        const uint4 pt = fixed_point(0.0, fs);
        t.zero = fold_fixed_phase_from<true, false>(fold_fixed_fpart(pt, p), pt, p);
    }
    return t;
}
// Whether the coarse fold serves a job (NaN: it does not).
__device__ inline bool coarse_range_ok(const JobState *st) {
    const double tau = __longlong_as_double((long long)st->tau_max_bits);
    const double f = 1.0 / __longlong_as_double((long long)st->pmin_bits);
    const double a = 0.5 * __longlong_as_double((long long)st->pdot_max_bits) * f * f;
    return tau * f < 2097152.0 && a * tau * tau < 262144.0;
}

// ------------------------------------------------------------------ entropy

// The counter slots a trial keeps: logical slots [zmin, zmax] (fine phase
// bins; 50 %-overlapping bins are formed from them in the epilogue).  FP64 and
// FIXED32 count phase bins directly.  SPLIT32's slot is floor(x n + n) for the
// fold residual x, and the kept range is set by a bound on |x|:
//   RANGE_WIDE: a job that passes the range check (cycles < 2^21) has |x| <=
//     3/4 + 2^-20 (r within 1/2, each cross term within 2^-24 |th fh| < 1/8,
//     three roundings), so slots outside [floor(n (1/4 - 2^-16)),
//     floor(n (7/4 + 2^-16))] are never reached;
//   RANGE_NARROW: every fold of the job re-reduces its residual to |x| <= 1/2
//     (jobs with a Pdot axis, whose folds do that anyway), and only
//     [floor(n (1/2 - 2^-16)), floor(n (3/2 + 2^-16))] is kept;
//   RANGE_MID: |x| <= 9/16 + 2^-16 is kept; a warp whose trials could fold
//     outside it (the bound of split_slot_window) re-reduces its folds as in
//     RANGE_NARROW, the others fold as in RANGE_WIDE.
enum { RANGE_WIDE = 0, RANGE_NARROW = 1, RANGE_MID = 2 };
struct SlotRange {
    int zmin, zmax;
};
__host__ __device__ inline SlotRange slot_range(int mode, int n_phase, int range) {
    if (mode != GCE_PHASE_SPLIT32) return {0, n_phase - 1};
    const double xw =
        (range == RANGE_NARROW ? 0.5 : range == RANGE_MID ? 0.5625 : 0.75) + 1.0 / 65536.0;
    int zmin = (int)floor((double)n_phase * (1.0 - xw));
    int zmax = (int)floor((double)n_phase * (1.0 + xw));
    if (zmin < 0) zmin = 0;
    if (zmax > 2 * n_phase - 1) zmax = 2 * n_phase - 1;
    return {zmin, zmax};
}
__host__ __device__ inline int slots_per_trial(int mode, int n_phase, int range) {
    const SlotRange r = slot_range(mode, n_phase, range);
    return r.zmax - r.zmin + 1;
}

// Byte offsets of the CE kernel's dynamic shared-memory regions, in order: the
// c ln c table (an even number of 8-byte entries, so the points after it stay
// 16-byte aligned), the staged points (8 bytes each for FP64 and for half
// points, else 16; the coarse fold's 12 and 24), the counters and the segment
// starts.  chunk is even, so that the words of the staged pairs lie on 16 bytes (a
// multiple of 32, but in the static entry's last resort a multiple of 8).  The host sizes the launch with `total` and the kernel carves its
// memory with the same offsets.  (k and block do not enter: each warp writes its
// top-k keys and moments straight to global memory.)
inline int half_chunk(int chunk) { return (chunk / 2 + 31) / 32 * 32; }
struct MainSmemLayout {
    unsigned int pts, cnt, seg, total;
};
__host__ __device__ inline MainSmemLayout main_smem_layout(int mode, int block, int tpt, int chunk,
                                                           int n_phase, int n_mag,
                                                           int table_smem, int range, int half) {
    MainSmemLayout L;
    const unsigned int pt = coarse_mode(mode) ? (half ? 12u : 24u)
                            : (mode == GCE_PHASE_FP64 || half) ? 8u : 16u;
    L.pts = 8u * (unsigned int)((table_smem + 1) & ~1);
    L.cnt = L.pts + pt * (unsigned int)chunk;
    L.seg = L.cnt + 4u * (unsigned int)(tpt * slots_per_trial(mode, n_phase, range) * block);
    L.total = L.seg + 4u * (unsigned int)(n_mag + 1);
    return L;
}

// Fixed-point table of c ln c: tab[c] = round(c ln(c) 2^32), tab[0] = tab[1] = 0.
// Eq. 4 rewritten with integer counts is
//   N H = sum_j c_j ln c_j - sum_ij c_ij ln c_ij,
// and summing the table's integers makes both sums exact and independent of
// order; the only error is the table's rounding (at most 2^-33 per term).
constexpr double kTabScale = 4294967296.0;  // 2^32
constexpr double kTabInvScale = 1.0 / 4294967296.0;

// ------------------------------------------------------------------ launches

struct PrepArgs {
    const double *times;
    const double *mags;
    const long long *offsets;  // device copy, n_curves + 1
    int n_curves;
    int n_mag;
    double t0;
    void *payload;             // ModeTraits<MODE>::point_t[sum N], sorted by mag bin per curve
    int *seg;                  // [n_curves][n_mag + 1] segment starts (relative to the curve);
                               // in the coarse fold's range segment_word()
    double *tau;               // coarse modes: tau in payload order, else nullptr
    const JobState *state;
    const unsigned char *bands;  // multi-filter input: filter of each point, or nullptr
    const double2 *band_stats;   // [n_curves][n_bands] {median, standard deviation}
    int n_bands;
};

struct TrialArgs {
    const double *periods;
    const double *pdots;
    int n_periods;
    int n_pdots;
    void *trialc;              // ModeTraits<MODE>::trial_t[n_periods * n_pdots]
    JobState *state;
};

// Moments of a tile's H values: count, mean, sum of squared deviations.
struct TileStats {
    double n, mean, m2;
};

// The moments of a block's records [0, n) merged: the mean from the sums of n and
// n mean, then M2 from the records' own and their means' distances, each in a fixed
// order (a strided run per thread, then a fixed tree), so the result is deterministic.
// Two passes instead of a pairwise update, which divides twice per merge.  A warp's
// binary64 operation holds the SM's unit for 16 cycles, however few lanes it is for,
// so the block's sums and the division are the first warp's alone (shuffle sums in
// every warp and the rest in every thread: the whole merge of 300 curves with 313 lists
// each 14.8 -> 10.2 us).
// sh: kMomentsBlock (the block's threads) doubles, twice.  Thread 0 returns all three.
constexpr int kMomentsBlock = 256;
__device__ inline double block_sum_fixed(const double *sh) {  // first warp; lane 0's result
    double v[kMomentsBlock / 32];
#pragma unroll
    for (int w = 0; w < kMomentsBlock / 32; ++w) v[w] = sh[threadIdx.x + 32 * w];
#pragma unroll
    for (int o = kMomentsBlock / 64; o > 0; o >>= 1)
#pragma unroll
        for (int w = 0; w < o; ++w) v[w] += v[w + o];
    for (int o = 16; o > 0; o >>= 1) v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
    return v[0];
}
__device__ inline TileStats block_moments(const TileStats *ts, int n, double *sh) {
    const int tid = threadIdx.x;
    double c = 0.0, m = 0.0;
#pragma unroll 4
    for (int i = tid; i < n; i += kMomentsBlock) {
        c += ts[i].n;
        m += ts[i].n * ts[i].mean;
    }
    sh[tid] = c;
    sh[kMomentsBlock + tid] = m;
    __syncthreads();
    TileStats r;
    if (tid < 32) {
        r.n = block_sum_fixed(sh);
        r.mean = block_sum_fixed(sh + kMomentsBlock);
        if (r.n > 0.0) r.mean /= r.n;
    }
    __syncthreads();
    if (tid == 0) sh[0] = r.mean;
    __syncthreads();
    const double mean = sh[0];
    double q = 0.0;
#pragma unroll 4
    for (int i = tid; i < n; i += kMomentsBlock) {
        const double d = ts[i].mean - mean;
        if (ts[i].n > 0.0) q += ts[i].m2 + ts[i].n * d * d;
    }
    sh[kMomentsBlock + tid] = q;
    __syncthreads();
    if (tid < 32) r.m2 = block_sum_fixed(sh + kMomentsBlock);
    return r;
}

// Trial tiles of one curve's grid for a launch of `block` threads x `tpt`
// trials.  With several Pdot values and tpt > 1 a tile is block periods x tpt
// consecutive Pdot values, so that a thread's trials share their period (and
// the fold's period part); otherwise a tile is a run of block x tpt flat trial
// indices q n_periods + p.
struct TileGrid {
    long long n_tiles;
    int n_ptiles, pd_major;
};
inline TileGrid tile_grid(long long n_periods, long long n_pdots, int block, int tpt) {
    TileGrid g;
    g.pd_major = (n_pdots > 1 && tpt > 1) ? 1 : 0;
    if (g.pd_major) {
        g.n_ptiles = (int)((n_periods + block - 1) / block);
        g.n_tiles = (long long)g.n_ptiles * ((n_pdots + tpt - 1) / tpt);
    } else {
        g.n_ptiles = 0;
        g.n_tiles = (n_periods * n_pdots + (long long)block * tpt - 1) / ((long long)block * tpt);
    }
    return g;
}

// Trial lists.  The trials of a warp whose threads have two or four are one or two
// lists of 64, and the moments of Eq. 5 are summed per list, so that they come out
// the same in every launch shape: flat list l holds trials t and t + 256 for the 32
// consecutive t from 512 (l / 8) + 32 (l % 8); with several Pdot values a list is 32
// consecutive periods x 2 consecutive Pdot values (tile_grid's tiles).
__host__ __device__ inline long long flat_list_trial(long long l) {
    return (l >> 3) * 512 + (l & 7) * 32;
}
inline long long flat_lists(long long n_trials) {
    const long long rest = n_trials % 512;
    return n_trials / 512 * 8 + (rest >= 256 ? 8 : (rest + 31) / 32);
}
// The tiles of a job: flat jobs with two or four trials per thread are cut into
// runs of block x tpt / 64 lists.
inline TileGrid job_tiles(long long n_periods, long long n_pdots, int block, int tpt) {
    TileGrid g = tile_grid(n_periods, n_pdots, block, tpt);
    if (!g.pd_major && tpt > 1) {
        const long long per = (long long)block * tpt / 64;
        g.n_tiles = (flat_lists(n_periods * n_pdots) + per - 1) / per;
    }
    return g;
}

struct MainArgs {
    const void *payload;
    const long long *offsets;
    const int *seg;
    const void *trialc;
    const int *order;          // curves in processing order (longest first)
    const unsigned long long *table;
    long long n_trials;
    int n_periods, n_pdots;
    int n_tiles;               // trial tiles per curve
    int n_ptiles;              // period-major tiling: tiles along the periods
    int pd_major;              // tile = block periods x tpt Pdot values (else flat runs)
    int range;                 // SPLIT32: the kept slot range (RANGE_*)
    long long n_items;         // n_curves * n_tiles
    // items [0, n_long_items) are (curve, tile) pairs of the first n_long curves
    // of `order`, curve-major; the rest pair the n_short curves after them with
    // the tiles tile-major (curve index fastest)
    long long n_long_items;
    int n_long, n_short;
    int grab;                  // items taken per work-counter increment
    int n_phase;
    int n_mag;
    int chunk;                 // points staged per pass
    int table_smem;            // table entries staged in shared memory
    float *out;                // grid or nullptr
    unsigned long long *cand;  // top-k candidates [n_curves][n_tiles][k] or nullptr
    int k;
    TileStats *stats;          // per-tile moments [n_curves][n_tiles] or nullptr
    int overlap;               // 50 %-overlapping phase bins
    // SPLIT32 / FIXED32 with one Pdot value: the staging buffer holds `chunk`
    // half points (8 bytes); a job whose Pdot is 0 stages half points, one whose
    // single Pdot is not 0 stages chunk / 2 whole points in the same bytes
    int half;
    int kv;                    // CE kernel variant (KV_*): overlapping bins or not
    int pdl;                   // host: launch with programmatic dependence
    // FP64 and FIXED32 jobs: every point's binary64 tau in payload order, and the
    // caller's trial arrays (for the points the coarse fold leaves undecided);
    // plain: payload and trials are in the mode's own format, with no tau
    int plain;
    const double *tau;
    const double *periods;
    const double *pdots;
    JobState *state;
};

// Instantiations of the CE kernel: without overlapping bins (snapshot counters),
// with them (packed two-segment counters for curves of at most 1023 points, snapshot
// counters for longer ones), and for small jobs without them (a CTA's warps share
// one set of 32 x tpt trials).
enum { KV_SNAP = 0, KV_OVL = 1, KV_SHARED = 2 };
inline int kernel_variant(bool overlap) { return overlap ? KV_OVL : KV_SNAP; }
// threads of a CTA with trials (and counters) of their own
inline int trial_threads(int kv, int block) { return kv == KV_SHARED ? 32 : block; }

// The CE kernel's mode for a job's phase mode.
inline int kernel_mode(int mode) {
    return mode == GCE_PHASE_FP64 ? (int)kJobFp64 : mode == GCE_PHASE_FIXED32 ? (int)kJobFixed32 : mode;
}
// The preparation's mode: the kernel's, but FIXED32's own where the coarse fold gains
// nothing over it: an undecided point makes its CTA some 8 us late (mostly fetching
// code that is not cached), which small kernels and many bins feel more than the saved
// multiplies (811 points x 50000 periods 67 us a call with FIXED32's own fold, 79 us
// with the coarse one; 639 x 317 x 2358 periods at 31 bins 491 and 535 us; 1671 x
// 119..952 x 3003 at 50 overlapping bins 2.34 and 2.43 ms; but 300 x 300..900 x 2e4 at
// 15 bins 1.69 and 1.59 ms, 294 x 209..627 x 1222 x 131 Pdot at 50 17.3 and 16.7 ms).
inline int job_prep_mode(const gce_config *cfg, long long n_trials, int n_pdots, int n_curves,
                         int n_sm) {
    const bool small = (n_trials + 31) / 32 * n_curves <= 400ll * n_sm;
    const bool own = small || (n_pdots == 1 && cfg->n_phase_bins > 31);
    return cfg->phase_mode == GCE_PHASE_FIXED32 && own ? (int)GCE_PHASE_FIXED32
                                                       : kernel_mode(cfg->phase_mode);
}
// The CE kernel's mode for a job prepared in job_prep_mode: the one FIXED32's own fold
// has to itself where that is known before the launch (40 curves x 600 points x 1e5
// periods: 50 bins 1.74 ms, 50 overlapping ones 1.70; 1.80 and 1.76 ms in the kernel
// that holds both folds).
inline int main_mode(int prep_mode, int mode) {
    return prep_mode == GCE_PHASE_FIXED32 ? prep_mode : kernel_mode(mode);
}
// The launch shape of a job that was not tuned (gce_api.cu).
int most_tpt(int mode);
int split_range(int mode, int n_pdots, int slot_range);
gce_tuning default_tuning(const gce_config *cfg, int n_pdots);
bool fit_to_job(gce_tuning &t, const gce_config *cfg, int n_pdots, long long n_trials,
                int n_curves, long long n_points, int n_sm, bool stats);

// Programmatic dependent launch.  A call's kernels follow one another on one stream
// and most are short, so each is launched while the one before it still runs and
// waits on the device: pdl_wait() returns when everything before it has completed
// and its writes are visible.  Every kernel that launch_pdl starts calls it before it
// touches what an earlier kernel writes (so completion is transitive), and
// pdl_trigger() lets the next one be scheduled.  The first kernel of a call is
// launched normally, after all of the caller's work.  Not under stream capture.  Only the
// caller's arrays are `const __restrict__` in these kernels: the workspace is written
// during a dependent kernel's lifetime.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;"); }
template <class... P, class... A>
inline cudaError_t launch_pdl(void (*kernel)(P...), unsigned int grid, unsigned int block,
                              size_t smem, cudaStream_t s, bool pdl, A... args) {
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = &attr;
    cfg.numAttrs = pdl ? 1u : 0u;
    return cudaLaunchKernelEx(&cfg, kernel, P(args)...);
}

// Kernel launchers (defined in the .cu files).
// h_offsets, h_order: pinned host memory read by the kernel itself (nullptr: offsets
// are on the device already, and the order is 0, 1, ...); launch_init_few takes the
// offsets of at most kFewCurves curves from any host memory, as a kernel argument
constexpr int kFewCurves = 255;
cudaError_t launch_init_few(JobState *st, const int64_t *h_offsets, long long *offsets, int *order,
                            int n_curves, cudaStream_t s);
cudaError_t launch_init(JobState *st, const long long *h_offsets, const int *h_order,
                        long long *offsets, int *order, int n_curves, cudaStream_t s);
cudaError_t launch_scan(const double *times, const double *mags, long long n_points,
                        const double *periods, int n_periods, const double *pdots, int n_pdots,
                        double t0, JobState *st, bool pdl, cudaStream_t s);
cudaError_t launch_trials(int mode, const TrialArgs &a, bool pdl, cudaStream_t s);
cudaError_t launch_prep(int mode, const PrepArgs &a, bool pdl, cudaStream_t s);
cudaError_t launch_band_stats(const double *mags, const unsigned char *bands,
                              const long long *offsets, int n_curves, int n_bands,
                              double2 *stats, JobState *st, bool pdl, cudaStream_t s);
cudaError_t launch_table(unsigned long long *table, int n_max, cudaStream_t s);
size_t main_smem_bytes(int mode, int block, int tpt, int chunk, int n_phase, int n_mag,
                       int table_smem, int range, int half);
size_t single_smem_bytes(int n_phase, int block);
size_t main_dynamic_smem_limit(int mode, int tpt, int block, int kv, size_t smem_optin);
cudaError_t main_kernel_attrs(int mode, int tpt, int block, int kv, size_t smem_optin);
const void *main_kernel_ptr(int mode, int tpt, int block, int kv);
// per fold mode and trials per thread (gce_main_<mode>_t<tpt>.cu)
#define GCE_MAIN_TU(name, t)                                                           \
    const void *main_kernel_ptr_##name##_t##t(int block, int kv);                       \
    cudaError_t launch_main_##name##_t##t(int block, int grid, size_t smem, const MainArgs &a, \
                                          cudaStream_t s);
GCE_MAIN_TU(fp64, 1)
GCE_MAIN_TU(fp64, 2)
GCE_MAIN_TU(fp64, 4)
GCE_MAIN_TU(split32, 1)
GCE_MAIN_TU(split32, 2)
GCE_MAIN_TU(split32, 4)
GCE_MAIN_TU(fixed32own, 1)
GCE_MAIN_TU(fixed32own, 2)
GCE_MAIN_TU(fixed32own, 4)
GCE_MAIN_TU(fixed32, 1)
GCE_MAIN_TU(fixed32, 2)
GCE_MAIN_TU(fixed32, 4)
#undef GCE_MAIN_TU
cudaError_t launch_main(int mode, int tpt, int block, int grid, size_t smem,
                        const MainArgs &a, cudaStream_t s);
// stats: stats_per moment records per candidate list
cudaError_t launch_topk_merge(const unsigned long long *cand, int n_curves, int n_tiles,
                              int k, int stats_per, float *topk_H, long long *topk_idx, const TileStats *stats,
                              double *mean, double *std_dev, float *rho, const JobState *st,
                              bool pdl, cudaStream_t s);
cudaError_t launch_single(const MainArgs &a, int curve, long long n_points, cudaStream_t s);
cudaError_t launch_counts(int mode, const MainArgs &a, long long n_cells,
                          const long long *cell_curve, const long long *cell_trial,
                          unsigned int *counts, cudaStream_t s);

}  // namespace gce
