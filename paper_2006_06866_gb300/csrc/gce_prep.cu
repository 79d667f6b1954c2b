// Trial-independent preparation (O(sum N + n_trials)): input checks and
// maxima, per-trial fold constants, per-curve magnitude binning with the
// points regrouped by magnitude bin, and the c ln c fixed-point table.
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <numeric>

#include "gce_internal.cuh"

namespace gce {

namespace {

constexpr unsigned long long kPosInfBits = 0x7ff0000000000000ull;

// The job state cleared, and the curves' offsets and processing order copied from
// the caller-side staging buffers (pinned host memory, read over the link: two copies
// on the stream cost more than the whole kernel for small batches).
__device__ __forceinline__ void clear_state(JobState *st) {
    st->tau_max_bits = 0ull;
    st->pmin_bits = kPosInfBits;
    st->pdot_max_bits = 0ull;
    st->err = 0u;
    st->work = 0ull;
    st->wide = 0u;
    st->epoch = 0u;
}
__global__ void k_init(JobState *st, const long long *h_offsets, const int *h_order,
                       long long *offsets, int *order, int n_curves) {
    pdl_trigger();
    const int i0 = blockIdx.x * blockDim.x + threadIdx.x;
    if (i0 == 0) clear_state(st);
    for (int i = i0; i <= n_curves; i += gridDim.x * blockDim.x) {
        if (h_offsets) offsets[i] = h_offsets[i];
        if (i < n_curves) order[i] = h_order ? h_order[i] : i;
    }
}

struct FewOffsets {
    int64_t v[kFewCurves + 1];
    unsigned char order[kFewCurves + 1];  // longest curve first
};
__global__ void k_init_few(JobState *st, const __grid_constant__ FewOffsets few, long long *offsets,
                           int *order, int n_curves) {
    pdl_trigger();
    const int i = threadIdx.x;
    if (i == 0) clear_state(st);
    if (i <= n_curves) offsets[i] = few.v[i];
    if (i < n_curves) order[i] = few.order[i];
}

// Non-negative binary64 values order like their bit patterns, so maxima and
// minima reduce with 64-bit integer atomics.
__device__ inline void atomic_max_pos(unsigned long long *dst, double v) {
    atomicMax(dst, (unsigned long long)__double_as_longlong(v));
}
__device__ inline void atomic_min_pos(unsigned long long *dst, double v) {
    atomicMin(dst, (unsigned long long)__double_as_longlong(v));
}

__device__ inline double warp_max(double v) {
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}
__device__ inline double warp_min(double v) {
    for (int o = 16; o > 0; o >>= 1) v = fmin(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

// t - t0 == 0, on the bits (binary64 arithmetic bounds the preparation)
__device__ inline bool at_epoch(double t, double t0) {
    const unsigned long long x = (unsigned long long)__double_as_longlong(t);
    const unsigned long long y = (unsigned long long)__double_as_longlong(t0);
    return x == y || ((x | y) << 1) == 0ull;
}

// Checks every time, magnitude, period and period derivative; reduces
// max |t - t0|, min P and max |Pdot|.
__global__ void k_scan(const double *__restrict__ times, const double *__restrict__ mags,
                       long long n_points, const double *__restrict__ periods, int n_periods,
                       const double *__restrict__ pdots, int n_pdots, double t0, JobState *st) {
    pdl_trigger();
    pdl_wait();
    unsigned int err = 0u, epoch = 0u;
    double tmax = 0.0, pmin = INFINITY, dmax = 0.0;
    long long stride = (long long)gridDim.x * blockDim.x;
    long long i0 = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    for (long long i = i0; i < n_points; i += stride) {
        double t = times[i], m = mags[i];
        if (!isfinite(t) || !isfinite(m)) err |= ERR_TIME;
        double tau = fabs(t - t0);
        epoch |= at_epoch(t, t0) ? 1u : 0u;
        if (isfinite(tau)) tmax = fmax(tmax, tau);
        else err |= ERR_TIME;
    }
    for (long long i = i0; i < n_periods; i += stride) {
        double p = periods[i];
        if (!isfinite(p) || !(p > 0.0)) err |= ERR_PERIOD;
        else pmin = fmin(pmin, p);
    }
    for (long long i = i0; i < n_pdots; i += stride) {
        double d = pdots[i];
        if (!isfinite(d)) err |= ERR_PDOT;
        else dmax = fmax(dmax, fabs(d));
    }
    tmax = warp_max(tmax);
    dmax = warp_max(dmax);
    pmin = warp_min(pmin);
    err = __reduce_or_sync(0xffffffffu, err);
    epoch = __reduce_or_sync(0xffffffffu, epoch);
    if ((threadIdx.x & 31) == 0) {
        if (tmax > 0.0) atomic_max_pos(&st->tau_max_bits, tmax);
        if (dmax > 0.0) atomic_max_pos(&st->pdot_max_bits, dmax);
        if (pmin < INFINITY) atomic_min_pos(&st->pmin_bits, pmin);
        if (err) atomicOr(&st->err, err);
        if (epoch) st->epoch = 1u;
    }
}

__device__ inline bool beyond_float(double v) { return isinf(__double2float_rn(v)); }

// Per flat trial t = q n_periods + p: f = 1/P, a = (0.5 Pdot) f f (the oracle's
// sequence), stored in the fold mode's format.  Bound by binary64 arithmetic at 2
// lanes per clock and SM, so what binary32 holds exactly is done there, and nothing
// for a Pdot of 0 (5e4 FIXED32 trials 8.4 -> 5.9 us).
template <int MODE>
__global__ void k_trials(TrialArgs a) {
    pdl_trigger();
    pdl_wait();
    const long long n = (long long)a.n_periods * a.n_pdots;
    const double tau_max = __longlong_as_double((long long)a.state->tau_max_bits);
    const FixedScale fs = fixed_scale_from(tau_max);
    // (of a coarse job: every thread that asks agrees, the maxima being final)
    const bool wide = coarse_mode(MODE) && !coarse_range_ok(a.state);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        // Range of the fold (checked once, from the maxima).
        const double pmin = __longlong_as_double((long long)a.state->pmin_bits);
        const double dmax = __longlong_as_double((long long)a.state->pdot_max_bits);
        if (pmin < INFINITY && pmin > 0.0) {
            const double fmax_ = 1.0 / pmin;
            const double amax = 0.5 * dmax * fmax_ * fmax_;
            bool bad = false;
            if (MODE == GCE_PHASE_SPLIT32) {
                // |x| < 1 needs |c| + |c2| < 1/2: cycles < 2^21 and Pdot cycles < 2^19
                bad = tau_max * fmax_ >= 2097152.0 || amax * tau_max * tau_max >= 524288.0;
                // and every value that a fold reads split into finite floats: an infinite
                // one makes the residual NaN, whose slot is no counter of the trial's
                bad = bad || beyond_float(tau_max) || beyond_float(fmax_) ||
                      (dmax > 0.0 && (beyond_float(amax) || beyond_float(tau_max * tau_max)));
            } else if (MODE == GCE_PHASE_FIXED32 || MODE == kJobFixed32) {
                bad = !fixed_range_ok(fmax_, amax, fs.e_tau);
            }
            if (bad) atomicOr(&a.state->err, ERR_RANGE);
        }
        if (coarse_mode(MODE)) a.state->wide = wide ? 1u : 0u;
    }
    for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < n;
         t += (long long)gridDim.x * blockDim.x) {
        const int p = (int)(t % a.n_periods);
        const int q = (int)(t / a.n_periods);
        const double f = 1.0 / a.periods[p];
        const double aa = (0.5 * a.pdots[q]) * f * f;
        if (MODE == GCE_PHASE_FP64 || (MODE == kJobFp64 && wide)) {
            reinterpret_cast<double2 *>(a.trialc)[t] = make_double2(f, aa);
        } else if (MODE == GCE_PHASE_FIXED32 || (MODE == kJobFixed32 && wide)) {
            reinterpret_cast<FixedTrial *>(a.trialc)[t] = fixed_trial(f, aa, fs);
        } else if (coarse_mode(MODE)) {
            reinterpret_cast<CoarseTrial *>(a.trialc)[t] =
                coarse_trial(f, aa, fs, MODE == kJobFixed32, a.state->epoch != 0u);
        } else {
            // f split, and -a split (the fold adds -a tau^2)
            const float fh = __double2float_rn(f);
            const float nah = __double2float_rn(-aa);
            reinterpret_cast<float4 *>(a.trialc)[t] =
                make_float4(fh, __double2float_rn(f - (double)fh), nah,
                            __double2float_rn(-aa - (double)nah));
        }
    }
}

constexpr int kPrepBlock = 256;
constexpr int kPrepMags = 1024, kPrepBins = 8192;

// Magnitude bin of Sec. 2.3 with the oracle's operation sequence:
// i = floor(((m - mn) / (mx - mn)) * n_mag), clamped; mx == mn -> 0.
__device__ inline int mag_bin(double m, double mn, double mx, int n_mag) {
    if (mx == mn) return 0;
    double v = __ddiv_rn(__dsub_rn(m, mn), __dsub_rn(mx, mn));
    int i = __double2int_rd(__dmul_rn(v, (double)n_mag));
    return max(min(i, n_mag - 1), 0);  // (a NaN, of flagged input or a range that overflows: bin 0)
}

// mag_bin, from a binary32 quotient where that decides it: four roundings leave v
// within 255 2^-22 = 6.1e-5 of the sequence's value, so a v farther than 1e-4 from
// the integers has its floor; the others, and ranges that binary32 does not hold
// well, take the binary64 division (some 25 operations at 2 lanes per clock).
struct MagBins {
    double mn, mx;
    float scale;
    int n_mag;
    bool fast;
    __device__ MagBins(double mn_, double mx_, int n_mag_) : mn(mn_), mx(mx_), n_mag(n_mag_) {
        const double range = __dsub_rn(mx, mn);
        fast = range > 1e-30 && range < 1e30;
        scale = fast ? __fdiv_rn((float)n_mag, __double2float_rn(range)) : 0.0f;
    }
    __device__ int operator()(double m) const {
        const float v = __double2float_rn(__dsub_rn(m, mn)) * scale;
        const float f = floorf(v), d = v - f;
        if (fast && d > 1e-4f && d < 1.0f - 1e-4f) return (int)f;
        return mag_bin(m, mn, mx, n_mag);
    }
};

// ------------------------------------------------------------------ filters

// Order-preserving map of binary64 to unsigned 64-bit keys (and back).
__device__ inline unsigned long long f64_key(double v) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
    return (b >> 63) ? ~b : (b | 0x8000000000000000ull);
}
__device__ inline double key_f64(unsigned long long k) {
    return __longlong_as_double((long long)((k >> 63) ? (k & 0x7fffffffffffffffull) : ~k));
}

// The kth smallest (0-based) magnitude of filter b among the curve's n points:
// an exact radix selection on the keys, 8 bits per pass from the top, with
// shared-memory digit histograms.  Every thread returns the value.
__device__ double band_select(const double *m, const unsigned char *bd, int n, int b, int kth,
                              unsigned int *hist, unsigned long long *s_pref, int *s_k) {
    unsigned long long prefix = 0ull;
    for (int shift = 56; shift >= 0; shift -= 8) {
        const unsigned long long high = shift == 56 ? 0ull : ~0ull << (shift + 8);
        for (int i = threadIdx.x; i < 256; i += blockDim.x) hist[i] = 0u;
        __syncthreads();
        for (int k = threadIdx.x; k < n; k += blockDim.x) {
            if (bd[k] != b) continue;
            const unsigned long long key = f64_key(m[k]);
            if ((key & high) == prefix) atomicAdd(&hist[(key >> shift) & 255u], 1u);
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            unsigned int cum = 0u;
            int d = 0;
            for (; d < 255; ++d) {
                if (cum + hist[d] > (unsigned int)kth) break;
                cum += hist[d];
            }
            *s_pref = prefix | ((unsigned long long)d << shift);
            *s_k = kth - (int)cum;
        }
        __syncthreads();
        prefix = *s_pref;
        kth = *s_k;
        __syncthreads();
    }
    return key_f64(prefix);
}

// Smallest (largest) 64-bit key of the warp: the high words first, then the low
// words among the lanes holding the best one.
__device__ inline unsigned long long warp_min_u64(unsigned long long v) {
    const unsigned int hi = __reduce_min_sync(0xffffffffu, (unsigned int)(v >> 32));
    const unsigned int lo =
        __reduce_min_sync(0xffffffffu, (unsigned int)(v >> 32) == hi ? (unsigned int)v : 0xffffffffu);
    return ((unsigned long long)hi << 32) | lo;
}
__device__ inline unsigned long long warp_max_u64(unsigned long long v) { return ~warp_min_u64(~v); }

// Longest curve whose magnitudes k_band_stats holds in shared memory.
constexpr int kBandCurve = 4096;

// The median and population standard deviation of v[0, cnt) (shared memory, in
// point order; overwritten), by one warp: the lower median by an exact radix
// selection on the keys, 8 bits per pass; the upper one, for an even count, is the
// same key or the next larger one; the sums by lane 0 in point order, the squares
// by all lanes.
__device__ double2 warp_band_stats(double *v, int cnt, unsigned int *hist) {
    const int lane = threadIdx.x & 31;
    unsigned long long prefix = 0ull;
    unsigned int kth = (unsigned int)(cnt - 1) / 2, same = 0u;
    for (int shift = 56; shift >= 0; shift -= 8) {
        const unsigned long long high = shift == 56 ? 0ull : ~0ull << (shift + 8);
        for (int i = lane; i < 256; i += 32) hist[i] = 0u;
        __syncwarp();
        for (int k = lane; k < cnt; k += 32) {
            const unsigned long long key = f64_key(v[k]);
            if ((key & high) == prefix) atomicAdd(&hist[(key >> shift) & 255u], 1u);
        }
        __syncwarp();
        unsigned int sum = 0u, incl;
        for (int i = 0; i < 8; ++i) sum += hist[lane * 8 + i];
        incl = sum;
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned int up = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += up;
        }
        // the lane whose eight digits hold the kth key, and the digit
        const int owner = __ffs((int)__ballot_sync(0xffffffffu, incl > kth)) - 1;
        unsigned int below = incl - sum, digit = 0u, count = 0u;
        if (lane == owner)
            for (int i = 0; i < 8; ++i) {
                count = hist[lane * 8 + i];
                digit = (unsigned int)(lane * 8 + i);
                if (below + count > kth) break;
                below += count;
            }
        kth -= __shfl_sync(0xffffffffu, below, owner);
        same = __shfl_sync(0xffffffffu, count, owner);
        prefix |= (unsigned long long)__shfl_sync(0xffffffffu, digit, owner) << shift;
        __syncwarp();
    }
    double med = key_f64(prefix);
    if ((cnt & 1) == 0) {
        unsigned long long next = ~0ull;
        for (int k = lane; k < cnt; k += 32) {
            const unsigned long long key = f64_key(v[k]);
            if (key > prefix && key < next) next = key;
        }
        next = warp_min_u64(next);
        const double hi = kth + 1u < same ? med : key_f64(next);
        med = __dmul_rn(__dadd_rn(med, hi), 0.5);
    }
    double sum = 0.0;
    if (lane == 0)
        for (int k = 0; k < cnt; ++k) sum = __dadd_rn(sum, v[k]);
    const double mean = __ddiv_rn(__shfl_sync(0xffffffffu, sum, 0), (double)cnt);
    for (int k = lane; k < cnt; k += 32) {
        const double d = __dsub_rn(v[k], mean);
        v[k] = __dmul_rn(d, d);
    }
    __syncwarp();
    double ss = 0.0;
    if (lane == 0)
        for (int k = 0; k < cnt; ++k) ss = __dadd_rn(ss, v[k]);
    ss = __shfl_sync(0xffffffffu, ss, 0);
    return make_double2(med, __dsqrt_rn(__ddiv_rn(ss, (double)cnt)));
}

// One CTA per curve: for each filter b, the median and the population standard
// deviation of its magnitudes (the per-filter normalisation of Sec. 2.3), in the
// operation order stated in gce.h: the median exactly (radix selection), the
// mean and the sum of squared deviations in binary64 in point order, so that the
// normalised values match a plain sequential statement bit for bit.  A filter with
// no points gets {0, 0}.  Band indices >= n_bands set ERR_BAND.
// Bound by the two chains of binary64 additions, so curves of up to kBandCurve points
// are split by filter into shared memory and each filter has a warp of its own (300
// curves of 300..900 points in two filters: 360 us when one thread walked global
// memory filter by filter, 58 us now).
__global__ void __launch_bounds__(256) k_band_stats(const double *__restrict__ mags,
                                                    const unsigned char *__restrict__ bands,
                                                    const long long *offsets,
                                                    int n_bands, double2 *stats, JobState *st) {
    __shared__ unsigned int hist[GCE_MAX_BANDS][256];
    __shared__ double vals[kBandCurve];
    __shared__ unsigned long long s_pref;
    __shared__ int s_k, s_cnt[GCE_MAX_BANDS];
    pdl_trigger();
    pdl_wait();
    const int c = blockIdx.x;
    const long long lo = offsets[c];
    const int n = (int)(offsets[c + 1] - lo);
    const double *m = mags + lo;
    const unsigned char *bd = bands + lo;
    if (threadIdx.x < GCE_MAX_BANDS) s_cnt[threadIdx.x] = 0;
    __syncthreads();
    bool bad = false;
    for (int k = threadIdx.x; k < n; k += blockDim.x) {
        const int b = bd[k];
        if (b >= n_bands) bad = true;
        else atomicAdd(&s_cnt[b], 1);
    }
    if (__syncthreads_or(bad)) {
        if (threadIdx.x == 0) atomicOr(&st->err, ERR_BAND);
        return;
    }
    if (n <= kBandCurve) {
        const int b = threadIdx.x >> 5, lane = threadIdx.x & 31;
        if (b >= n_bands) return;
        int first = 0;
        for (int i = 0; i < b; ++i) first += s_cnt[i];
        const int cnt = s_cnt[b];
        int at = first;
#pragma unroll 4
        for (int k0 = 0; k0 < n; k0 += 32) {
            const int k = k0 + lane;
            const bool mine = k < n && bd[k] == b;
            const unsigned int all = __ballot_sync(0xffffffffu, mine);
            if (mine) vals[at + __popc(all & ((1u << lane) - 1u))] = m[k];
            at += __popc(all);
        }
        __syncwarp();
        const double2 r = cnt > 0 ? warp_band_stats(vals + first, cnt, hist[b]) : make_double2(0.0, 0.0);
        if (lane == 0) stats[(long long)c * n_bands + b] = r;
        return;
    }
    for (int b = 0; b < n_bands; ++b) {
        const int cnt = s_cnt[b];
        double2 r = make_double2(0.0, 0.0);
        if (cnt > 0) {
            double med = band_select(m, bd, n, b, (cnt - 1) / 2, hist[0], &s_pref, &s_k);
            if ((cnt & 1) == 0) {
                const double hi = band_select(m, bd, n, b, cnt / 2, hist[0], &s_pref, &s_k);
                med = __dmul_rn(__dadd_rn(med, hi), 0.5);
            }
            if (threadIdx.x == 0) {
                double sum = 0.0;
                for (int k = 0; k < n; ++k)
                    if (bd[k] == b) sum = __dadd_rn(sum, m[k]);
                const double mean = __ddiv_rn(sum, (double)cnt);
                double ss = 0.0;
                for (int k = 0; k < n; ++k)
                    if (bd[k] == b) {
                        const double d = __dsub_rn(m[k], mean);
                        ss = __dadd_rn(ss, __dmul_rn(d, d));
                    }
                r = make_double2(med, __dsqrt_rn(__ddiv_rn(ss, (double)cnt)));
            }
        }
        if (threadIdx.x == 0) stats[(long long)c * n_bands + b] = r;
    }
}

// The magnitude the bins of Sec. 2.3 see: the raw value, or with multi-filter
// input (m - median) / sd of the point's filter (0 when sd is 0).
struct MagView {
    const double *m;
    const unsigned char *bd;  // nullptr: raw magnitudes
    const double2 *bs;        // this curve's {median, sd} per filter
    int nb;
    __device__ double operator[](int k) const {
        if (!bd) return m[k];
        const int b = bd[k];
        if (b >= nb) return 0.0;  // flagged by k_band_stats; never read past the table
        const double2 s = bs[b];
        return s.y > 0.0 ? __ddiv_rn(__dsub_rn(m[k], s.x), s.y) : 0.0;
    }
};

// One CTA per curve: min/max of the magnitudes, magnitude bins, a counting sort
// of the points by magnitude bin (segment starts written to seg), and the
// points' fold payload written in the sorted order.  The order of points inside
// a segment is arbitrary (counts do not depend on it), but that a coarse job's points
// at the epoch come last (segment_word).
template <int MODE>
__global__ void __launch_bounds__(kPrepBlock) k_prep(PrepArgs a) {
    __shared__ unsigned long long sh_min[kPrepBlock / 32], sh_max[kPrepBlock / 32];
    __shared__ int hist[GCE_MAX_MAG_BINS + 1], zeros[GCE_MAX_MAG_BINS + 1];
    // the first points' magnitudes and bins, each computed once (binary64 arithmetic
    // bounds this kernel: the divisions of the filters' and the bins' normalisation)
    __shared__ double s_m[kPrepMags];
    __shared__ unsigned char s_bin[kPrepBins];
    pdl_trigger();
    pdl_wait();
    const int c = blockIdx.x;
    const long long lo = a.offsets[c];
    const int n = (int)(a.offsets[c + 1] - lo);
    // (the state first: its loads run beside the magnitudes', and k_trials, which is over,
    // has taken the binary64 division that decides wide)
    const FixedScale fs = fixed_scale_from(__longlong_as_double((long long)a.state->tau_max_bits));
    const uint4 flags = job_flags(a.state);
    const bool wide = coarse_mode(MODE) && flags.y;
    const bool apart = coarse_mode(MODE) && !wide && flags.z;  // points at the epoch come last
    const MagView m{a.mags + lo, a.bands ? a.bands + lo : nullptr,
                    a.bands ? a.band_stats + (long long)c * a.n_bands : nullptr, a.n_bands};
    const double *t = a.times + lo;
    unsigned long long kmin = ~0ull, kmax = 0ull;
    for (int k = threadIdx.x; k < n; k += blockDim.x) {
        const double v = m[k];
        if (k < kPrepMags) s_m[k] = v;
        const unsigned long long key = f64_key(v);
        kmin = key < kmin ? key : kmin;
        kmax = key > kmax ? key : kmax;
    }
    kmin = warp_min_u64(kmin);
    kmax = warp_max_u64(kmax);
    if ((threadIdx.x & 31) == 0) {
        sh_min[threadIdx.x >> 5] = kmin;
        sh_max[threadIdx.x >> 5] = kmax;
    }
    for (int i = threadIdx.x; i <= a.n_mag; i += blockDim.x) hist[i] = zeros[i] = 0;
    __syncthreads();
#pragma unroll
    for (int w = 0; w < kPrepBlock / 32; ++w) {
        kmin = sh_min[w] < kmin ? sh_min[w] : kmin;
        kmax = sh_max[w] > kmax ? sh_max[w] : kmax;
    }
    const MagBins bins(key_f64(kmin), key_f64(kmax), a.n_mag);
    for (int k = threadIdx.x; k < n; k += blockDim.x) {
        const int b = bins(k < kPrepMags ? s_m[k] : m[k]);
        if (k < kPrepBins) s_bin[k] = (unsigned char)b;
        atomicAdd(&hist[b], 1);
        if (apart && at_epoch(t[k], a.t0)) atomicAdd(&zeros[b], 1);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        int run = 0;
        int *seg = a.seg + (long long)c * (a.n_mag + 1);
        for (int i = 0; i < a.n_mag; ++i) {
            const int h = hist[i], z = apart ? zeros[i] : 0;
            hist[i] = run;
            seg[i] = (int)segment_word(run, z);
            run += h;
            if (apart) zeros[i] = run;
        }
        seg[a.n_mag] = run;
    }
    __syncthreads();
    for (int k = threadIdx.x; k < n; k += blockDim.x) {
        const int b = k < kPrepBins ? s_bin[k] : bins(k < kPrepMags ? s_m[k] : m[k]);
        const int pos = apart && at_epoch(t[k], a.t0) ? atomicAdd(&zeros[b], -1) - 1 : atomicAdd(&hist[b], 1);
        const double tau = __dsub_rn(t[k], a.t0);
        if (coarse_mode(MODE)) a.tau[lo + pos] = tau;
        if (MODE == GCE_PHASE_FP64) {
            reinterpret_cast<double *>(a.payload)[lo + pos] = tau;
        } else if (MODE == GCE_PHASE_FIXED32 || (MODE == kJobFixed32 && wide)) {
            reinterpret_cast<uint4 *>(a.payload)[lo + pos] = fixed_point(tau, fs);
        } else if (coarse_mode(MODE)) {
            reinterpret_cast<CoarsePoint *>(a.payload)[lo + pos] = coarse_point(tau, fs.e_tau);
        } else {
            const double tau2 = __dmul_rn(tau, tau);
            const float th = __double2float_rn(tau);
            const float t2h = __double2float_rn(tau2);
            reinterpret_cast<float4 *>(a.payload)[lo + pos] =
                make_float4(th, __double2float_rn(tau - (double)th), t2h,
                            __double2float_rn(tau2 - (double)t2h));
        }
    }
}

__global__ void k_table(unsigned long long *table, int n_max) {
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c <= n_max; c += gridDim.x * blockDim.x) {
        double v = c > 1 ? (double)c * log((double)c) * kTabScale : 0.0;
        table[c] = (unsigned long long)__double2ll_rn(v);
    }
}

int grid_for(long long n, int block, int cap) {
    long long g = (n + block - 1) / block;
    if (g < 1) g = 1;
    if (g > cap) g = cap;
    return (int)g;
}

}  // namespace

cudaError_t launch_init(JobState *st, const long long *h_offsets, const int *h_order,
                        long long *offsets, int *order, int n_curves, cudaStream_t s) {
    k_init<<<grid_for((long long)n_curves + 1, 256, 152), 256, 0, s>>>(st, h_offsets, h_order,
                                                                       offsets, order, n_curves);
    return cudaGetLastError();
}

cudaError_t launch_init_few(JobState *st, const int64_t *h_offsets, long long *offsets, int *order,
                            int n_curves, cudaStream_t s) {
    if (n_curves > kFewCurves) return cudaErrorInvalidValue;
    FewOffsets few;
    for (int i = 0; i <= kFewCurves; ++i) few.v[i] = h_offsets[i <= n_curves ? i : n_curves];
    std::iota(few.order, few.order + n_curves, (unsigned char)0);
    std::stable_sort(few.order, few.order + n_curves, [&](int a, int b) {
        return h_offsets[a + 1] - h_offsets[a] > h_offsets[b + 1] - h_offsets[b];
    });
    k_init_few<<<1, kFewCurves + 1, 0, s>>>(st, few, offsets, order, n_curves);
    return cudaGetLastError();
}

cudaError_t launch_scan(const double *times, const double *mags, long long n_points,
                        const double *periods, int n_periods, const double *pdots, int n_pdots,
                        double t0, JobState *st, bool pdl, cudaStream_t s) {
    long long n = n_points;
    if (n_periods > n) n = n_periods;
    if (n_pdots > n) n = n_pdots;
    return launch_pdl(k_scan, grid_for(n, 256, 1216), 256, 0, s, pdl, times, mags, n_points, periods,
                      n_periods, pdots, n_pdots, t0, st);
}

cudaError_t launch_trials(int mode, const TrialArgs &a, bool pdl, cudaStream_t s) {
    long long n = (long long)a.n_periods * a.n_pdots;
    int g = grid_for(n, 256, 4864);
    switch (mode) {
        case GCE_PHASE_FP64: return launch_pdl(k_trials<GCE_PHASE_FP64>, g, 256, 0, s, pdl, a);
        case GCE_PHASE_SPLIT32: return launch_pdl(k_trials<GCE_PHASE_SPLIT32>, g, 256, 0, s, pdl, a);
        case kJobFp64: return launch_pdl(k_trials<kJobFp64>, g, 256, 0, s, pdl, a);
        case kJobFixed32: return launch_pdl(k_trials<kJobFixed32>, g, 256, 0, s, pdl, a);
        default: return launch_pdl(k_trials<GCE_PHASE_FIXED32>, g, 256, 0, s, pdl, a);
    }
}

cudaError_t launch_band_stats(const double *mags, const unsigned char *bands,
                              const long long *offsets, int n_curves, int n_bands,
                              double2 *stats, JobState *st, bool pdl, cudaStream_t s) {
    if (n_curves <= 0) return cudaSuccess;
    return launch_pdl(k_band_stats, n_curves, 256, 0, s, pdl, mags, bands, offsets, n_bands, stats, st);
}

cudaError_t launch_prep(int mode, const PrepArgs &a, bool pdl, cudaStream_t s) {
    if (a.n_curves <= 0) return cudaSuccess;
    const unsigned int g = a.n_curves;
    switch (mode) {
        case GCE_PHASE_FP64: return launch_pdl(k_prep<GCE_PHASE_FP64>, g, kPrepBlock, 0, s, pdl, a);
        case GCE_PHASE_SPLIT32: return launch_pdl(k_prep<GCE_PHASE_SPLIT32>, g, kPrepBlock, 0, s, pdl, a);
        case kJobFp64: return launch_pdl(k_prep<kJobFp64>, g, kPrepBlock, 0, s, pdl, a);
        case kJobFixed32: return launch_pdl(k_prep<kJobFixed32>, g, kPrepBlock, 0, s, pdl, a);
        default: return launch_pdl(k_prep<GCE_PHASE_FIXED32>, g, kPrepBlock, 0, s, pdl, a);
    }
}

cudaError_t launch_table(unsigned long long *table, int n_max, cudaStream_t s) {
    k_table<<<grid_for((long long)n_max + 1, 256, 1024), 256, 0, s>>>(table, n_max);
    return cudaGetLastError();
}

}  // namespace gce
