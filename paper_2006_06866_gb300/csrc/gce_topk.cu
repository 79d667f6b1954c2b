// First level of the per-curve top-k merge.  The persistent CE kernel leaves k
// candidate keys per (curve, trial tile, warp) -- a "tile" below is one such
// list; a grid of 5e6 periods x 512 Pdot values has millions per curve, and one block per curve scanning them
// k times would leave the rest of the GPU idle.  Here many blocks per curve
// each stage one group of tiles' keys in shared memory once, keep its k
// smallest, and merge the group's tile moments (Eq. 5), so that the final
// per-curve merge reads a few thousand keys.
#include <cstdint>

#include "gce_topk.cuh"

namespace gce {

namespace {

constexpr unsigned long long kEmptyKey = ~0ull;
constexpr int kReduceBlock = kMomentsBlock;

// Smallest 64-bit key of the warp: the smallest high word, then the smallest
// low word among the lanes holding it.
__device__ __forceinline__ unsigned long long warp_min_u64(unsigned long long v) {
    const unsigned int hi = __reduce_min_sync(0xffffffffu, (unsigned int)(v >> 32));
    const unsigned int lo =
        __reduce_min_sync(0xffffffffu, (unsigned int)(v >> 32) == hi ? (unsigned int)v : 0xffffffffu);
    return ((unsigned long long)hi << 32) | lo;
}

__global__ void __launch_bounds__(kReduceBlock)
    k_topk_reduce(const unsigned long long *cand, int n_tiles, int k,
                  int tiles_per_group, int n_groups, int stats_per,
                  const TileStats *stats,
                  unsigned long long *cand2, TileStats *stats2,
                  const JobState *st) {
    __shared__ unsigned long long s_keys[kReduceKeys];
    __shared__ unsigned long long s_warp[kReduceBlock / 32];
    __shared__ double s_mom[2 * kMomentsBlock];
    pdl_trigger();
    pdl_wait();
    if (st->err) return;
    const long long b = blockIdx.x;
    const int c = (int)(b / n_groups);
    const int g = (int)(b - (long long)c * n_groups);
    const int t0 = g * tiles_per_group;
    const int nt = min(tiles_per_group, n_tiles - t0);
    const int n = nt * k;  // <= kReduceKeys by the choice of tiles_per_group
    const unsigned long long *src = cand + ((long long)c * n_tiles + t0) * k;
    for (int i = threadIdx.x; i < n; i += kReduceBlock) s_keys[i] = src[i];
    __syncthreads();
    unsigned long long *dst = cand2 + (long long)b * k;
    // k rounds of "smallest key above the previous one"; keys are unique
    unsigned long long last = 0ull;
    for (int r = 0; r < k; ++r) {
        unsigned long long mine = kEmptyKey;
        for (int i = threadIdx.x; i < n; i += kReduceBlock) {
            const unsigned long long v = s_keys[i];
            if ((r == 0 || v > last) && v < mine) mine = v;
        }
        mine = warp_min_u64(mine);
        if ((threadIdx.x & 31) == 0) s_warp[threadIdx.x >> 5] = mine;
        __syncthreads();
        unsigned long long m = s_warp[0];
#pragma unroll
        for (int w = 1; w < kReduceBlock / 32; ++w) m = s_warp[w] < m ? s_warp[w] : m;
        __syncthreads();
        last = m;
        if (threadIdx.x == 0) dst[r] = m;
    }
    if (!stats) return;
    // the group's moments
    const TileStats m = block_moments(stats + ((long long)c * n_tiles + t0) * stats_per, nt * stats_per, s_mom);
    if (threadIdx.x == 0) stats2[b] = m;
}

}  // namespace

cudaError_t launch_topk_reduce(const unsigned long long *cand, int n_curves, int n_tiles, int k,
                               int tiles_per_group, int n_groups, int stats_per,
                               const TileStats *stats,
                               unsigned long long *cand2, TileStats *stats2, const JobState *st,
                               bool pdl, cudaStream_t s) {
    if (n_curves <= 0 || n_groups <= 0) return cudaSuccess;
    if (k < 1 || (long long)tiles_per_group * k > kReduceKeys) return cudaErrorInvalidValue;
    const long long blocks = (long long)n_curves * n_groups;
    if (blocks > 0x7fffffffll) return cudaErrorInvalidValue;
    return launch_pdl(k_topk_reduce, (unsigned int)blocks, kReduceBlock, 0, s, pdl, cand, n_tiles, k,
                      tiles_per_group, n_groups, stats_per, stats, cand2, stats2, st);
}

}  // namespace gce
