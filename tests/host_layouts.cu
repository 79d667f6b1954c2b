// The coarse fold's shared-memory layout and the flat trial lists, from the library's own
// headers, on the CPU.  Built and run by tests/test_host_layouts.py.
#include <cstdio>
#include <random>
#include <vector>

#include "../paper_2006_06866_gb300/csrc/gce_internal.cuh"

using namespace gce;

static int g_fail = 0;
#define CHECK(cond, ...)                         \
    do {                                         \
        if (!(cond) && g_fail++ < 20) {          \
            std::printf("FAIL %s: ", #cond);     \
            std::printf(__VA_ARGS__);            \
            std::printf("\n");                   \
        }                                        \
    } while (0)

// Every chunk that a plan comes to is a multiple of 32 and ends at 32 or more.
static void check_chunks() {
    for (int c = 32; c <= 8192; c += 32) {
        for (int x = c; x > 64;) {
            const int h = half_chunk(x);
            CHECK(h < x && h % 32 == 0 && h >= 32 && 2 * h >= x, "%d halves to %d", x, h);
            x = h;
        }
    }
}

// stage_coarse's words (kernel header: pairs of 16 bytes from 0, then from 8 and 16 chunk
// bytes on) lie in the staged region and on their alignment, and so do the points of the
// mode's own fold, which runs in the same layout beyond the coarse range.
static void check_coarse_layout(std::mt19937_64 &rng) {
    for (int it = 0; it < 40000; ++it) {
        const int mode = rng() % 2 ? (int)kJobFp64 : (int)kJobFixed32;
        const int own = mode == kJobFp64 ? (int)GCE_PHASE_FP64 : (int)GCE_PHASE_FIXED32;
        const int chunk = 8 * (1 + (int)(rng() % 1024)), half = (int)(rng() % 2);
        const int blocks[] = {32, 64, 128, 256, 512}, tpts[] = {1, 2, 4};
        const int B = blocks[rng() % 5], T = tpts[rng() % 3];
        const int n_phase = 1 + (int)(rng() % GCE_MAX_PHASE_BINS), n_mag = 1 + (int)(rng() % GCE_MAX_MAG_BINS);
        const int table = 1 + (int)(rng() % 2048);
        const MainSmemLayout L = main_smem_layout(mode, B, T, chunk, n_phase, n_mag, table, RANGE_WIDE, half);
        const MainSmemLayout P = main_smem_layout(own, B, T, chunk, n_phase, n_mag, table, RANGE_WIDE, half);
        const unsigned int bytes = L.cnt - L.pts;
        CHECK(L.pts % 16 == 0 && L.cnt % 4 == 0 && L.pts >= 8u * (unsigned int)table, "pts %u cnt %u", L.pts, L.cnt);
        CHECK(L.seg == L.cnt + 4u * (unsigned int)(T * n_phase * B), "seg %u", L.seg);
        CHECK(L.total == L.seg + 4u * (unsigned int)(n_mag + 1), "total %u", L.total);
        CHECK(P.total <= L.total, "plain %u coarse %u", P.total, L.total);
        for (int job_pdot = 0; job_pdot < 2; ++job_pdot) {
            const bool halves = half && !job_pdot;
            const int pts = half && job_pdot ? (chunk >> 1) & ~1 : chunk;
            if (pts == 0) continue;
            // last byte of the last pair, and the alignment of the second and third words
            const unsigned int pairs = (unsigned int)pts / 2u, second = 8u * (unsigned int)pts;
            const unsigned int end = halves ? second + 8u * pairs : 2u * second + 16u * pairs;
            CHECK(pts % 2 == 0 && second % 16 == 0, "%d points", pts);
            CHECK(end <= bytes, "chunk %d half %d pdot %d: %u of %u bytes", chunk, half, job_pdot, end, bytes);
            const unsigned int one = own == GCE_PHASE_FP64 || halves ? 8u : 16u;
            CHECK(one * (unsigned int)pts <= bytes, "own points: %u x %d in %u", one, pts, bytes);
        }
    }
}

// The tiles of a flat job: every trial in exactly one thread's slot, whatever the shape.
static void check_lists(std::mt19937_64 &rng) {
    std::vector<unsigned char> seen;
    for (int it = 0; it < 400; ++it) {
        const long long n = it < 200 ? 1 + it * 7 : 1 + (long long)(rng() % 30000);
        for (int B : {32, 64, 128, 256, 512})
            for (int T : {1, 2, 4}) {
                if (B * T < 64) continue;
                const TileGrid g = job_tiles(n, 1, B, T);
                seen.assign((size_t)n, 0);
                for (long long tile = 0; tile < g.n_tiles; ++tile) {
                    int in_tile = 0;
                    for (int tid = 0; tid < B; ++tid)
                        for (int s = 0; s < T; ++s) {
                            const long long t = T == 1 ? tile * B + tid
                                : flat_list_trial((tile * (B / 32) + tid / 32) * (T / 2) + s / 2) + (s % 2) * 256 + tid % 32;
                            if (t >= n) continue;
                            ++seen[(size_t)t];
                            ++in_tile;
                        }
                    CHECK(in_tile > 0, "n %lld block %d x %d: tile %lld empty", n, B, T, tile);
                }
                for (long long t = 0; t < n; ++t)
                    CHECK(seen[(size_t)t] == 1, "n %lld block %d x %d: trial %lld %d times", n, B, T, t, seen[(size_t)t]);
            }
    }
}

// A segment word holds every start and count that a curve can have.
static void check_segment_words() {
    for (int start = 0; start <= GCE_MAX_CURVE_POINTS; start += 13)
        for (int zeros : {0, 1, 2, 255, 32767, 32768, GCE_MAX_CURVE_POINTS}) {
            const unsigned int w = segment_word(start, zeros);
            CHECK(segment_start(w) == start && segment_zeros(w) == zeros, "%d %d", start, zeros);
        }
}

int main() {
    std::mt19937_64 rng(7);
    check_chunks();
    check_coarse_layout(rng);
    check_lists(rng);
    check_segment_words();
    if (g_fail) {
        std::printf("%d checks failed\n", g_fail);
        return 1;
    }
    std::printf("ok\n");
    return 0;
}
