// The handle's workspace policy (gce_workspace.h) against a stand-in for the device's
// memory.  Built and run on the CPU by tests/test_host_workspace.py.
#include <cstdio>
#include <map>

#include "../paper_2006_06866_gb300/csrc/gce_workspace.h"

using namespace gce;

static size_t g_budget, g_used;
static int g_ops;
static std::map<void *, size_t> g_live;
static size_t g_next = 256;

static const DevMemory kFake = {
    [](void **p, size_t n) {
        ++g_ops;
        if (g_used + n > g_budget) return false;
        *p = reinterpret_cast<void *>(g_next);
        g_next += n + 256;
        g_live[*p] = n;
        g_used += n;
        return true;
    },
    [](void *p) {
        ++g_ops;
        g_used -= g_live.at(p);
        g_live.erase(p);
    },
    []() { return true; }, []() { return g_budget - g_used; }};

#define CHECK(c)                                              \
    do {                                                      \
        if (!(c)) {                                           \
            std::printf("FAIL line %d: %s\n", __LINE__, #c); \
            return 1;                                         \
        }                                                     \
    } while (0)

int main() {
    const size_t M = (size_t)1 << 20;
    // payload, trial constants, tau, candidates: a coarse job's bytes and the plain one's
    const size_t c[4] = {240 * M, 320 * M, 80 * M, 100 * M}, q[4] = {80 * M, 160 * M, 0, 100 * M};
    for (size_t budget = 0; budget <= 900 * M; budget += M) {
        for (int before = 0; before < 3; ++before) {  // nothing, a small coarse job, another plain one
            g_budget = 900 * M;
            g_used = 0;
            g_live.clear();
            DevBuf b[4];
            Need cn[4], pn[4];
            bool coarse = false, ask = false;
            for (int i = 0; i < 4; ++i) {
                cn[i] = {&b[i], before == 1 ? c[i] / 4 : c[i]};
                pn[i] = {&b[i], before == 2 ? q[i] / 2 : q[i]};
            }
            if (before) CHECK(job_buffers(kFake, before == 1 ? cn : nullptr, pn, 4, 3, &coarse, &ask) == GROWN);
            if (g_used > budget) continue;
            g_budget = budget;
            for (int i = 0; i < 4; ++i) {
                cn[i] = {&b[i], c[i]};
                pn[i] = {&b[i], q[i]};
            }
            const Growth g = job_buffers(kFake, cn, pn, 4, 3, &coarse, &ask);
            // what fits plain (340 MiB) is taken, whatever the buffers held
            CHECK((g == GROWN) == (budget >= 340 * M));
            CHECK(g_used <= g_budget);
            if (g != GROWN) continue;
            for (int i = 0; i < 4; ++i)
                CHECK((coarse ? c[i] : q[i]) == 0 || (b[i].p && b[i].bytes >= (coarse ? c[i] : q[i])));
            CHECK(coarse || budget < 740 * M + 8 * M);
            CHECK(!coarse || budget >= 740 * M);
            // the same call again allocates and frees nothing
            const int ops = g_ops;
            bool again = false;
            CHECK(job_buffers(kFake, cn, pn, 4, 3, &again, &ask) == GROWN && again == coarse && g_ops == ops);
            // with memory to spare again, it runs coarse
            g_budget = 2000 * M;
            CHECK(job_buffers(kFake, cn, pn, 4, 3, &again, &ask) == GROWN && again);
        }
    }
    // small growth: tried without asking, and after one that failed asked for, so that calls
    // in the plain form allocate nothing from the second on
    const size_t K = (size_t)1 << 10;
    for (size_t budget = 0; budget <= 900 * K; budget += K) {
        g_budget = budget;
        g_used = 0;
        g_live.clear();
        DevBuf b[4];
        Need cn[4], pn[4];
        bool coarse = false, ask = false;
        for (int i = 0; i < 4; ++i) {
            cn[i] = {&b[i], c[i] / M * K};
            pn[i] = {&b[i], q[i] / M * K};
        }
        const Growth g = job_buffers(kFake, cn, pn, 4, 3, &coarse, &ask);
        CHECK((g == GROWN) == (budget >= 340 * K) && coarse == (budget >= 740 * K) && g_used <= g_budget);
        if (g != GROWN) continue;
        const int ops = g_ops;
        for (int rep = 0; rep < 3; ++rep) {
            bool again = false;
            CHECK(job_buffers(kFake, cn, pn, 4, 3, &again, &ask) == GROWN && again == coarse && g_ops == ops);
        }
    }
    std::printf("ok\n");
    return 0;
}
