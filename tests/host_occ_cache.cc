// OccCache on the CPU (tests/test_host_occ_cache.py).
#include <cstdio>
#include <type_traits>

#include "../paper_2006_06866_gb300/csrc/gce_occ_cache.h"

using gce::OccCache;
static_assert(std::is_trivially_copyable<OccCache>::value, "allocates nothing");

int main() {
    OccCache c;
    const int n = 3 * OccCache::kSize + 5;
    int keys[n], v = -1;
    for (int i = 0; i < n; ++i) {
        if (c.find(&keys[i], 100u + i, &v)) return 1;
        c.put(&keys[i], 100u + i, i);
        for (int j = 0; j <= i; ++j) {
            const bool kept = j > i - OccCache::kSize;
            if (c.find(&keys[j], 100u + j, &v) != kept || (kept && v != j)) return 2;
            if (c.find(&keys[j], 101u + j, &v)) return 3;
        }
    }
    c.clear();
    if (c.find(&keys[n - 1], 99u + n, &v)) return 4;
    std::puts("ok");
    return 0;
}
