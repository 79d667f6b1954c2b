// The last answers to "how many CTAs of this kernel with this much dynamic shared memory fit
// on an SM".  A fixed array: an entry point of the C ABI that holds one lets no exception out
// and allocates nothing.
#pragma once

#include <cstddef>

namespace gce {

struct OccCache {
    static constexpr int kSize = 64;
    struct Entry {
        const void *kernel;
        size_t smem;
        int occ;
    };
    Entry entry[kSize] = {};
    int used = 0, next = 0;

    void clear() { used = next = 0; }
    bool find(const void *kernel, size_t smem, int *occ) const {
        for (int i = 0; i < used; ++i)
            if (entry[i].kernel == kernel && entry[i].smem == smem) {
                *occ = entry[i].occ;
                return true;
            }
        return false;
    }
    // (the oldest goes when it is full)
    void put(const void *kernel, size_t smem, int occ) {
        entry[next] = Entry{kernel, smem, occ};
        next = (next + 1) % kSize;
        used = used < kSize ? used + 1 : kSize;
    }
};

}  // namespace gce
