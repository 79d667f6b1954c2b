// The handle's grow-only device buffers and how a job gets them.  The device's allocator
// comes as a table of functions, so that the policy can be run on the CPU against a
// stand-in with little memory.
#pragma once

#include <algorithm>
#include <cstddef>

namespace gce {

struct DevBuf {
    void *p = nullptr;
    size_t bytes = 0;
};

struct DevMemory {
    bool (*alloc)(void **, size_t);
    void (*release)(void *);
    bool (*wait)();             // for the work that may still read a buffer
    size_t (*available)();      // free bytes
};

// One buffer of a job and the bytes that the job needs of it (0: none).
struct Need {
    DevBuf *buf;
    size_t bytes;
};

enum Growth { GROWN = 0, NO_MEMORY = 1, WAIT_FAILED = 2 };

inline Growth drop(const DevMemory &m, DevBuf &b) {
    if (!b.p) return GROWN;
    if (!m.wait()) return WAIT_FAILED;
    m.release(b.p);
    b.p = nullptr;
    b.bytes = 0;
    return GROWN;
}

// At least `bytes` in b, half as much again as it had where that fits (contents are lost).
inline Growth grow(const DevMemory &m, DevBuf &b, size_t bytes) {
    if (bytes <= b.bytes && b.p) return GROWN;
    size_t want = std::max(std::max(bytes, (size_t)256), b.bytes + b.bytes / 2);
    if (drop(m, b) != GROWN) return WAIT_FAILED;
    if (!m.alloc(&b.p, want)) {
        want = bytes;
        if (!m.alloc(&b.p, want)) {
            b.p = nullptr;
            return NO_MEMORY;
        }
    }
    b.bytes = want;
    return GROWN;
}

inline Growth grow_all(const DevMemory &m, const Need *need, int n) {
    for (int i = 0; i < n; ++i) {
        if (need[i].bytes == 0) continue;
        const Growth g = grow(m, *need[i].buf, need[i].bytes);
        if (g != GROWN) return g;
    }
    return GROWN;
}

// Whether the buffers that have to grow find the memory (each rounded up to the
// allocator's 2 MiB pages; what they hold is given back first).  Asking the device takes
// some 25 us, a fifth of a small job's first call, so a growth of up to 64 MiB is tried
// without asking until one has failed (ask).
inline bool fits(const DevMemory &m, const Need *need, int n, bool ask) {
    const size_t page = (size_t)2 << 20;
    size_t more = 0, back = 0;
    for (int i = 0; i < n; ++i)
        if (need[i].bytes > need[i].buf->bytes) {
            more += (need[i].bytes + page - 1) / page * page;
            back += need[i].buf->bytes;
        }
    if (more == 0 || (!ask && more <= ((size_t)64 << 20))) return true;
    return more <= m.available() + back;
}

// The buffers of a job.  coarse (or nullptr) and plain: its needs in either form, of the
// same buffers; the coarse form holds two to four times the bytes per point and trial, so
// it is taken only where all of the job's buffers fit beside it, asked before anything is
// given up, so that a job that does not fit runs plain call after call without allocating.
// The first n_forms buffers are the ones whose size the form decides: where the plain form
// does not fit either, what they hold from other jobs is given back first.  ask: the
// handle's (see fits).
inline Growth job_buffers(const DevMemory &m, const Need *coarse, const Need *plain, int n,
                          int n_forms, bool *is_coarse, bool *ask) {
    *is_coarse = coarse != nullptr;
    if (coarse && fits(m, coarse, n, *ask)) {
        const Growth g = grow_all(m, coarse, n);
        if (g != NO_MEMORY) return g;
        *ask = true;
    }
    *is_coarse = false;
    Growth g = grow_all(m, plain, n);
    if (g != NO_MEMORY) return g;
    for (int i = 0; i < n_forms; ++i)
        if ((g = drop(m, *plain[i].buf)) != GROWN) return g;
    return grow_all(m, plain, n);
}

}  // namespace gce
