// The device buffer a handle keeps for the grids between passes (host code without CUDA types; Memory
// gives int alloc(void **, size_t), int sync() and int free(void *), 0 on success, oom on lack of memory).
//
// A graph captured from a run holds the buffer's address, so a buffer used under capture is not freed
// when a later run needs a larger one: it is kept until the handle is destroyed, or until a run that cannot
// do without the larger one finds no other memory.
#pragma once
#include <cstddef>
#include <new>

namespace stn {

struct Scratch {
    void *p = nullptr;
    size_t bytes = 0;
    int dev = -1;
    bool captured = false;         // a captured graph uses p
    struct Kept {
        void *p;
        Kept *next;
    } *kept = nullptr;             // earlier buffers that captured graphs use
    size_t refused = 0;            // the last optional size that could not be had
    int skip = 0;                  // optional requests of at least that size not to try

    bool fits(size_t n, int d) const { return p && bytes >= n && dev == d; }
};

constexpr int kScratchRetry = 64;   // optional requests between two failing allocations

// Gives up p: kept where a captured graph uses it, else freed once the device's work is done.
template <class Memory> int scratch_drop(Scratch &s, Memory &m)
{
    if (!s.p) return 0;
    if (s.captured) {
        auto *k = new (std::nothrow) Scratch::Kept{s.p, s.kept};
        if (!k) return m.oom;
        s.kept = k;
    } else {
        int rc = m.sync();
        if (!rc) rc = m.free(s.p);
        if (rc) return rc;
    }
    s.p = nullptr;
    s.bytes = 0;
    s.captured = false;
    return 0;
}

template <class Memory> void scratch_free_kept(Scratch &s, Memory &m)
{
    while (s.kept) {
        Scratch::Kept *k = s.kept;
        s.kept = k->next;
        m.free(k->p);
        delete k;
    }
}

// At least n bytes on device d, which the run cannot do without.
template <class Memory> int scratch_need(Scratch &s, size_t n, int d, Memory &m)
{
    if (s.fits(n, d)) return 0;
    int rc = scratch_drop(s, m);
    if (rc) return rc;
    void *q = nullptr;
    rc = m.alloc(&q, n);
    if (rc == m.oom && s.kept) {
        rc = m.sync();
        if (rc) return rc;
        scratch_free_kept(s, m);
        rc = m.alloc(&q, n);
    }
    if (rc) return rc;
    s.p = q;
    s.bytes = n;
    s.dev = d;
    return 0;
}

// As scratch_need for a route that another one can stand in for: where there is no memory, p stays as it
// is (what stands in uses it), nothing waits, and the next requests of this size do not try again.
template <class Memory> int scratch_want(Scratch &s, size_t n, int d, Memory &m, bool *ok)
{
    *ok = s.fits(n, d);
    if (*ok) return 0;
    if (s.refused && n >= s.refused && s.skip > 0) {
        --s.skip;
        return 0;
    }
    void *q = nullptr;
    int rc = m.alloc(&q, n);
    if (rc == m.oom) {
        s.refused = n;
        s.skip = kScratchRetry;
        return 0;
    }
    if (rc) return rc;
    rc = scratch_drop(s, m);
    if (rc) {
        m.free(q);
        return rc;
    }
    s.p = q;
    s.bytes = n;
    s.dev = d;
    s.refused = 0;
    *ok = true;
    return 0;
}

}  // namespace stn
