"""The handle's scratch buffer, compiled on the host over a fake device memory: a larger optional request that
cannot be had leaves the buffer where it is (no synchronisation, no free, no retry on every call), a buffer that
a captured graph uses is not freed by a later run that needs a larger one, and a request that nothing stands in
for gets memory whenever there is any."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2002_05983_gb300", "csrc")

PROGRAM = r'''
#include <cassert>
#include <cstdio>
#include <map>
#include "scratch.h"
struct Fake {
    const int oom = -4;
    std::map<void *, size_t> live;
    size_t cap, used = 0, next = 0x1000;
    int allocs = 0, syncs = 0, frees = 0;
    explicit Fake(size_t c) : cap(c) {}
    int alloc(void **p, size_t n) {
        ++allocs;
        if (used + n > cap) return oom;
        *p = reinterpret_cast<void *>(next);
        next += 0x1000;
        live[*p] = n;
        used += n;
        return 0;
    }
    int sync() { ++syncs; return 0; }
    int free(void *p) { assert(live.count(p)); ++frees; used -= live[p]; live.erase(p); return 0; }
};
using namespace stn;
int main()
{
    bool ok;
    {   // two padded grids do not fit, one grid does: the grid stays put over repeated runs
        Fake m(150);
        Scratch s;
        assert(scratch_want(s, 200, 0, m, &ok) == 0 && !ok);
        assert(scratch_need(s, 100, 0, m) == 0);
        void *p = s.p;
        const int allocs = m.allocs;
        for (int i = 0; i < kScratchRetry - 1; ++i) {
            assert(scratch_want(s, 200, 0, m, &ok) == 0 && !ok);
            assert(scratch_need(s, 100, 0, m) == 0 && s.p == p);
        }
        assert(m.allocs == allocs && m.syncs == 0 && m.frees == 0);
        assert(scratch_want(s, 200, 0, m, &ok) == 0 && !ok);   // the last skipped one
        m.cap = 1000;
        assert(scratch_want(s, 200, 0, m, &ok) == 0 && ok && s.bytes == 200 && m.used == 200);   // tried again
        assert(scratch_need(s, 100, 0, m) == 0 && s.bytes == 200);
        assert(scratch_want(s, 150, 0, m, &ok) == 0 && ok && m.live.size() == 1);
    }
    {   // a smaller optional size is tried although a larger one was refused
        Fake m(150);
        Scratch s;
        assert(scratch_want(s, 200, 0, m, &ok) == 0 && !ok);
        assert(scratch_want(s, 120, 0, m, &ok) == 0 && ok);
    }
    {   // buffers of captured graphs outlive growth of either kind
        Fake m(10000);
        Scratch s;
        assert(scratch_need(s, 100, 0, m) == 0);
        void *a = s.p;
        s.captured = true;
        assert(scratch_want(s, 200, 0, m, &ok) == 0 && ok && m.live.count(a) && !s.captured && m.frees == 0);
        void *b = s.p;
        s.captured = true;
        assert(scratch_need(s, 300, 0, m) == 0 && m.live.count(a) && m.live.count(b));
        assert(scratch_need(s, 400, 0, m) == 0 && m.live.size() == 3);   // the 300 was not captured
        assert(scratch_need(s, 400, 1, m) == 0 && s.dev == 1 && m.live.size() == 3);
        scratch_free_kept(s, m);
        assert(m.live.size() == 1 && !s.kept);
    }
    {   // a run without an alternative still gets the memory that kept buffers hold
        Fake m(500);
        Scratch s;
        assert(scratch_need(s, 100, 0, m) == 0);
        s.captured = true;
        assert(scratch_want(s, 450, 0, m, &ok) == 0 && !ok && s.bytes == 100 && s.captured);
        assert(scratch_need(s, 450, 0, m) == 0 && s.bytes == 450 && m.used == 450 && m.syncs == 1);
        Fake t(50);
        Scratch u;
        assert(scratch_need(u, 100, 0, t) == t.oom && !u.p);
    }
    std::puts("ok");
}
'''


def test_scratch(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no host C++ compiler")
    src = tmp_path / "scratch.cpp"
    src.write_text(PROGRAM)
    exe = tmp_path / "scratch"
    subprocess.run([cxx, "-std=c++17", "-I" + CSRC, str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout == "ok\n"
    with open(os.path.join(CSRC, "stencil_api.cu")) as fh:
        api = fh.read()
    assert "ensure_scratch" not in api and "cudaFree(h->scratch)" not in api   # the runs use it
