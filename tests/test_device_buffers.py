"""The growth of a context's device buffers (csrc/devbuf.h) with a host allocator that fails on demand: a captured
launch sequence is keyed by the buffers' generation, so the generation has to move whenever an address it may hold is
given up."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1807_02718_gb300", "csrc")

HEAD = r'''
#include <cstdio>
#include <cstdlib>
#include "devbuf.h"
struct Memory {
    size_t room = 1 << 20;   // bytes the device has left
    int live = 0;
    int alloc(void **p, size_t n) {
        if (n > room) return 2;
        room -= n;
        size_t *q = static_cast<size_t *>(std::malloc(n + 16));
        *q = n;
        *p = q;
        ++live;
        return 0;
    }
    void release(void *p) {
        room += *static_cast<size_t *>(p);
        std::free(p);
        --live;
    }
};
#define CHECK(x) do { if (!(x)) { std::printf("line %d: %s\n", __LINE__, #x); return 1; } } while (0)
'''

CASES = {
    # an address is kept while the buffer is large enough
    "keeps": r'''
    Memory m; fh::DevBuf b; long long g = 0;
    CHECK(fh::grow(m, b, 1000, g) == 0 && b.cap >= 1000 && g == 1);
    void *p = b.p;
    CHECK(fh::grow(m, b, 1000, g) == 0 && fh::grow(m, b, 10, g) == 0 && b.p == p && g == 1 && m.live == 1);
''',
    # growth fails after the old buffer went: no launch captured before may be replayed, whatever the next call's size
    "growth fails": r'''
    Memory m; fh::DevBuf b; long long g = 0;
    CHECK(fh::grow(m, b, 1000, g) == 0);
    const long long captured = g;
    CHECK(fh::grow(m, b, 1 << 21, g) == 2 && !b.p && b.cap == 0 && m.live == 0);
    CHECK(g != captured);
    m.room = 0;                                    // now the smaller size cannot be had either
    CHECK(fh::grow(m, b, 1000, g) == 2 && !b.p && g != captured);
    m.room = 1 << 20;
    CHECK(fh::grow(m, b, 1000, g) == 0 && b.p && g != captured);
''',
    # a buffer that can be done without makes room for one that cannot, and its address is given up with it
    "spare": r'''
    Memory m; fh::DevBuf b, c, spare; long long g = 0;
    CHECK(fh::grow(m, spare, 600000, g, &spare) == 0 && fh::grow(m, b, 300000, g, &spare) == 0 && spare.p && g == 2);
    CHECK(fh::grow(m, c, 500000, g, &spare) == 0 && c.p && b.p && !spare.p && spare.cap == 0 && g == 4);
    CHECK(fh::grow(m, spare, 600000, g, &spare) == 2 && !spare.p && b.p && c.p && g == 4);
    CHECK(fh::grow(m, spare, 100000, g, &spare) == 0 && fh::grow(m, b, 1 << 21, g, &spare) == 2);
    CHECK(!b.p && !spare.p && c.p && g == 7 && m.live == 1);
''',
}


@pytest.mark.parametrize("name", list(CASES))
def test_growth(name, tmp_path):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(HEAD + "int main() {" + CASES[name] + "    return 0;\n}\n")
    subprocess.run(["g++", "-std=c++17", "-Wall", "-Werror", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
