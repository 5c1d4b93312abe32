"""Bookkeeping of a served case's device memory (csrc/slab.h), compiled as
plain C++: carved blocks never overlap, start on multiples of 256 bytes, freed
neighbours merge, a full or absent slab gives null."""
import shutil
import subprocess

import pytest

from paper_2505_17287_gb300 import build

SRC = r"""
#include <stdio.h>
#include <stdlib.h>
#include <vector>
#include "slab.h"
#define CHECK(e) do { if (!(e)) { printf("line %d: %s\n", __LINE__, #e); return 1; } } while (0)
int main() {
    using namespace ibm;
    Slab s;
    CHECK(!s.take(1));                       // no slab
    s.open(nullptr, 1 << 20);                // refused by the pool
    CHECK(!s.take(1) && !s.holds(nullptr));
    char *base = (char *)0x100000;           // (never dereferenced)
    s.open(base, 4096 + 100);                // cut down to a multiple of 256
    CHECK(s.bytes == 4096);
    void *a = s.take(1000), *b = s.take(256), *c = s.take(257), *d = s.take(2304);
    CHECK(a == base && b == base + 1024 && c == base + 1280 && d == base + 1792);
    CHECK(s.ranges.empty() && !s.take(1));   // full
    CHECK(s.holds(base) && s.holds(base + 4095) && !s.holds(base + 4096) && !s.holds(base - 1));
    s.give(a, 1000);
    s.give(c, 257);
    CHECK(s.ranges.size() == 2 && !s.take(1025));   // 1536 bytes free, in two ranges
    s.give(b, 256);                          // joins both neighbours
    CHECK(s.ranges.size() == 1 && s.ranges[0] == 1792);
    CHECK(s.take(1025) == base);             // and is used again
    s.give(base, 1025);
    s.give(d, 2304);
    CHECK(s.ranges.size() == 1 && s.ranges[0] == 4096);
    // random blocks against a map of bytes
    srand(7);
    const size_t N = 1 << 16;
    s.open(base, N);
    std::vector<char> used(N, 0);
    struct B { char *p; size_t n; };
    std::vector<B> live;
    for (int it = 0; it < 20000; ++it) {
        if (rand() % 2) {
            const size_t n = 1 + rand() % 4000, r = (n + 255) / 256 * 256;
            char *p = (char *)s.take(n);
            if (p) {
                const size_t o = p - base;
                CHECK(o % 256 == 0 && o + r <= N);
                for (size_t q = o; q < o + r; ++q) { CHECK(!used[q]); used[q] = 1; }
                live.push_back({p, n});
            } else {   // no free run is long enough
                size_t run = 0;
                for (size_t q = 0; q < N; ++q) { run = used[q] ? 0 : run + 1; CHECK(run < r); }
            }
        } else if (!live.empty()) {
            const size_t k = rand() % live.size(), o = live[k].p - base, r = (live[k].n + 255) / 256 * 256;
            s.give(live[k].p, live[k].n);
            for (size_t q = o; q < o + r; ++q) used[q] = 0;
            live[k] = live.back();
            live.pop_back();
        }
    }
    for (auto &l : live) s.give(l.p, l.n);
    CHECK(s.ranges.size() == 1 && s.ranges[0] == N);
    return 0;
}
"""


def test_slab_carves_merges_and_refuses(tmp_path):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no g++")
    src, exe = tmp_path / "slab.cpp", tmp_path / "slab"
    src.write_text(SRC)
    subprocess.run([cxx, "-std=c++17", "-O1", "-I", build.CSRC, "-o", str(exe), str(src)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
