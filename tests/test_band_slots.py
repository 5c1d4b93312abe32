"""Entries of the near-body band's neighbour-major arrays (band_slot() in
csrc/common.cuh), evaluated on the host: exact and inside the arrays also
where eight entries a row no longer fit 32 bits, and used by every access."""
import os
import re
import subprocess

import pytest

from paper_2505_17287_gb300 import build

SRC = r"""
#include "common.cuh"
int main() {
    long long a[3];
    while (scanf("%lld %lld %lld", &a[0], &a[1], &a[2]) == 3)
        printf("%llu\n", (unsigned long long)ibm::band_slot((int)a[0], (int)a[1], (int)a[2]));
    return 0;
}
"""


def test_band_slots_past_32_bits(tmp_path):
    if not os.path.exists(build.NVCC):
        pytest.skip("no nvcc")
    src, exe = tmp_path / "slots.cu", tmp_path / "slots"
    src.write_text(SRC)
    subprocess.run([build.NVCC, *build.COMMON, "-I", build.CSRC, "-o", str(exe), str(src)], check=True)
    q = [(nb, m, r) for nb in (1, 16384, 2**28 - 1, 2**28, 2**28 + 1, 300_000_000) for m in range(8)
         for r in {0, nb // 2, nb - 1}]
    out = subprocess.run([str(exe)], input="\n".join("%d %d %d" % t for t in q), capture_output=True, text=True,
                         check=True).stdout.split()
    assert [int(x) for x in out] == [m * nb + r for nb, m, r in q]
    assert all(int(x) < 8 * nb for x, (nb, _, _) in zip(out, q))


def test_no_other_slot_arithmetic_in_the_band():
    text = open(os.path.join(build.CSRC, "band.cuh")).read()
    assert not re.search(r"\bm\s*\*\s*(\(size_t\)\s*)?(b\.)?nb\b", text)
