"""Integer helpers of the FP64 mode's fixed point (sre_tile.cuh), compiled for
the host and compared with Python integers."""
import os
import shutil
import subprocess

import pytest

from paper_2512_24685_gb300 import build

SOURCE = r"""
#include <stdio.h>
#include "sre_tile.cuh"
int main() {
    long long a;
    int q, few;
    while (scanf("%lld %d %d", &a, &q, &few) == 3)
        printf("%lld\n", few ? sre::dev::fx_shift_few(a, q) : sre::dev::fx_shift(a, q));
    return 0;
}
"""


@pytest.fixture(scope="module")
def shifted(tmp_path_factory):
    if not (shutil.which("nvcc") or os.path.exists("/usr/local/cuda/bin/nvcc")):
        pytest.skip("needs nvcc")
    d = tmp_path_factory.mktemp("fx")
    src, exe = d / "shift.cu", d / "shift"
    src.write_text(SOURCE)
    subprocess.run([build.nvcc(), "-std=c++17", "-O2", *build.ARCH, "-I", build.CSRC, str(src), "-o", str(exe)],
                   check=True)

    def run(pairs, few=0):
        text = "".join(f"{a} {q} {few}\n" for a, q in pairs)
        return list(map(int, subprocess.run([str(exe)], input=text, capture_output=True, text=True,
                                            check=True).stdout.split()))

    return run


def test_shift_rounds_half_up_over_the_whole_range(shifted):
    top = (1 << 63) - 1
    values = [s * v for s in (1, -1) for v in (0, 1, 3, 12345, 1 << 40, int(0.997 * 2 ** 63), top - 511, top)]
    pairs = [(a, q) for a in values for q in range(-2, 70)]
    want = [a if q <= 0 else 0 if q > 62 else (a + (1 << (q - 1))) >> q for a, q in pairs]
    assert shifted(pairs) == want


def test_short_shift_rounds_alike_below_the_top(shifted):
    top = (1 << 63) - (1 << 10)
    pairs = [(s * v, q) for s in (1, -1) for v in (0, 1, 7, 128, 99991, 1 << 50, top - 1, top) for q in range(0, 9)]
    assert shifted(pairs, 1) == shifted(pairs)
