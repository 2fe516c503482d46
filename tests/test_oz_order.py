"""The MMAs of one K block of the digit-slice GEMM (csrc/oz_order.h, the header
the kernel issues from): any two that touch a common accumulator column have the
same base and width, which is the only case in which tcgen05.mma instructions are
ordered; every digit product of the kept levels is formed once, at its level; B
planes outside the eight digits are the zero planes only.  Host code alone."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1606_06790_gb300", "csrc")
MAIN = r"""
#include <cstdio>
#include "oz_order.h"
int main() {
  using namespace idmrg;
  printf("%d %d\n", OZ_PLANES, OZ_ZERO);
  oz_for_each_mma([](int p, int q0, int level, int n) { printf("%d %d %d %d\n", p, q0, level, n); });
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="no host compiler")
def test_mmas_of_a_k_block(tmp_path):
    src, exe = tmp_path / "main.cpp", tmp_path / "main"
    src.write_text(MAIN)
    subprocess.run(["g++", "-std=c++17", "-I" + CSRC, str(src), "-o", str(exe)], check=True)
    lines = [tuple(map(int, x.split())) for x in subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.splitlines()]
    planes, zero = lines[0]
    mmas = lines[1:]
    products, first = [], set()
    for p, q0, level, n in mmas:
        assert 0 <= p < planes and level >= 0 and level + n <= planes
        assert n * 64 <= 256  # the widest MMA
        assert -zero <= q0 and q0 + n <= planes
        products += [(p, q0 + j, level + j) for j in range(n) if q0 + j >= 0]
        # the first MMA of a window overwrites it (p = 0), the others add
        assert (level in first) == (p > 0)
        first.add(level)
    assert sorted(products) == sorted((p, q, p + q) for p in range(planes) for q in range(planes - p))
    for i, (_, _, a, na) in enumerate(mmas):
        for _, _, b, nb in mmas[:i]:
            assert (a, na) == (b, nb) or a + na <= b or b + nb <= a
