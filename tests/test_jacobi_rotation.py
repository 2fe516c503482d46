"""The rotation of the FP32 tournament (csrc/jacobi_rotation.h, which the kernel
includes) against 64 bits: b - a, z, z^2 + 1 (halved by the root), the root, the
sum and the quotient round once each, so t is within 5.5 * 2^-24 of the exact angle
for the same a, b, g, and the relative overlap within 4 * 2^-24.  Overlaps at
most tol, zero columns and non-finite input are no rotation.  Host code alone."""
import os
import shutil
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1606_06790_gb300", "csrc")
MAIN = r"""
#include <cstdio>
#include "jacobi_rotation.h"
int main() {
  float x[4];
  while (fread(x, 4, 4, stdin) == 4) {
    float y[5] = {0, 0, 0, 0, 0};
    y[0] = idmrg::js_rotation(x[0], x[1], x[2], x[3], y[1], y[2], y[3], y[4]) ? 1.0f : 0.0f;
    fwrite(y, 4, 5, stdout);
  }
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="no host compiler")
def test_rotation_against_64_bits(tmp_path):
    src, exe = tmp_path / "main.cpp", tmp_path / "main"
    src.write_text(MAIN)
    subprocess.run(["g++", "-std=c++17", "-O2", "-I" + CSRC, str(src), "-o", str(exe)], check=True)

    def call(x):
        out = subprocess.run([str(exe)], input=x.astype(np.float32).tobytes(), capture_output=True, check=True).stdout
        return np.frombuffer(out, dtype=np.float32).reshape(-1, 5).astype(np.float64)

    rng = np.random.default_rng(7)
    n = 200000
    a = 10.0 ** rng.uniform(-20, 0, n)
    b = np.where(rng.random(n) < 0.5, a * (1 + rng.uniform(-1e-3, 1e-3, n)), 10.0 ** rng.uniform(-20, 0, n))
    x = np.stack([a, b, np.sqrt(a * b) * 10.0 ** rng.uniform(-6, 0, n) * rng.choice([-1, 1], n), np.full(n, 2e-6)], 1).astype(np.float32)
    y = call(x)
    a, b, g, tol = x.astype(np.float64).T
    ratio = np.abs(g) / np.sqrt(a * b)
    z = (b - a) / (2 * g)
    t = np.where(z == 0, 1.0, np.sign(z) / (np.abs(z) + np.hypot(z, 1)))
    on = y[:, 0] == 1
    clear = np.abs(ratio / tol - 1) > 1e-6
    # (angles below 2^-126 and those whose z^2 overflows are no rotation)
    assert np.all(on[clear & (np.abs(z) < 1e18)] == (ratio > tol)[clear & (np.abs(z) < 1e18)])
    assert np.max(np.abs(y[on, 1] / ratio[on] - 1)) <= 4 * 2.0**-24
    assert np.max(np.abs(y[on, 2] / t[on] - 1)) <= 5.5 * 2.0**-24
    assert np.max(np.abs(y[on, 3] ** 2 + y[on, 4] ** 2 - 1)) <= 8 * 2.0**-24
    assert not np.any(call(np.array([[0, 1, 0, 0], [1, 0, 0.1, 0], [1, 1, np.nan, 0], [1, 1, 1e-7, 1e-6]]))[:, 0])
