"""Host-side check of the radial sort's 64-bit keys: for FP32 coordinates the
integer evaluation of the FP64 bit pattern of r^2 = (x*x + y*y) + z*z
(etics_r2.h, plain C++) equals FP64 arithmetic bit for bit, over random bit
patterns, equal and widely different exponents, short mantissas (ties of the
roundings) and zeros; subnormal and non-finite coordinates are left to FP64."""
import os
import shutil
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1406_4254_gb300", "csrc")

PROGRAM = r"""
#include "etics_r2.h"
#include <cstdio>
int main() {
    uint32_t c[3];
    while (std::fread(c, 4, 3, stdin) == 3) {
        uint64_t bits = 0;
        const uint64_t ok = etics::r2_bits_from_f32(c[0], c[1], c[2], bits) ? 1 : 0;
        std::fwrite(&ok, 8, 1, stdout);
        std::fwrite(&bits, 8, 1, stdout);
    }
    return 0;
}
"""


def coordinates(rng, n):
    exps = rng.integers(64, 190, (n, 3))
    near = 127 + rng.integers(-3, 4, (n, 3))
    apart = 127 - np.arange(3)[None, :] * 13 + rng.integers(-2, 3, (n, 3))
    frac = rng.integers(0, 1 << 23, (n, 3))
    short = frac & ~((1 << rng.integers(0, 23, (n, 3))) - 1)
    zero = np.where(rng.random((n, 3)) < 0.4, 0, (near << 23) | frac)
    anything = rng.integers(0, 1 << 32, (n, 3), dtype=np.uint64)
    parts = [(exps << 23) | frac, (near << 23) | frac, (apart << 23) | frac, (near << 23) | short,
             (apart << 23) | short, zero, anything]
    out = np.concatenate([np.asarray(p).astype(np.uint64) for p in parts]).astype(np.uint32)
    return out ^ (rng.integers(0, 2, out.shape).astype(np.uint32) << 31)


def test_r2_bits_equal_fp64(tmp_path):
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("g++ not available")
    src, exe = tmp_path / "r2.cpp", tmp_path / "r2"
    src.write_text(PROGRAM)
    r = subprocess.run([gxx, "-std=c++17", "-O1", "-I", CSRC, "-o", str(exe), str(src)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    c = coordinates(np.random.default_rng(7), 200000)
    got = np.frombuffer(subprocess.run([str(exe)], input=c.tobytes(), capture_output=True,
                                       check=True).stdout, dtype=np.uint64).reshape(-1, 2)
    mag = c & 0x7fffffff
    usual = ((mag == 0) | ((mag >= 0x00800000) & (mag < 0x7f800000))).all(axis=1)
    assert np.array_equal(got[:, 0] == 1, usual)
    x = c.view(np.float32).astype(np.float64)
    with np.errstate(all="ignore"):
        r2 = (x[:, 0] * x[:, 0] + x[:, 1] * x[:, 1]) + x[:, 2] * x[:, 2]
    assert np.array_equal(got[usual, 1], r2.view(np.uint64)[usual])
