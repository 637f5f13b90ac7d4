"""Host-side check of how many particles' FP32 partial sums the general SCF
coefficient kernel adds up before they enter FP64: at most 2048, the span of the
register-tile kernel it replaced."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(ROOT, "paper_1406_4254_gb300", "csrc")

PROGRAM = r"""
#include "etics_scf_coeffs.cuh"
#include <cstdio>
using namespace etics;
template <int NR, int LMU> int span() {
    const int s = coeff_flush_tiles<NR, LMU>() * coeff_tile<NR, LMU>();
    std::printf("%d %d %d\n", NR, LMU, s);
    return s < 1 || s > 2048;
}
template <int NR> int both() { return span<NR, 8>() + span<NR, kLmaxLimit>(); }
int main() {
    return both<3>() + both<5>() + both<7>() + both<9>() + both<11>() + both<13>() + both<15>() +
           both<17>();
}
"""


def test_partial_sums_span_at_most_2048_particles(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    src, exe = tmp_path / "flush.cu", tmp_path / "flush"
    src.write_text(PROGRAM)
    r = subprocess.run([nvcc, "-std=c++17", "--expt-relaxed-constexpr",
                        "-gencode", "arch=compute_103a,code=sm_103a", "-I", CSRC, "-I",
                        os.path.join(ROOT, "include"), "-o", str(exe), str(src)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    out = subprocess.run([str(exe)], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout
