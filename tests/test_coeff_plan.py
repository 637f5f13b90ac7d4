"""Host-side check of the plans of the mixed-precision SCF coefficient pass
(etics_scf_coeffs.cuh) for every (n_max, l_max) and a range of N: each harmonic
column belongs to exactly one bin of one level, the groups hold consecutive
bins within the warps of a block, the two shared-memory buffers and the FP64
sums fit, every group has blocks, their particle ranges cover [0, N) once, and
the workspace holds every block's partial sums."""
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
static int bad = 0;
#define CHECK(c) do { if (!(c)) { ++bad; printf("BAD %s rows %d l %d N %lld\n", #c, NR, l_max, (long long)N); } } while (0)
template <int NR> void check(int64_t N, int num_sms) {
    constexpr int CAP = PairShape<NR>::kCap, W = PairShape<NR>::kWarps;
    for (int l_max = 0; l_max <= kLmaxLimit; ++l_max) {
        const CoeffPlan p = make_coeff_plan(NR, l_max, CAP, W, N, num_sms);
        int seen[(kLmaxLimit + 1) * (kLmaxLimit + 1)] = {};
        CHECK(p.nbins <= kCoeffMaxBins && p.ngroups <= kCoeffMaxGroups && p.ngroups >= 1);
        for (int b = 0; b < p.nbins; ++b) {
            CHECK(p.bin[b].nc >= 1 && p.bin[b].nc <= CAP && p.bin[b].c0 + p.bin[b].nc <= 2 * p.bin[b].l + 1);
            CHECK(b == 0 || p.bin[b].l >= p.bin[b - 1].l);
            for (int c = 0; c < p.bin[b].nc; ++c) ++seen[p.bin[b].l * p.bin[b].l + p.bin[b].c0 + c];
        }
        for (int j = 0; j < (l_max + 1) * (l_max + 1); ++j) CHECK(seen[j] == 1);
        CHECK(p.warps == W);
        CHECK((coeff_tile<NR, 8>() <= W * 32 && coeff_tile<NR, kLmaxLimit>() <= W * 32));
        CHECK((l_max <= 8 ? coeff_smem<NR, 8>(p) : coeff_smem<NR, kLmaxLimit>(p)) <= 227 * 1024);
        CHECK((size_t)p.nblocks * p.slots * NR * CAP * 8 <= scf_coeff_plan_workspace<NR>(l_max, num_sms));
        int bin = 0, block = 0;
        for (int g = 0; g < p.ngroups; ++g) {
            const CoeffGroup& q = p.group[g];
            CHECK(q.bin0 == bin && q.block0 == block && q.nblocks >= 1 && q.teams >= 1);
            CHECK(q.nbins * q.teams <= p.warps && q.nbins <= p.slots);
            for (int b = q.bin0; b < q.bin0 + q.nbins; ++b)
                CHECK(p.bin[b].l >= q.l_lo && p.bin[b].l <= q.l_hi);
            bin += q.nbins;
            block += q.nblocks;
            const int64_t per = ((N + q.nblocks - 1) / q.nblocks + 1) / 2 * 2;
            CHECK(per * q.nblocks >= N);
        }
        CHECK(bin == p.nbins && block == p.nblocks);
    }
}
int main() {
    for (int sms : {152, 148, 80})
        for (int64_t N : {1LL, 2LL, 63LL, 65LL, 1000LL, 4219LL, 100003LL, 1LL << 20, (1LL << 30) - 1}) {
            check<3>(N, sms); check<5>(N, sms); check<7>(N, sms); check<9>(N, sms);
            check<11>(N, sms); check<13>(N, sms); check<15>(N, sms); check<17>(N, sms);
        }
    printf("%d bad\n", bad);
    return bad != 0;
}
"""


def test_coefficient_plans(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    src, exe = tmp_path / "plan.cu", tmp_path / "plan"
    src.write_text(PROGRAM)
    r = subprocess.run([nvcc, "-std=c++17", "--expt-relaxed-constexpr",
                        "-gencode", "arch=compute_103a,code=sm_103a", "-I", CSRC, "-I",
                        os.path.join(ROOT, "include"), "-o", str(exe), str(src)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    out = subprocess.run([str(exe)], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout[-2000:]
