"""Sizes at the edges of the kernels' tiles, against the FP64 oracle: one
particle more or less than a tile, a thread's pair or a bucket holds, and
the smallest sizes.  Tolerances are those of the parity tests (eq. 23 errors
of the mixed path; FP64 relative to the largest force, as in their edge
cases: with few particles single forces nearly vanish)."""
import numpy as np
import pytest

import oracle
from helpers import device_particles, hernquist, rounded
from paper_1406_4254_gb300 import etics

pytestmark = pytest.mark.gpu


def close(o, acc_ref, pot_ref, precision, what):
    tol = 1e-11 if precision == "fp64" else 2e-5
    amax = np.max(np.linalg.norm(acc_ref, axis=1))
    assert np.max(np.abs(o[:, :3] - acc_ref)) <= tol * amax, what
    assert np.max(np.abs(o[:, 3] - pot_ref)) <= tol * np.max(np.abs(pot_ref)), what


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("l_max", [0, 3, 6, 7, 10])
def test_mex_tile_edges(precision, l_max):
    """MEX tiles hold 256 particles, two per thread; 0, 3, 6: one level group
    with 2, 32 and 98 components (a part of a warp, whole warps, a leftover
    pair), 7 and 10: two and three groups."""
    for n in (2, 255, 256, 257, 511, 513, 769):
        pm = hernquist(n, seed=n)
        ref = rounded(pm, precision)
        acc, pot, _ = oracle.mex_field(ref[:, :3], ref[:, 3], l_max)
        o = etics.mex_field(device_particles(pm, precision), l_max).cpu().numpy()
        etics.check_error()
        close(o, acc, pot, precision, (n, l_max))


def order_of(pm):
    x = pm[:, :3]
    r2 = (x[:, 0] * x[:, 0] + x[:, 1] * x[:, 1]) + x[:, 2] * x[:, 2]
    return np.lexsort((np.arange(len(x)), r2))


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_radial_order_across_the_sort_paths(precision):
    """The order is exact on both sides of every line the sort draws by size:
    one block up to 7168, one to eight particles per thread (154624 each) in
    the partition, buckets of mean 1024 up to 2^20 and of mean 2048 up
    to 1867776, the radix passes above; particles already in radial order, in two
    interleaved populations, and with one radius crowding (more equal keys
    than a bucket or a bin holds)."""
    rng = np.random.default_rng(3)
    for n in (1023, 7167, 7168, 7169, 8193, 9217, 154625, (1 << 18) + 1, 400001, 800001, (1 << 20) + 1,
              1867776, 1867777):
        pm = hernquist(n, seed=5)
        if n == 8193:
            pm = pm[order_of(pm)]                      # sorted already
        if n == 9217:
            pm[::2, :3] *= 1e-3                        # two interleaved populations
        if n == (1 << 18) + 1:
            u = rng.normal(size=(20000, 3))            # a shell: r^2 within a few ulps of 4
            pm[1000:21000, :3] = 2.0 * u / np.linalg.norm(u, axis=1, keepdims=True)
            pm[30000:30300, :3] = pm[30000, :3]        # one point, 300 times
        got = etics.radial_order(device_particles(pm, precision)).cpu().numpy()
        etics.check_error()
        assert np.array_equal(got, order_of(rounded(pm, precision))), n


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("basis", [0, 1])
def test_scf_field_edges(precision, basis):
    """The field pass takes two particles per thread (one in FP64), two radial
    rows per round and, while a quarter of the threads would do (about 38000
    particles at l_max <= 6, 19000 above 8), splits the levels from 2 up over
    four warps: odd counts, odd and even n_max, either side of the split, each
    register class of l_max, and (10, 6), (14, 8) with their unrolled rows."""
    sizes = [(1, 0, 0), (2, 1, 1), (3, 2, 2), (65, 0, 4), (257, 3, 6), (303, 10, 6), (304, 11, 7),
             (305, 14, 8), (1215, 5, 10), (77, 2, 14), (20001, 2, 9), (38911, 10, 6), (38913, 10, 6)]
    for n, n_max, l_max in sizes:
        pm = hernquist(n, seed=n)
        ref = rounded(pm, precision)
        c = oracle.scf_coeffs(ref[:, :3], ref[:, 3], n_max, l_max, basis=basis)
        acc, pot = oracle.scf_field(ref[:, :3], n_max, l_max, c, basis=basis)
        d = device_particles(pm, precision)
        o, _ = etics.scf_force(d, n_max, l_max, basis=basis)
        etics.check_error()
        close(o.cpu().numpy(), acc, pot, precision, (n, n_max, l_max))


@pytest.mark.parametrize("basis", [0, 1])
@pytest.mark.parametrize("nl", [(10, 6), (14, 8), (0, 0), (1, 1), (8, 4), (12, 5), (16, 14)])
def test_scf_coefficient_tile_edges(nl, basis):
    """Around the tiles of the mixed-precision coefficient kernels (192 to 576
    particles, pairs of particles per lane) and their flushes.  Tolerance, of
    the largest coefficient: the parity tests' 2e-6, or what the roundings of
    one particle's value may add up to (5 per level for the harmonic and the
    radial prefactor, 2 per row, 10 for radius, xi and direction), as with few
    particles they do not average out."""
    n_max, l_max = nl
    for n in (1, 2, 63, 191, 193, 383, 511, 513, 575, 577, 1153, 90001):
        pm = hernquist(n, seed=n)
        ref = rounded(pm, "mixed")
        want = oracle.scf_coeffs(ref[:, :3], ref[:, 3], n_max, l_max, basis=basis)
        got = etics.scf_coeffs(device_particles(pm, "mixed"), n_max, l_max, basis=basis).cpu().numpy()
        etics.check_error()
        tol = max(2e-6, (10 + 5 * l_max + 2 * n_max) * 2.0 ** -24)
        assert np.max(np.abs(got.reshape(want.shape) - want)) <= tol * np.max(np.abs(want)), n


@pytest.mark.parametrize("tile", [0, 64, 320])
def test_batch_step_edges(tile):
    """The mixed-precision batch takes 256 particles a step, adds its FP32 sums
    in FP64 every 16 steps and walks chunks of 2 to 16 tiles of the plan: sizes around
    each, odd sizes, and every l_max (a layout of its own).  Tolerance as above."""
    sizes = [1, 2, 255, 256, 257, 511, 513, 1023, 1025, 4095, 4096, 4097, 5119, 5121, 8191, 8193, 12289]
    n_maxes = [14 - i % 15 for i in range(len(sizes))]
    l_maxes = [i % 9 for i in range(len(sizes))]
    pms = [hernquist(n, seed=n) for n in sizes]
    tuning = etics.BatchTuning(tile, 0, 0, 0) if tile else None
    plan = etics.BatchPlan(sizes, n_maxes, l_maxes, precision=etics.MIXED, tuning=tuning)
    d = device_particles(np.concatenate(pms), "mixed")
    packed, out = etics.scf_batch(d, plan)
    etics.check_error()
    out = out.cpu().numpy()
    first = 0
    for i, (n, n_max, l_max) in enumerate(zip(sizes, n_maxes, l_maxes)):
        ref = rounded(pms[i], "mixed")
        want = oracle.scf_coeffs(ref[:, :3], ref[:, 3], n_max, l_max)
        got = plan.coeffs_of(packed, i).cpu().numpy().reshape(want.shape)
        tol = max(2e-6, (10 + 5 * l_max + 2 * n_max) * 2.0 ** -24)
        assert np.max(np.abs(got - want)) <= tol * np.max(np.abs(want)), (n, n_max, l_max)
        acc, pot = oracle.scf_field(ref[:, :3], n_max, l_max, want)
        close(out[first:first + n], acc, pot, "mixed", (n, n_max, l_max))
        first += n
