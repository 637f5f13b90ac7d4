"""The paths of the radial sort (one block, buckets, radix passes) answer alike:
what one reports the others report."""
import numpy as np
import pytest
import torch

from paper_1406_4254_gb300 import etics, inputs

pytestmark = pytest.mark.gpu

DTYPES = {"mixed": torch.float32, "fp64": torch.float64}
# one block up to 7168 particles, buckets up to 1867776, radix passes above
ONE_BLOCK, BUCKETS, RADIX = 7168, 1867776, 1867777


def oracle_order(pm):
    x = pm[:, :3]
    r2 = (x[:, 0] * x[:, 0] + x[:, 1] * x[:, 1]) + x[:, 2] * x[:, 2]
    return np.lexsort((np.arange(len(x)), r2))


def seen(pm, precision):
    return pm.astype(np.float32).astype(np.float64) if precision == "mixed" else pm


def shells(n, count, seed, same=False):
    """n particles on `count` thin shells (r^2 of a shell within a few ulps) or,
    same=True, at `count` points (equal r^2: ordered by index alone), shuffled."""
    rng = np.random.default_rng(seed)
    u = rng.normal(size=(n, 3))
    which = rng.integers(0, count, n)
    if same:
        u = rng.normal(size=(count, 3))[which]
    r = np.geomspace(0.05, 20.0, count)[which]
    pm = np.empty((n, 4))
    pm[:, :3] = u / np.linalg.norm(u, axis=1)[:, None] * r[:, None]
    pm[:, 3] = 1.0 / n
    return pm


def device(pm, precision):
    return torch.tensor(pm, dtype=DTYPES[precision], device="cuda")


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("bad", [float("nan"), float("inf"), -float("inf")])
@pytest.mark.parametrize("n", [1, 5000, ONE_BLOCK, ONE_BLOCK + 1, RADIX])
def test_order_reports_a_nonfinite_particle(n, bad, precision):
    x = device(inputs.hernquist(n, seed=3), precision)
    for at, column in ((0, 0), (n // 2, 2), (n - 1, 3)):   # the mass counts as well
        y = x.clone()
        y[at, column] = bad
        order = etics.radial_order(y)
        assert etics.get_error() == etics.ERR_NONFINITE, (at, column)
        assert int(order[-1]) == at       # such a particle sorts last
        etics.mex_field(y, 2)
        assert etics.get_error() == etics.ERR_NONFINITE, (at, column)
    etics.radial_order(x)
    assert etics.get_error() == 0


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("same", [False, True])
@pytest.mark.parametrize("n,count", [(7169, 1), (7169, 2), (12289, 3), (154625, 7), (300007, 40),
                                     (1048577, 150), (BUCKETS, 300)])
def test_order_of_crowded_buckets(n, count, same, precision):
    """Buckets beyond a block's room: their first places, the runs of every tile
    and the sort of the lot, at the edges of the tile and bucket sizes."""
    pm = shells(n, count, 17 + count, same)
    pm[: n // 20] = inputs.hernquist(n // 20, seed=5)      # and ordinary ones beside them
    got = etics.radial_order(device(pm, precision)).cpu().numpy()
    etics.check_error()
    assert np.array_equal(got, oracle_order(seen(pm, precision)))


@pytest.mark.parametrize("same", [False, True])
def test_crowded_buckets_cost_what_they_hold(same):
    """2^20 particles on 300 shells: every shell of 3500 is more than its bucket
    has room for.  A bucket's block then goes over its own members at most 13 times (a
    count of all digits, a placement for each of up to 12) in steps of 2048: about
    25 steps of a few us beside the ordinary sort of as many particles, so at most
    ten times that.  Reading all particles for each such bucket would take 4096
    steps."""
    n = 1 << 20

    def best(pm):
        x = device(pm, "mixed")
        for _ in range(3):
            etics.radial_order(x)
        t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        times = []
        for _ in range(10):
            t0.record()
            etics.radial_order(x)
            t1.record()
            torch.cuda.synchronize()
            times.append(t0.elapsed_time(t1))
        etics.check_error()
        return min(times)

    plain, crowded = best(inputs.hernquist(n, seed=1)), best(shells(n, 300, 2, same))
    print(f"plain {plain * 1e3:.0f} us, crowded {crowded * 1e3:.0f} us")
    assert crowded <= 10 * plain, (plain, crowded)


def test_workspace_does_not_shrink_with_more_particles():
    """A workspace sized for the largest call serves every smaller one, across
    the lines between the paths and between their tile and bucket sizes."""
    sizes = sorted({max(1, c + d) for c in (1, 1024, ONE_BLOCK, 154624, 309248, 463872, 1 << 20,
                                            (1 << 20) + 2048, 1300000, 1800000, BUCKETS, 2500000,
                                            4000000)
                    for d in (-1025, -1, 0, 1, 1025)})
    for method, l_max in ((etics.MEX, 0), (etics.MEX, 6), (etics.MEX, 10), (etics.SCF, 6)):
        for prec in (etics.MIXED, etics.FP64):
            need = [etics.workspace_bytes(n, 10, l_max, method, prec) for n in sizes]
            assert all(b >= a for a, b in zip(need, need[1:])), (method, l_max, prec)


def test_a_workspace_for_more_particles_is_accepted():
    n, most = 1800000, 2500000
    x = device(inputs.hernquist(n, seed=9), "mixed")
    ws = torch.empty(etics.workspace_bytes(most, 0, 4, etics.MEX, etics.MIXED) + 256,
                     dtype=torch.uint8, device="cuda")
    ref = etics.mex_field(x, 4)
    out = etics.mex_field(x, 4, ws=ws)
    etics.check_error()
    assert torch.equal(out, ref)


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("l_max", [0, 3, 5])
def test_scans_only_the_components_there_are(l_max, precision):
    """The workspace has room for 49 components per side up to l_max = 6; the
    carry scan of fewer must not read the rest of it, which nothing writes, nor
    write sums of that: the end of the workspace, which holds the last
    components' carries, stays as it was."""
    n = 100000
    x = device(inputs.hernquist(n, seed=5), precision)
    prec = etics.MIXED if precision == "mixed" else etics.FP64
    need = etics.workspace_bytes(n, 0, l_max, etics.MEX, prec)
    ws = torch.empty(need + 256, dtype=torch.uint8, device="cuda")
    ws.fill_(0x11)
    out = etics.mex_field(x, l_max, ws=ws)
    etics.check_error()
    assert torch.isfinite(out).all()
    at = (-ws.data_ptr()) % 256
    tiles = (n + 255) // 256
    missing = 49 - (l_max + 1) ** 2
    assert (ws[at + need - missing * tiles * 8:] == 0x11).all()


# ---- the radix path, and calls that no other test makes on it --------------------
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_radix_path_orders_long_runs(precision):
    """Above the buckets: two shell halves of 100000 equal keys each, sorted by
    one block across many tiles, 3000 copies of a point, runs of 17 to 300, and
    then nothing but coincident points and few distinct radii in sorted order."""
    from test_parity_mex import long_tie_particles
    shell, copies = 200000, 3000
    pm = long_tie_particles(shell, copies, RADIX - shell - copies, seed=41)
    assert len(pm) >= RADIX
    got = etics.radial_order(device(pm, precision)).cpu().numpy()
    etics.check_error()
    assert np.array_equal(got, oracle_order(seen(pm, precision)))
    few = shells(RADIX + 5, 300, 43, same=True)
    few = few[oracle_order(few)[::-1]]           # radii falling: every run reversed
    got = etics.radial_order(device(few, precision)).cpu().numpy()
    etics.check_error()
    assert np.array_equal(got, oracle_order(seen(few, precision)))


def test_both_paths_give_the_same_field():
    """One massless particle far outside takes the call to the radix path and
    changes nothing else (the carry scan is cut into other runs: FP64 roundings)."""
    pm = inputs.hernquist(BUCKETS, seed=21, axes=(1.0, 0.8, 0.6))
    pm[:, :3] = np.clip(pm[:, :3], -5e5, 5e5)
    far = np.concatenate([pm, [[1e6, 0.0, 0.0, 0.0]]])
    a = etics.mex_field(device(pm, "mixed"), 4)
    b = etics.mex_field(device(far, "mixed"), 4)
    etics.check_error()
    rel = (b[:-1] - a).norm(dim=1) / a.norm(dim=1)
    assert rel.max().item() < 1e-5 and rel.median().item() == 0.0


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("n", [RADIX, 1 << 21])
def test_radix_path_with_a_one_poll_lookback_bound_returns_and_reports(n, precision):
    x = device(inputs.hernquist(n, seed=11), precision)
    ref = etics.mex_field(x, 2)
    assert etics.get_error() == 0
    outcomes = []
    try:
        etics.set_wait_limit(1)
        for _ in range(20):
            etics.mex_field(x, 2)
            outcomes.append(etics.get_error())
            if etics.ERR_TIMEOUT in outcomes:
                break
    finally:
        etics.set_wait_limit(0)
    assert etics.ERR_TIMEOUT in outcomes, outcomes
    assert set(outcomes) <= {0, etics.ERR_TIMEOUT}, outcomes
    again = etics.mex_field(x, 2)
    assert etics.get_error() == 0
    assert torch.equal(again, ref)


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("n", [5000, 100003, RADIX])
def test_captured_call_gives_the_same_bits(n, precision):
    """One block, buckets and radix passes (the latter two behind a memset node)
    in a CUDA graph, replayed on other particles in the same buffers."""
    x = device(inputs.hernquist(n, seed=7), precision)
    y = device(inputs.hernquist(n, seed=8), precision)
    prec = etics.MIXED if precision == "mixed" else etics.FP64
    ws = torch.empty(etics.workspace_bytes(n, 0, 3, etics.MEX, prec) + 256, dtype=torch.uint8,
                     device="cuda")
    want = [etics.mex_field(x, 3), etics.mex_field(y, 3)]
    posm, out = x.clone(), torch.empty_like(x)
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        etics.mex_field(posm, 3, out=out, ws=ws)
    torch.cuda.current_stream().wait_stream(side)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        etics.mex_field(posm, 3, out=out, ws=ws)
    for particles, ref in zip((x, y, x), (want[0], want[1], want[0])):
        posm.copy_(particles)
        out.zero_()
        graph.replay()
        assert etics.get_error() == 0
        assert torch.equal(out, ref)
