"""The mixed-precision field pass of the smallest expansions."""
import pytest
import torch

from paper_1406_4254_gb300 import etics, inputs

pytestmark = pytest.mark.gpu


def _best(call, calls=10):
    for _ in range(3):
        call()
    t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    times = []
    for _ in range(12):
        t0.record()
        for _ in range(calls):
            call()
        t1.record()
        torch.cuda.synchronize()
        times.append(t0.elapsed_time(t1) / calls)
    return min(times)


@pytest.mark.parametrize("n_max,l_max", [(0, 0), (1, 0), (2, 2), (16, 0), (16, 2)])
@pytest.mark.parametrize("n", [1, 2, 63, 64, 65, 1000, 311297, 311298, 1000003])
def test_potential_alone_is_that_of_both(n_max, l_max, n):
    """Its kernel runs two blocks per SM and gives a thread particles far apart:
    sizes around a warp, a round of both kernels (2 x 304 x 512) and a ragged one."""
    x = torch.tensor(inputs.hernquist(n, seed=n), dtype=torch.float32, device="cuda")
    c = etics.scf_coeffs(x, n_max, l_max)
    both = etics.scf_field(x, c, n_max, l_max)
    pot = etics.scf_field(x, c, n_max, l_max, out_mask=etics.OUT_POT)
    etics.check_error()
    assert torch.all(pot[:, :3] == 0)
    # another instantiation of the same sums (as in the MEX parity test)
    assert torch.allclose(pot[:, 3], both[:, 3], rtol=1e-6, atol=0)


def test_potential_alone_is_bound_by_memory():
    """n_max = l_max = 0 at 2^21 particles: the bytes of a copy and a few
    instructions; 1.36 times a copy before the pass ran on particle pairs, 2.2 with
    one block of pairs per SM."""
    x = torch.tensor(inputs.hernquist(1 << 21, seed=1), dtype=torch.float32, device="cuda")
    c = etics.scf_coeffs(x, 0, 0)
    out = torch.empty_like(x)
    copy = _best(lambda: out.copy_(x))
    field = _best(lambda: etics.scf_field(x, c, 0, 0, out=out, out_mask=etics.OUT_POT))
    print(f"copy {copy * 1e3:.1f} us, field {field * 1e3:.1f} us")
    assert field <= 1.8 * copy, (field, copy)


@pytest.mark.parametrize("n", [500, 4219])
def test_many_rows_cost_a_small_call_little(n):
    """l_max = 0: the block builds a table of 17 rows instead of two and walks them,
    half a microsecond beside a launch of five; a table loaded row by row by one
    warp cost more than half as much again."""
    x = torch.tensor(inputs.hernquist(n, seed=2), dtype=torch.float32, device="cuda")
    out = torch.empty_like(x)
    times = {}
    for n_max in (1, 16):
        c = etics.scf_coeffs(x, n_max, 0)
        times[n_max] = _best(lambda: etics.scf_field(x, c, n_max, 0, out=out))
    print({k: round(v * 1e3, 1) for k, v in times.items()})
    assert times[16] <= 1.3 * times[1], times
