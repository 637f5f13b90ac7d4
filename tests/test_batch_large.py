"""Batches of few large systems: many partial sums per coefficient."""
import numpy as np
import pytest
import torch

from paper_1406_4254_gb300 import etics, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [etics.MIXED, etics.FP64])
@pytest.mark.parametrize("sizes", [[8192], [8193], [16385, 3], [70001, 0, 128], [300007, 5000]])
def test_many_segments_match_the_single_call(sizes, precision):
    """Tiles of 64 leave a segment per 128 particles (mixed) or one per block
    (FP64): around 64, 65, 129, 547 and 2344 of them, systems of one beside."""
    dtype = torch.float32 if precision == etics.MIXED else torch.float64
    x = torch.tensor(np.concatenate([inputs.hernquist(n, seed=n, axes=(1.0, 0.8, 0.6))
                                     for n in sizes if n]), dtype=dtype, device="cuda")
    orders = [(10, 6), (4, 3), (14, 8)][:len(sizes)]
    plan = etics.BatchPlan(sizes, [a for a, _ in orders], [b for _, b in orders],
                           precision=precision, tuning=etics.BatchTuning(64, 2, 128, 2048))
    coeffs, _ = etics.scf_batch(x, plan, with_field=False)
    again, _ = etics.scf_batch(x, plan, with_field=False)
    etics.check_error()
    assert torch.equal(coeffs, again)
    tol = 2e-6 if precision == etics.MIXED else 1e-12       # as in test_batch
    for i, (n, (nm, lm)) in enumerate(zip(sizes, orders)):
        got = plan.coeffs_of(coeffs, i)
        if n == 0:
            assert torch.all(got == 0)
            continue
        a = plan.particle_offsets[i]
        ref = etics.scf_coeffs(x[a:a + n].contiguous(), nm, lm)
        assert (got - ref).abs().max() <= tol * ref.abs().max(), i


def _best(call):
    for _ in range(3):
        call()
    t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    times = []
    for _ in range(10):
        t0.record()
        call()
        t1.record()
        torch.cuda.synchronize()
        times.append(t0.elapsed_time(t1))
    return min(times)


@pytest.mark.parametrize("n", [1 << 20, 1 << 22])
def test_a_batch_of_one_large_system_costs_about_a_single_call(n):
    """The batch kernels take up to half as long again as those written for
    (10, 6); the ordered sum of one system's segments (1024 and 2731 here) by 32
    lanes is 32 and 85 dependent additions, a few us: at most twice a single
    call, where a sum by one thread adds 240 and 1080 us to 130 and 420."""
    x = torch.tensor(inputs.hernquist(n, seed=2), dtype=torch.float32, device="cuda")
    plan = etics.BatchPlan([n], [10], [6])
    coeffs = torch.empty(plan.coeff_count, dtype=torch.float64, device="cuda")
    out = torch.empty_like(x)
    single = _best(lambda: etics.scf_force(x, 10, 6, out=out))
    batch = _best(lambda: etics.scf_batch(x, plan, coeffs=coeffs, out=out))
    etics.check_error()
    print(f"single {single * 1e3:.0f} us, batch {batch * 1e3:.0f} us")
    assert batch <= 2 * single, (single, batch)
