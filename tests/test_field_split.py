"""The mixed-precision field pass where its levels are split over four, two or one
warps: the lines lie where the particle pairs, times the warps, fill the SMs (152
SMs: 19456 and 38912 particles above l_max = 8, 29184 and 58368 at 7 and 8, 38912
and 77824 below)."""
import pytest
import torch

from paper_1406_4254_gb300 import etics, inputs

pytestmark = pytest.mark.gpu


def _lines(l_max):
    threads = 512 if l_max <= 6 else 384 if l_max <= 8 else 256
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    return [2 * sms * threads // 4, 2 * sms * threads // 2]


@pytest.mark.parametrize("basis", [etics.BASIS_HO, etics.BASIS_CB])
@pytest.mark.parametrize("n_max,l_max", [(10, 2), (5, 3), (10, 6), (14, 8), (6, 7), (12, 9), (4, 14)])
def test_splits_agree(n_max, l_max, basis):
    """The same particles alone and at the front of calls on both sides of each
    line; the split only changes the order in which the levels are added."""
    lines = _lines(l_max)
    x = torch.tensor(inputs.hernquist(lines[1] + 7, seed=3), dtype=torch.float32, device="cuda")
    c = etics.scf_coeffs(x, n_max, l_max, basis=basis)
    k = 1001
    ref = etics.scf_field(x[:k].contiguous(), c, n_max, l_max, basis=basis)
    for n in (lines[0], lines[0] + 1, lines[0] + 3, lines[1], lines[1] + 3):
        y = x[:n].contiguous()
        out = etics.scf_field(y, c, n_max, l_max, basis=basis)
        pot = etics.scf_field(y, c, n_max, l_max, basis=basis, out_mask=etics.OUT_POT)
        etics.check_error()
        # a level's sum is FP32: up to l_max + 1 roundings of the largest value
        tol = 2.0 ** -23 * (l_max + 1) * ref.abs().max()
        assert (out[:k] - ref).abs().max() <= tol, n
        assert (pot[:, 3] - out[:, 3]).abs().max() <= tol, n
        assert torch.isfinite(out).all() and (out[-1] != 0).any()


@pytest.mark.parametrize("n_max,l_max", [(16, 12), (12, 9)])
def test_no_step_at_the_first_line(n_max, l_max):
    """44 particles more take two warps per pair instead of four: each walks half
    of the levels instead of a quarter, but the harmonics of all of them either
    way, and the launch and the table stay: less than a third more.  (With one warp
    the step was 1.55 and 1.62.)"""
    line = _lines(l_max)[0]
    x = torch.tensor(inputs.hernquist(line + 44, seed=4), dtype=torch.float32, device="cuda")
    c = etics.scf_coeffs(x, n_max, l_max)

    def best(n):
        y = x[:n].contiguous()
        out = torch.empty_like(y)
        times = []
        t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        for _ in range(12):
            t0.record()
            for _ in range(10):
                etics.scf_field(y, c, n_max, l_max, out=out)
            t1.record()
            torch.cuda.synchronize()
            times.append(t0.elapsed_time(t1))
        return min(times)

    below, above = best(line), best(line + 44)
    print(f"{below * 100:.1f} us, {above * 100:.1f} us")
    assert above <= 1.35 * below, (below, above)
