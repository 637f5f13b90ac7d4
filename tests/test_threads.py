"""Host threads with streams of their own call the library at once: kernels whose
shared memory differs from call to call must not take it from one another."""
import threading

import pytest
import torch

from paper_1406_4254_gb300 import etics, inputs

pytestmark = pytest.mark.gpu


def _run(jobs, rounds):
    """Every job in a thread of its own; the errors they met."""
    errors = []
    start = threading.Barrier(len(jobs))

    def work(job):
        stream = torch.cuda.Stream()
        with torch.cuda.stream(stream):
            call = job(stream)
            start.wait()
            try:
                for i in range(rounds):
                    call()
                    if i % 64 == 63:
                        stream.synchronize()
            except etics.EticsError as e:
                errors.append(str(e))
            stream.synchronize()

    threads = [threading.Thread(target=work, args=(j,)) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    return errors


def _batch(l_max, precision, tile):
    def job(stream):
        dtype = torch.float32 if precision == etics.MIXED else torch.float64
        x = torch.tensor(inputs.hernquist(600, seed=l_max), dtype=dtype, device="cuda")
        plan = etics.BatchPlan([200, 400], [4, 6], [l_max, l_max], precision=precision,
                               tuning=etics.BatchTuning(tile, 1, 128, 2048))
        coeffs = torch.empty(plan.coeff_count, dtype=torch.float64, device="cuda")
        return lambda: etics.scf_batch(x, plan, coeffs=coeffs, with_field=False, stream=stream)
    return job


def _coeffs(n_max, l_max):
    def job(stream):
        x = torch.tensor(inputs.hernquist(500, seed=l_max), dtype=torch.float64, device="cuda")
        ws = torch.empty(etics.workspace_bytes(500, n_max, l_max, etics.SCF, etics.FP64) + 256,
                         dtype=torch.uint8, device="cuda")
        out = torch.empty((n_max + 1, (l_max + 1) ** 2), dtype=torch.float64, device="cuda")
        return lambda: etics.scf_coeffs(x, n_max, l_max, out=out, ws=ws, stream=stream)
    return job


@pytest.mark.parametrize("jobs", [
    [_batch(0, etics.MIXED, 64), _batch(8, etics.MIXED, 64)],
    [_batch(2, etics.FP64, 8), _batch(2, etics.FP64, 64)],
    [_coeffs(10, 0), _coeffs(10, 6)],        # one kernel each, by the rows
    [_coeffs(14, 7), _coeffs(14, 10)],
], ids=["batch mixed", "batch fp64", "coeffs low", "coeffs high"])
def test_calls_of_different_sizes_at_once(jobs):
    assert _run(jobs + jobs, 3000) == []
    assert etics.get_error() == 0
