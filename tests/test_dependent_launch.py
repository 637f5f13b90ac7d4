"""Source check of the kernels started by programmatic dependent launch.

Such a kernel may run while the kernel before it in its stream still writes,
until its pdl_wait().  A pointer parameter marked __restrict__ promises the
compiler that nothing else touches the data while the kernel runs, which lets
it move loads to the read-only path and above the wait; the promise does not
hold there.  The only exception is the plan of a batch, which no kernel writes.
Loads past the L1 cache go through ld_cg (etics_common.cuh), which cannot be
moved across the wait either."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1406_4254_gb300", "csrc")
FILES = sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh")))


def _code(path):
    """The file without comments."""
    with open(path) as f:
        text = f.read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return re.sub(r"//[^\n]*", "", text)


def _balanced(text, at, opening, closing):
    """End of the bracketed text that begins at text[at]."""
    depth = 0
    for i in range(at, len(text)):
        depth += text[i] == opening
        depth -= text[i] == closing
        if depth == 0:
            return i + 1
    raise ValueError("unbalanced")


def kernels(text):
    """(name, parameter list, body) of every __global__ function."""
    for m in re.finditer(r"__global__", text):
        at = m.end()
        bounds = re.compile(r"\s*(?:void)?\s*__launch_bounds__\s*").match(text, at)
        if bounds:
            at = _balanced(text, bounds.end(), "(", ")")
        head = re.compile(r"\s*(?:void)?\s*(\w+)\s*").match(text, at)
        end = _balanced(text, head.end(), "(", ")")
        body = re.compile(r"\s*\{").match(text, end)
        if body:
            yield head.group(1), text[head.end():end], text[end:_balanced(text, body.end() - 1, "{", "}")]


def test_the_scan_sees_the_kernels():
    names = {n for f in FILES for n, _, b in kernels(_code(f)) if "pdl_wait()" in b}
    assert {"onesweep_kernel", "bucket_sort_kernel", "mex_pass2_kernel", "scf_field_kernel",
            "scf_coeff_plan_kernel", "mlp_adam_kernel", "gemm_tma_kernel",
            "batch_field_kernel"} <= names


@pytest.mark.parametrize("path", FILES, ids=os.path.basename)
def test_dependent_kernels_make_no_promise_about_their_inputs(path):
    bad = []
    for name, params, body in kernels(_code(path)):
        if "pdl_wait()" not in body:
            continue
        for p in params[1:-1].split(","):
            if "__restrict__" in p and not re.search(r"__restrict__\s*plan\s*$", p):
                bad.append(f"{name}: {' '.join(p.split())}")
    assert not bad, bad


@pytest.mark.parametrize("path", FILES, ids=os.path.basename)
def test_cached_loads_go_through_the_ordered_helper(path):
    assert not re.search(r"\b__ld(cg|g|ca|cs)\s*\(", _code(path))


def test_a_plan_is_read_early_only_behind_the_coefficient_kernel():
    """The batch's finalize reads the plan before its wait.  That is safe behind
    the coefficient kernel, an ordinary launch that began after whatever wrote
    the plan; a batch without particles has no such kernel and its finalize must
    be an ordinary launch itself."""
    code = _code(os.path.join(CSRC, "etics_batch.cu"))
    body = next(b for n, _, b in kernels(code) if n == "batch_finalize_kernel")
    assert body.index("plan_table") < body.index("pdl_wait()")
    at = code.index("launch_pdl(batch_finalize_kernel")
    guard = re.findall(r"if \(hd\.ntiles > 0\) \{\s*if \($", code[:at])
    assert guard, "dependent launch of the finalize without a coefficient kernel before it"


@pytest.mark.gpu
def test_batch_without_particles_whose_plan_a_kernel_wrote():
    import torch

    from paper_1406_4254_gb300 import etics
    plan = etics.BatchPlan([0, 0, 0], [10, 4, 14], [6, 0, 8])
    filler = torch.ones(1 << 24, device="cuda")
    host = plan.dev.clone()
    for _ in range(20):
        plan.dev.zero_()
        coeffs = torch.full((plan.coeff_count,), 3.0, dtype=torch.float64, device="cuda")
        filler.mul_(1.0)
        torch.add(host, 0, out=plan.dev)   # a kernel, not a copy
        etics.scf_batch(filler[:4].reshape(1, 4)[:0], plan, coeffs=coeffs, with_field=False)
        assert etics.get_error() == 0
        assert torch.all(coeffs == 0)
