"""Range of the MEX potential: few particles whose radii span up to 2^22 in one
tile.  In the tile's unit (halfway between the first and the last radius) the
inner terms of the potential reach rho^-11 = 2^121 at l_max = 10; the force's
rho^-12 no longer fits FP32 there, so only the potential is asked for.  (From 2^23
on the outermost particle's own moment m rho^10 leaves FP32.)  From 2^21 on the
outer moments m rho^-11 of the outer particles are subnormal, with few bits: the
call has to be accepted, but only two particles, of which the outer one has
nothing outside it, are accurate."""
import numpy as np
import pytest

import oracle
from helpers import device_particles, rounded
from paper_1406_4254_gb300 import etics

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("exponent", [20, 21, 22])
@pytest.mark.parametrize("n", [2, 9, 200])
def test_potential_alone_of_radii_far_apart(n, exponent):
    rng = np.random.default_rng(n)
    u = rng.normal(size=(n, 3))
    r = np.sort(rng.uniform(1.0, 1.9, n))
    r[0] = 1.25 * 2.0 ** -exponent
    pm = np.zeros((n, 4))
    pm[:, :3] = u / np.linalg.norm(u, axis=1)[:, None] * r[:, None]
    pm[:, 3] = 1.0 / n
    ref = rounded(pm, "mixed")
    _, pot, _ = oracle.mex_field(ref[:, :3], ref[:, 3], 10)
    out = etics.mex_field(device_particles(pm, "mixed"), 10, out_mask=etics.OUT_POT).cpu().numpy()
    assert etics.get_error() == 0
    assert np.isfinite(out).all()
    # the tolerance of the edge cases of few particles (test_parity_mex)
    if n == 2 or exponent == 20:
        assert np.max(np.abs(out[:, 3] - pot)) <= 2e-5 * np.max(np.abs(pot))
