"""Contact systems every free pivot of which is below the integer reciprocal's
range (2^-126), so that each tile is factored by divisions; the rows of fixed
DOFs keep a pivot of 1."""
import numpy as np
import pytest

import workloads
from test_gpu_contact_levels import _steps

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nodes", [60, 262])  # 239 and 1047 DOFs: 8 and 33 tile columns
def test_scaled_far_below_the_range(nodes):
    """Masses, stiffnesses and contact stiffness times 2^-200 leave the motion
    as it is."""
    desc, params, _ = workloads.coil(N=nodes, pitch_factor=2.05)
    f = 2.0 ** -200
    x, r = np.asarray(desc["x0"]).reshape(-1, 3), desc["radius"][0]
    length = np.linalg.norm(np.diff(x, axis=0), axis=1)
    # the largest entries: stretching, mass over dt^2, contact
    most = max(4.0 * desc["E"][0] * np.pi * r * r / length.min(),
               2.0 * desc["rho"][0] * np.pi * r * r * length.max() / params["dt"] ** 2, 100.0 * params["pair_kc"])
    assert most * f < 2.0 ** -140
    tiny = dict(desc, E=np.asarray(desc["E"]) * f, rho=np.asarray(desc["rho"]) * f)
    tparams = dict(params, pair_kc=params["pair_kc"] * f, eta=params.get("eta", 0.0) * f)
    q, v, pairs, its = _steps(desc, params, 3)
    qs, vs, pairs_s, its_s = _steps(tiny, tparams, 3)
    assert pairs == pairs_s > 0 and its == its_s
    # both end at the Newton tolerance 1e-10 of the scaled residual
    assert np.abs(q - qs).max() < 1e-10
    assert np.abs(v - vs).max() < 1e-10 / params["dt"]
