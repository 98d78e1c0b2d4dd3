"""The contact systems' elimination by levels: batches large enough that every
system gets one block and no cluster, a pattern of more than 32 tile columns,
and pivots outside the range of the integer reciprocal."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu

KEYS = ("nodes_per_rod", "x0", "E", "nu", "rho", "radius", "fixed")


def _steps(desc, params, n):
    from paper_2311_18126_gb300 import System
    s = System(desc, params)
    for _ in range(n):
        s.step(1)
    q, v = s.get_state()
    pairs, its = s.contact_pairs(), s.stats.max_iterations
    s.close()
    return np.array(q), np.array(v), pairs, its


def test_more_systems_than_multiprocessors():
    nodes = [56, 60, 66]  # a turn has about 50 nodes
    descs = [workloads.coil(N=n, pitch_factor=2.05)[0] for n in nodes]
    params = workloads.coil(N=nodes[0], pitch_factor=2.05)[1]
    copies = 60  # 180 systems
    batch = {k: np.concatenate([np.concatenate([d[k] for d in descs])] * copies) for k in KEYS}
    q, v, pairs, _ = _steps(batch, params, 3)
    alone = [_steps(d, params, 3) for d in descs]
    assert pairs == copies * sum(a[2] for a in alone) and pairs > 0
    # the same operations but for the order of the blocks' partial sums
    assert np.abs(q.reshape(copies, -1) - np.concatenate([a[0] for a in alone])).max() < 1e-12
    assert np.abs(v.reshape(copies, -1) - np.concatenate([a[1] for a in alone])).max() < 1e-12 / params["dt"]


@pytest.mark.parametrize("nodes", [60, 262])  # 239 and 1047 DOFs: 8 and 33 tile columns
def test_scaled_stiffness_and_mass(nodes):
    """Masses, stiffnesses and contact stiffness times 2^-140 leave the motion
    as it is but put every pivot far below the integer reciprocal's range (the
    division's tile factorisation): two factorisations of one matrix."""
    desc, params, _ = workloads.coil(N=nodes, pitch_factor=2.05)
    f = 2.0 ** -140
    tiny = dict(desc, E=np.asarray(desc["E"]) * f, rho=np.asarray(desc["rho"]) * f)
    tparams = dict(params, pair_kc=params["pair_kc"] * f, eta=params.get("eta", 0.0) * f)
    q, v, pairs, its = _steps(desc, params, 3)
    qs, vs, pairs_s, its_s = _steps(tiny, tparams, 3)
    assert pairs == pairs_s > 0 and its == its_s
    # both end at the Newton tolerance 1e-10 of the scaled residual; the
    # reciprocals differ in the last bit
    assert np.abs(q - qs).max() < 1e-10
    assert np.abs(v - vs).max() < 1e-10 / params["dt"]
