"""The tiled LU of contact systems at the sizes where its 32-row tiles end:
coils whose turns touch, of 31 to 479 DOFs, solved as one batch (systems of
different tile counts side by side) against each solved alone."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu

NODES = [8, 9, 16, 17, 25, 56, 60, 104, 120]  # 31, 35, 63, 67, 99, 223, 239, 415, 479 DOFs


def test_batch_of_coils_matches_each_alone():
    from paper_2311_18126_gb300 import System
    descs = []
    for n in NODES:
        desc, params, _ = workloads.coil(N=n, pitch_factor=2.05)
        descs.append(desc)
    keys = ("nodes_per_rod", "x0", "E", "nu", "rho", "radius", "fixed")
    batch = System({k: np.concatenate([d[k] for d in descs]) for k in keys}, params)
    single = [System(d, params) for d in descs]
    touching = 0
    for _ in range(3):
        batch.step(1)
        for s in single:
            s.step(1)
        touching += batch.contact_pairs()
    assert touching > 100
    q, v = batch.get_state()
    parts = [s.get_state() for s in single]
    # the same operations; only the contact terms' sums may come in another
    # order: a few roundings of entries of 0.3 m at most, velocities over dt
    assert np.abs(q - np.concatenate([p[0] for p in parts])).max() < 1e-12
    assert np.abs(v - np.concatenate([p[1] for p in parts])).max() < 1e-12 / params["dt"]
    for s in single + [batch]:
        s.close()
