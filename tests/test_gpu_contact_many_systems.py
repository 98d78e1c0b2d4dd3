"""More contact systems than a grid has rows (65535): 65600 rods of three nodes
and, last, a coil whose turns touch, stepped and differentiated as the coil
alone is."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


def test_more_contact_systems_than_grid_rows():
    from paper_2311_18126_gb300 import System
    desc, params, _ = workloads.coil(N=60, pitch_factor=2.05)
    many, side = 65600, 257
    k = np.arange(many)
    at = np.stack([1.0 + 0.0625 * (k % side), 0.0625 * (k // side), np.zeros(many)], axis=1)
    x = at[:, None, :] + np.array([[0.0, 0.0, 0.0], [2.0 ** -8, 0.0, 0.0], [2.0 ** -7, 0.0, 0.0]])
    batch = dict(nodes_per_rod=np.concatenate([np.full(many, 3), desc["nodes_per_rod"]]).astype(np.int32),
                 x0=np.concatenate([x.reshape(-1, 3), np.asarray(desc["x0"]).reshape(-1, 3)]),
                 fixed=np.concatenate([np.zeros(11 * many, np.uint8), desc["fixed"]]),
                 **{f: np.concatenate([np.full(many, desc[f][0]), desc[f]]) for f in ("E", "nu", "rho", "radius")})
    rng = np.random.default_rng(3)
    w = rng.standard_normal((2, len(desc["fixed"])))
    out = []
    for d, n in ((batch, 11 * many), (desc, 0)):
        s = System(d, params)
        s.step(2)
        q0, v0 = (np.array(a) for a in s.get_state())
        s.step(1)
        q1 = np.array(s.get_state()[0])
        assert s.contact_pairs() > 0
        s.set_state(q0, v0)
        pad = np.zeros(n)
        g = s.step_adjoint(q1, np.concatenate([pad, w[0]]), np.concatenate([pad, w[1]]))
        out.append([q1[n:]] + [np.asarray(a)[n if i else n // 11:] for i, a in enumerate(g)])
        if n:  # the short rods only fall
            z = q1[:n].reshape(many, 11)
            assert np.abs(z[:, [2, 6, 10]] - z[0, 2]).max() < 1e-10 and z[0, 2] < 0.0
        s.close()
    for a, b in zip(*out):  # the same operations but for the order of the blocks' partial sums
        assert np.abs(a - b).max() <= 1e-10 * max(1.0, np.abs(b).max())
