"""Line search of a batch that mixes a rod network (its trial points evaluated
inside the line search) with free single rods (in rounds of their own), away
from the ground, where single rods keep the rod solver; all of them pulled
back at least once."""
import numpy as np
import pytest

import workloads  # noqa: F401  (path set-up)
from oracle import OracleSystems

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("seed,speed", [(2, 0.15), (7, 0.15), (8, 0.1)])
def test_network_and_single_rods_are_pulled_back(seed, speed):
    from paper_2311_18126_gb300 import System
    rng = np.random.default_rng(seed)
    h, ds = 2e-3, 0.004
    x, v, npr = [], [], []
    for n, a in ((7, 0.0), (8, 2.1), (9, 4.2)):
        x.append(ds * np.arange(n)[:, None] * np.array([[np.cos(a), np.sin(a), 0.0]]))
        v.append(speed * rng.normal(size=(n, 3)))
        v[-1][0] = 0.0
        npr.append(n)
    for n in (9, 12):
        x.append(np.c_[ds * np.arange(n), np.full(n, 1.0 + n), np.zeros(n)])
        v.append(speed * rng.normal(size=(n, 3)))
        npr.append(n)
    R = len(npr)
    desc = dict(nodes_per_rod=npr, x0=np.concatenate(x), v0=np.concatenate(v), E=[1e6] * R, nu=[0.5] * R,
                rho=[1e3] * R, radius=[h] * R, joints=[[(0, 0), (1, 0), (2, 0)]],
                fixed=np.zeros(sum(4 * n - 1 for n in npr), np.uint8))
    params = dict(dt=3e-3, tol=1e-10, max_iter=60, g=(0, 0, -9.81), eta=0.05, line_search=True)
    off = np.concatenate([[0], np.cumsum([4 * n - 1 for n in npr])])
    ora, plain = OracleSystems(desc, params), OracleSystems(desc, dict(params, line_search=False))
    assert all(s[0] == 0 for s in ora.step(1))
    plain.step(1)
    qo, qp = (np.asarray(o.get_state()[0]) for o in (ora, plain))
    for a, b in ((0, off[3]), (off[3], off[4]), (off[4], off[5])):
        # without a pull-back both take the same iterates, to the last bit
        assert np.any(qo[a:b] != qp[a:b])
    gpu = System(desc, params)
    gpu.step(1)
    q = np.array(gpu.get_state()[0])
    gpu.close()
    assert np.abs(q - qo).max() < 1e-10 * 13.0  # the Newton tolerance, at 13 m
