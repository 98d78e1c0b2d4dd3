"""Bend-twist stencils at the twist angles where their formulas change: the
series of the angle below 1/8 and the general function above it, around a
half turn and several turns per node (the reference twist continues from its
committed value), on curved and on nearly folded rods, with the middle rod of
a joint reversed."""
import numpy as np
import pytest

import workloads
from oracle import OracleSystems
from test_gpu_parity import _assert_close, _gpu

pytestmark = pytest.mark.gpu

TWIST = [0.0, 0.124, 0.125, 0.126, 1.5, 3.1, 3.2, -3.2, 10.0, -25.0]


def _rods(fold):
    rng = np.random.default_rng(23)
    N, x0 = 6, []
    for k, _ in enumerate(TWIST):
        turn = fold * np.arange(N - 1) * (1.0 if k % 2 else -1.0)
        e = np.c_[np.cos(turn), np.sin(turn), 0.2 * rng.normal(size=N - 1)]
        e *= 0.02 / np.linalg.norm(e, axis=1)[:, None]
        x0.append(np.vstack([np.zeros(3), np.cumsum(e, axis=0)]) + [0.0, 0.5 * k, 0.0])
    R = len(TWIST)
    desc = dict(nodes_per_rod=[N] * R, x0=np.concatenate(x0), E=[1e6] * R, nu=[0.5] * R, rho=[1e3] * R,
                radius=[2e-3] * R)
    theta = [t * np.arange(N - 1) for t in TWIST]
    params = dict(dt=2e-5, tol=1e-10, max_iter=40, g=(0, 0, -9.81), eta=0.0)
    return desc, params, theta


def _start(sysm, N, theta):
    q, v = sysm.get_state()
    q = np.array(q)
    for r, t in enumerate(theta):
        q[r * (4 * N - 1) + 3:(r + 1) * (4 * N - 1):4] = t
    return q, np.array(v)


@pytest.mark.parametrize("fold", [0.05, 1.0, 2.3])
def test_twisted_rods_against_oracle(fold):
    desc, params, theta = _rods(fold)
    gpu, ora = _gpu(desc, params), OracleSystems(desc, params)
    q, v = _start(ora, 6, theta)
    for s in (gpu, ora):
        s.set_state(q, v)
    L = max(1.0, float(np.abs(desc["x0"]).max()))
    for _ in range(3):
        gpu.step(1)
        st = ora.step(1)
        assert all(x[0] == 0 for x in st), st
        qg, _ = gpu.get_state()
        qo, vo = ora.get_state()
        _assert_close(qg, qo, desc["nodes_per_rod"], L, 1e-10)  # the Newton tolerance
        _, bg = gpu.get_frames()
        d1, bo = ora.get_frames()
        assert np.abs(np.asarray(bg) - np.asarray(bo)).max() < 1e-9  # angles of up to 100 rad
        gpu.set_state(qo, vo)
        gpu.set_frames(d1, bo)


def test_reversed_edges_with_large_twist():
    desc, params, _ = workloads.star_robots(n_robots=1, seed=5, nodes_per_limb=6)
    # the first rod reversed: its edges enter the joint stencils flipped
    n0 = desc["nodes_per_rod"][0]
    x = np.array(desc["x0"])
    x[:n0] = x[:n0][::-1]
    desc = dict(desc, x0=x, joints=[[(r, n0 - 1 - k if r == 0 else k) for r, k in j] for j in desc["joints"]])
    params = dict(params, ground=False)
    gpu, ora = _gpu(desc, params), OracleSystems(desc, params)
    q, v = ora.get_state()
    q = np.array(q)
    off = np.concatenate([[0], np.cumsum([4 * n - 1 for n in desc["nodes_per_rod"]])])
    for r, n in enumerate(desc["nodes_per_rod"]):
        q[off[r] + 3:off[r + 1]:4] = 0.3 * (r + 1) * np.arange(n - 1)
    for s in (gpu, ora):
        s.set_state(q, np.array(v))
    gpu.step(1)
    st = ora.step(1)
    assert all(x[0] == 0 for x in st), st
    _assert_close(gpu.get_state()[0], ora.get_state()[0], desc["nodes_per_rod"], 1.0, 1e-10)
