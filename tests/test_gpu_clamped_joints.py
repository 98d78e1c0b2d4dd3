"""Rod networks whose joints are clamped (the joint node, its neighbours and
the twist angles at it fixed): the limbs there have no border left and are
eliminated from a twist angle on.  Stars with a clamped hub, and chains of
which the near, the far or an inner joint is clamped, so that a limb with
joints at both ends is condensed from either; on the ground with friction and
without; steps and the step adjoint against the oracle."""
import numpy as np
import pytest

import workloads  # noqa: F401  (path set-up)
from oracle import OracleSystems
from oracle.adjoint import step_adjoint
from test_gpu_general import _run
from test_gpu_parity import _gpu

pytestmark = pytest.mark.gpu

H, SPACING = 2e-3, 0.1 / 29


def _clamp(fixed, npr, rod, end):
    """The joint node, its neighbour and the twist angle between them."""
    o, n = int(np.sum(4 * np.asarray(npr[:rod]) - 1)), npr[rod]
    first = 4 * n - 8 if end else 0
    fixed[o + first:o + first + 7] = 1


def _star(n, ends):
    """Rods of n, n + 1, ... nodes meeting at their first (0) or last (1) node."""
    x, npr, hub = [], [], []
    for j, end in enumerate(ends):
        k, a = n + j, 2 * np.pi * j / len(ends) + 0.3
        p = SPACING * np.arange(k)[:, None] * np.array([[np.cos(a), np.sin(a), 0.0]]) + [0.0, 0.0, 0.99 * H]
        x.append(p[::-1] if end else p)
        npr.append(k)
        hub.append((j, k - 1 if end else 0))
    fixed = np.zeros(int(sum(4 * k - 1 for k in npr)), np.uint8)
    for j, end in enumerate(ends):
        _clamp(fixed, npr, j, end)
    return npr, x, [hub], fixed


def _chain(n, clamped, turned):
    """Three rods end to end along x (the middle one against it if `turned`),
    the listed joints clamped."""
    npr = [n, n + 1, n + 2]
    x, joints, o = [], [], 0.0
    for j, k in enumerate(npr):
        p = np.c_[o + SPACING * np.arange(k), np.zeros(k), np.full(k, 0.99 * H)]
        x.append(p[::-1] if turned and j == 1 else p)
        o = p[-1, 0]
    ends = [(0, k - 1) for k in npr]  # the nodes a rod starts and ends with along x
    if turned:
        ends[1] = ends[1][::-1]
    joints = [[(0, ends[0][1]), (1, ends[1][0])], [(1, ends[1][1]), (2, ends[2][0])]]
    fixed = np.zeros(sum(4 * k - 1 for k in npr), np.uint8)
    for c in clamped:
        for rod, node in joints[c]:
            _clamp(fixed, npr, rod, 0 if node == 0 else 1)
    return npr, x, joints, fixed


CASES = {
    "star": lambda n: _star(n, [0, 0, 0]),
    "star, last nodes": lambda n: _star(n, [1, 0, 1]),
    "chain, near joint": lambda n: _chain(n, [0], False),
    "chain, far joint": lambda n: _chain(n, [1], False),
    "chain, near joint, turned": lambda n: _chain(n, [0], True),
    "chain, far joint, turned": lambda n: _chain(n, [1], True),
    "chain, both joints": lambda n: _chain(n, [0, 1], False),
}


def _system(case, n, ground, integrator="be"):
    npr, x, joints, fixed = CASES[case](n)
    R = len(npr)
    rng = np.random.default_rng(23)
    x = np.concatenate(x)
    v = np.c_[0.02 * rng.normal(size=(len(x), 2)), np.zeros(len(x))]
    o = np.concatenate([[0], np.cumsum(npr)])
    for ends in joints:  # one velocity per joint
        for r, node in ends:
            v[o[r] + node] = v[o[ends[0][0]] + ends[0][1]]
    d0 = np.concatenate([[0], np.cumsum(4 * np.asarray(npr) - 1)])
    for r in range(R):  # what is clamped rests
        for i in range(npr[r]):
            if fixed[d0[r] + 4 * i]:
                v[o[r] + i] = 0.0
    desc = dict(nodes_per_rod=npr, x0=x, v0=v, E=[1e6] * R, nu=[0.5] * R, rho=[1e3] * R, radius=[H] * R,
                joints=joints, fixed=fixed)
    params = dict(dt=5e-3, tol=1e-10, max_iter=60, g=(0.5, 0.2, -9.81), eta=0.05, integrator=integrator)
    if ground:
        kc = 10.0 * 1000.0 * np.pi * H * H * SPACING * 9.81 / 1e-3
        desc.update(ground_mu=[0.4] * R, ground_kc=[kc] * R)
        params.update(ground=True, ground_z=0.0, delta=1e-3, nu_slip=5e-2, line_search=True)
    return desc, params


@pytest.mark.parametrize("ground", [False, True])
@pytest.mark.parametrize("n", [5, 12, 30])
@pytest.mark.parametrize("case", CASES)
def test_steps_against_oracle(case, n, ground):
    desc, params = _system(case, n, ground)
    _run(desc, params, 3, 1e-10)  # the Newton tolerance both sides step to


@pytest.mark.parametrize("ground", [False, True])
@pytest.mark.parametrize("integrator", ["be", "midpoint"])
@pytest.mark.parametrize("case", CASES)
def test_step_adjoint_against_oracle(case, integrator, ground):
    desc, params = _system(case, 12, ground, integrator)
    gpu, ora = _gpu(desc, params), OracleSystems(desc, params)
    for _ in range(3):
        ora.step(1)
    q0, v0 = ora.get_state()
    d1, beta = ora.get_frames()
    ora.step(1)
    q1, _ = ora.get_state()
    rng = np.random.default_rng(29)
    wq, wv = rng.normal(size=len(q0)), rng.normal(size=len(q0))
    ora.set_state(q0, v0)
    ora.set_frames(d1, beta)
    want = step_adjoint(ora, q1, wq, wv)
    gpu.set_state(q0, v0)
    gpu.set_frames(d1, beta)
    got = gpu.step_adjoint(q1, wq, wv)
    for a, b in zip(got, want):
        scale = max(1.0, float(np.abs(b).max()))
        assert np.abs(a - b).max() <= 1e-8 * scale, np.abs(a - b).max() / scale
