"""Limbs of the condensation path, whose rows the elimination forms from the
element terms: rods of every length around the four-row period, the 12-column
block and the 32-lane pass, joined at their first or last node, with fixed
DOFs at the free end, next to the joint and inside, on the ground with
friction and without."""
import numpy as np
import pytest

import workloads  # noqa: F401  (path set-up)
from test_gpu_general import _run

pytestmark = pytest.mark.gpu


def _networks(lengths, ground):
    """Per entry of `lengths` a network of three rods of n, n + 1 and n + 2
    nodes, joined at the first, last and first node."""
    x, npr, joints, fixed, v = [], [], [], [], []
    rng = np.random.default_rng(17)
    y0, h = 0.0, 0.01
    for k, n0 in enumerate(lengths):
        dirs = np.array([[1.0, 0.0, 0.0], [-0.5, 0.8, 0.0], [-0.4, -0.9, 0.0]])
        ends = []
        for j in range(3):
            n = n0 + j
            s = np.linspace(0, 0.03 * (n - 1), n)[:, None]
            # (not at height h itself: there the oracle's softplus differentiates its kink)
            p = np.array([0.0, y0, 0.99 * h]) + s * dirs[j] / np.linalg.norm(dirs[j])
            if j == 1:
                p = p[::-1]
            x.append(p)
            ends.append((3 * k + j, n - 1 if j == 1 else 0))
            npr.append(n)
            v.append(np.c_[0.02 * rng.normal(size=(n, 2)), np.zeros(n)])
            f = np.zeros(4 * n - 1, np.uint8)
            if j == 0 and k % 3 == 0:
                f[-3:] = 1          # free end clamped
            if j == 1 and k % 3 == 1 and n > 4:
                f[4 * (n - 3) + 2] = 1  # a height next to the joint
            if j == 2 and k % 3 == 2:
                f[4 * (n // 2) - 1] = 1  # a twist inside
            fixed.append(f)
        joints.append(ends)
        # rods of one joint meet in one point
        y0 += 0.08 * (n0 + 3)
    R = len(npr)
    desc = dict(nodes_per_rod=npr, x0=np.concatenate(x), E=[1e6] * R, nu=[0.5] * R, rho=[1e3] * R,
                radius=[h] * R, joints=joints, fixed=np.concatenate(fixed), v0=None)
    params = dict(dt=2e-3, tol=1e-10, max_iter=60, g=(0.5, 0, -9.81), eta=0.05)
    if ground:
        nodes = np.concatenate(x).shape[0]
        kc = 10.0 * (1000.0 * np.pi * h * h * 0.03) * 9.81 / 2e-3
        desc.update(ground_mu=[0.4] * R, ground_kc=[kc] * R)
        params.update(ground=True, ground_z=0.0, delta=2e-3, nu_slip=5e-2)
        assert nodes == sum(npr)
    vel = np.concatenate(v)
    o = np.concatenate([[0], np.cumsum(npr)])
    for ends in joints:  # one velocity per joint
        i0 = o[ends[0][0]] + ends[0][1]
        for r, node in ends:
            vel[o[r] + node] = vel[i0]
    desc["v0"] = vel
    return desc, params


@pytest.mark.parametrize("ground", [False, True])
@pytest.mark.parametrize("lengths", [[2, 3, 4, 5, 6, 7], [8, 9, 10, 11], [30, 31, 32]])
def test_limb_lengths_against_oracle(lengths, ground):
    desc, params = _networks(lengths, ground)
    _run(desc, params, 3, 1e-10)  # the Newton tolerance both sides step to


def test_line_search_inside_and_across_rounds():
    """Trial points of small general systems are evaluated inside the line
    search, those of larger systems (over 4096 DOFs) and of single rods in
    rounds of their own; both follow the oracle's backtracking."""
    from oracle import OracleSystems
    from paper_2311_18126_gb300 import System
    desc, params, _ = workloads.star_robots(n_robots=2, seed=9, nodes_per_limb=7)
    rng = np.random.default_rng(2)
    big, N = 1100, 9  # 4399 DOFs
    x = [np.asarray(desc["x0"])]
    for n, y in ((big, 3.0), (N, 4.0)):
        x.append(np.c_[0.004 * np.arange(n), np.full(n, y), np.full(n, desc["radius"][0])])
    x0 = np.concatenate(x)
    npr = list(desc["nodes_per_rod"]) + [big, N]
    R = len(npr)
    ext = lambda k: np.concatenate([np.asarray(desc[k], float), [desc[k][0]] * 2])
    v0 = np.zeros_like(x0)
    v0[-(big + N):, 2] = np.repeat(0.3 * rng.normal(size=(big + N + 4) // 4), 4)[:big + N]  # rough: trial points fail
    d = dict(nodes_per_rod=npr, x0=x0, v0=v0, joints=desc["joints"],
             fixed=np.zeros(int(sum(4 * n - 1 for n in npr)), np.uint8),
             **{k: ext(k) for k in ("E", "nu", "rho", "radius", "ground_mu", "ground_kc")})
    p = dict(params, line_search=True)
    s = System(d, p)
    s.step(1)
    together = np.array(s.get_state()[0])
    s.close()
    # the large rod alone, its trial points in rounds, against the whole batch,
    # where the same kernels ran beside the robots' loop
    off = np.concatenate([[0], np.cumsum([4 * n - 1 for n in npr])])
    small = [r for r in range(R) if npr[r] != big]
    keep = np.concatenate([np.arange(off[r], off[r + 1]) for r in small])
    nodes = np.concatenate([[0], np.cumsum(npr)])
    kn = np.concatenate([np.arange(nodes[r], nodes[r + 1]) for r in small])
    ds = dict(d, nodes_per_rod=[npr[r] for r in small], x0=x0[kn], v0=v0[kn], fixed=d["fixed"][keep],
              **{k: d[k][small] for k in ("E", "nu", "rho", "radius", "ground_mu", "ground_kc")})
    ora = OracleSystems(ds, p)
    st = ora.step(1)
    assert all(t[0] == 0 for t in st), st
    qo = np.asarray(ora.get_state()[0])
    assert np.abs(together[keep] - qo).max() < 1e-10 * 4.0  # the Newton tolerance, at 4 m
    dl = dict(d, nodes_per_rod=[big], x0=x0[nodes[-3]:nodes[-2]], v0=v0[nodes[-3]:nodes[-2]], joints=[],
              fixed=d["fixed"][off[-3]:off[-2]],
              **{k: d[k][-2:-1] for k in ("E", "nu", "rho", "radius", "ground_mu", "ground_kc")})
    s = System(dl, p)
    s.step(1)
    assert np.array_equal(np.array(s.get_state()[0]), together[off[-3]:off[-2]])
    s.close()
