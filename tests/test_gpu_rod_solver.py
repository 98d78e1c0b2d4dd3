"""The rod solver's two lane splits (16 lanes per chain for small batches,
8 for large ones) at the sizes where its blocks and chains end: systems
shorter than the twisted factorisation, at its threshold, and around
multiples of the 12-column block, in batches on both sides of the split."""
import numpy as np
import pytest
import torch

import workloads

pytestmark = pytest.mark.gpu

SIZES = [1, 2, 7, 11, 12, 13, 23, 24, 31, 32, 33, 34, 44, 45, 46, 56, 57, 58, 80, 81, 82, 83]


def _band_batch(copies):
    rng = np.random.default_rng(7)
    ndof = np.array(SIZES)
    mats, rhs = [], []
    for n in ndof:
        B = np.tril(rng.normal(size=(n, n))) * (np.abs(np.subtract.outer(np.arange(n), np.arange(n))) <= 10)
        A = B @ B.T + 30.0 * np.eye(n)  # half bandwidth 10, conditioned below 1e3
        mats.append(np.where(np.abs(np.subtract.outer(np.arange(n), np.arange(n))) <= 10, A, 0.0))
        rhs.append(rng.normal(size=n))
    n1 = int(ndof.sum())
    band = np.full((11, n1), 5.0)  # entries outside a system are not read
    off = np.concatenate([[0], np.cumsum(ndof)])
    for k, A in enumerate(mats):
        for d in range(min(11, len(A))):
            band[d, off[k] + d:off[k + 1]] = np.diagonal(A, -d)
    ref = np.concatenate([np.linalg.solve(A, b) for A, b in zip(mats, rhs)])
    dof0 = np.concatenate([off[:-1] + n1 * c for c in range(copies)])
    return (dof0, np.tile(ndof, copies), np.tile(band, (1, copies)), np.tile(np.concatenate(rhs), copies),
            np.tile(ref, copies))


@pytest.mark.parametrize("copies", [1, 60])  # 22 systems: 16 lanes per chain; 1320: 8
def test_band_sizes_against_dense(copies):
    from paper_2311_18126_gb300 import dismech
    dof0, ndof, band, rhs, ref = _band_batch(copies)
    x = torch.full((len(rhs),), np.nan, dtype=torch.float64, device="cuda")
    dismech.solve_band(dof0, ndof, torch.from_numpy(band).cuda(), torch.from_numpy(rhs).cuda(), x)
    err = np.abs(x.cpu().numpy() - ref).max() / np.abs(ref).max()
    assert err < 1e-12  # condition < 1e3 times a few hundred roundings


def test_lane_splits_agree_on_rods():
    """Rods of 2 to 24 nodes stepped alone (16 lanes per chain) and as one of
    70 copies (8 lanes): the same operations in the same order, so bit for
    bit the same; and against the oracle."""
    from oracle import OracleSystems
    from paper_2311_18126_gb300 import System
    npr = np.arange(2, 25)
    R = len(npr)
    rng = np.random.default_rng(3)
    x0, fixed = [], []
    for n in npr:
        x = np.zeros((n, 3))
        x[:, 0] = 0.02 * np.arange(n)
        x[:, 2] = 1e-3 * np.cumsum(rng.normal(size=n))
        x0.append(x)
        m = np.zeros(4 * n - 1, np.uint8)
        m[:7 if n > 2 else 4] = 1
        fixed.append(m)

    def desc(copies):
        return dict(nodes_per_rod=np.tile(npr, copies).astype(np.int32), x0=np.concatenate(x0 * copies),
                    E=np.full(R * copies, 1e6), nu=np.full(R * copies, 0.5), rho=np.full(R * copies, 1000.0),
                    radius=np.full(R * copies, 2e-3), fixed=np.concatenate(fixed * copies))

    params = dict(workloads.CANTILEVER_PARAMS)
    small, large, ora = System(desc(1), params), System(desc(70), params), OracleSystems(desc(1), params)
    for _ in range(3):
        small.step(1)
        large.step(1)
        ora.step(1)
    a, b = small.get_state(), large.get_state()
    for k in range(2):
        assert np.array_equal(np.tile(a[k], 70), b[k])
    assert np.abs(a[0] - ora.get_state()[0]).max() < 1e-10
    small.close()
    large.close()
