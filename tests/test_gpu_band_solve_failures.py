"""What dm_solve_band and dm_solve_band_noalloc leave in x: the solution of
every system that has one, zeros for the systems that fail and for entries
outside every system, whatever x held before."""
import numpy as np
import pytest

from test_gpu_band_solve import random_band_batch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name", ["solve_band", "solve_band_noalloc"])
@pytest.mark.parametrize("gap", [0, 3])
def test_failed_systems_are_zero(name, gap):
    import torch
    from paper_2311_18126_gb300 import dismech, ensure_built
    ensure_built()
    sizes = [5, 31, 32, 60, 41, 200, 9]
    band, rhs, dense = random_band_batch(sizes, 3)
    off = np.concatenate([[0], np.cumsum(sizes)])
    # a zero row in: a short system, a twisted one's top and bottom chain and its separator
    fails = {1: 30, 2: 0, 3: 59, 5: 99}
    for k, row in fails.items():
        for d in range(11):
            band[d, off[k] + row] = 0.0
            if row + d < sizes[k]:
                band[d, off[k] + row + d] = 0.0
    d0 = off[:-1] + gap * np.arange(len(sizes))
    ntot = off[-1] + gap * len(sizes)
    at = np.concatenate([np.arange(a, a + n) for a, n in zip(d0, sizes)])
    b, r = np.zeros((11, ntot)), np.zeros(ntot)
    b[:, at], r[at] = band, rhs
    tb, tr = torch.tensor(b, device="cuda"), torch.tensor(r, device="cuda")
    tx = torch.full((ntot,), float("nan"), dtype=torch.float64, device="cuda")
    with pytest.raises(dismech.DismechError):
        getattr(dismech, name)(d0, sizes, tb, tr, tx)
    x = tx.cpu().numpy()
    outside = np.ones(ntot, bool)
    outside[at] = False
    assert np.all(x[outside] == 0.0)
    for k, (a, n) in enumerate(zip(d0, sizes)):
        if k in fails:
            assert np.all(x[a:a + n] == 0.0), k
        else:
            np.testing.assert_allclose(x[a:a + n], np.linalg.solve(dense[k], rhs[off[k]:off[k + 1]]), rtol=1e-12,
                                       atol=1e-14)
