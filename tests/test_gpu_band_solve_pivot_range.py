"""Separator pivots of the twisted solve up to the largest number with a normal
reciprocal (below 2^1022) are divided by; larger ones are refused, not turned
into a wrong x."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("copies", [1, 1300])  # 16 and 8 lanes per chain
@pytest.mark.parametrize("exponent,solved", [(-1022, True), (-300, True), (200, True), (1021, True), (1022, False),
                                              (1023, False)])
def test_separator_pivots(exponent, solved, copies):
    import torch
    from paper_2311_18126_gb300 import dismech, ensure_built
    ensure_built()
    n = 40  # rows 15 .. 24 are the separator
    diag = np.ones(n)
    diag[18] = 1.5 * 2.0 ** exponent
    band = np.zeros((11, n * copies))
    band[0] = np.tile(diag, copies)
    rhs = np.ones(n * copies)
    rhs[18::n] = diag[18]
    tb, tr = torch.tensor(band, device="cuda"), torch.tensor(rhs, device="cuda")
    tx = torch.empty_like(tr)
    solve = lambda: dismech.solve_band(n * np.arange(copies), [n] * copies, tb, tr, tx)
    if not solved:
        with pytest.raises(dismech.DismechError):
            solve()
        return
    solve()
    assert np.abs(tx.cpu().numpy() - 1.0).max() <= 2.0 ** -52  # a reciprocal and a product
