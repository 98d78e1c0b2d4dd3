"""Host emulation (numpy, CPU) of the limb elimination's envelope: columns with
10, 9, 8 and 7 rows below them in turn, from the limb's first x on (from its
last z on where it is eliminated from its last row), the columns before that
with ten rows; against a dense solve of matrices with a rod Jacobian's
pattern, friction's nonsymmetric node blocks among them."""
import numpy as np
import pytest


def _rod_matrix(N, rng):
    """Random matrix with the couplings of a rod of N nodes (Eq. 1 layout): the
    bend-twist stencils' 11 x 11 blocks, the edges' node pairs, the nodes'
    3 x 3 blocks (nonsymmetric), diagonally dominant."""
    n = 4 * N - 1
    J = np.zeros((n, n))
    for m in range(1, N - 1):
        s = slice(4 * m - 4, 4 * m + 7)
        b = rng.standard_normal((11, 11))
        J[s, s] += b + b.T
    for i in range(N - 1):
        r = np.r_[4 * i:4 * i + 3, 4 * i + 4:4 * i + 7]
        b = rng.standard_normal((6, 6))
        J[np.ix_(r, r)] += b + b.T
    for i in range(N):
        J[4 * i:4 * i + 3, 4 * i:4 * i + 3] += rng.standard_normal((3, 3))
    return J + np.diag(2.0 + np.abs(J).sum(axis=1))


def _limb_lead(first, n, direction):
    return (first + n - 1 + 2) & 3 if direction else (4 - (first & 3)) & 3


def _eliminate(A, y, lead):
    """In order, a column's update over the rows and columns of its type."""
    A, y, n = A.copy(), y.copy(), len(y)
    for p in range(n):
        R = min(10 if p < lead else 10 - ((p - lead) & 3), n - 1 - p)
        rows = np.arange(p + 1, p + 1 + R)
        m = A[rows, p] / A[p, p]
        A[np.ix_(rows, rows)] -= np.outer(m, A[p, rows])
        y[rows] -= m * y[p]
    x = np.zeros(n)
    for p in range(n - 1, -1, -1):
        k = np.arange(p + 1, min(p + 11, n))
        x[p] = (y[p] - A[p, k] @ x[k]) / A[p, p]
    return x


@pytest.mark.parametrize("direction", [0, 1])
@pytest.mark.parametrize("first", [0, 1, 2, 3, 7])
@pytest.mark.parametrize("cut", [0, 1, 2, 3, 7])  # rows of the rod behind the limb
def test_envelope_of_every_phase(first, cut, direction):
    rng = np.random.default_rng(100 * first + 10 * cut + direction)
    for N in (4, 5, 9, 30):
        n = 4 * N - 1 - first - cut
        if n < 1:
            continue
        J = _rod_matrix(N, rng)[first:first + n, first:first + n]
        y = rng.standard_normal(n)
        if direction:
            J, y = J[::-1, ::-1], y[::-1]
        lead = _limb_lead(first, n, direction)
        # rows of the rod that the elimination meets, in its order: none beyond
        # the envelope couples to a column
        for p in range(n):
            R = 10 if p < lead else 10 - ((p - lead) & 3)
            assert not J[p + 1 + R:, p].any() and not J[p, p + 1 + R:].any()
        ref = np.linalg.solve(J, y)
        # backward stable for a diagonally dominant matrix: a few ulps of the solution
        assert np.abs(_eliminate(J, y, lead) - ref).max() <= 1e-13 * np.abs(ref).max()
