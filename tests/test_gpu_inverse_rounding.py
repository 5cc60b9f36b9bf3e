"""The blocked coarsest-level inverse takes the steps of the unblocked one in
the same order, each a correctly rounded square root, quotient or fused
multiply-add: it equals a Python model of those steps bit for bit.

With one level the V-cycle is K^{-1} r; of a unit vector it is a column of the
stored inverse exactly (products with 1 and 0).  The systems are chosen so that
K is known exactly: dyadic weights, A = c I, lambda = 1.
"""
import math
from fractions import Fraction

import numpy as np
import pytest

from oracle import operators as ops
import problemgen as pg

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2306_11067_gb300 import lcmg as L  # noqa: E402
from paper_2306_11067_gb300 import Solver  # noqa: E402


def _fma(a, b, c):
    return float(Fraction(a) * Fraction(b) + Fraction(c))


def _inverse(M):
    """L L^T = M, X = L^{-1}, X^T X, every sum in increasing order."""
    n = len(M)
    A = [[float(v) for v in row] for row in M]
    for k in range(n):
        A[k][k] = math.sqrt(A[k][k])
        for i in range(k + 1, n):
            A[i][k] /= A[k][k]
        for i in range(k + 1, n):
            for j in range(k + 1, i + 1):
                A[i][j] = _fma(-A[i][k], A[j][k], A[i][j])
    X = np.zeros((n, n))
    for c in range(n):
        for i in range(c, n):
            s = 1.0 if i == c else 0.0
            for k in range(c, i):
                s = _fma(-A[i][k], X[k][c], s)
            X[i][c] = s / A[i][i]
    K = np.zeros((n, n))
    for p in range(n):
        for q in range(p + 1):
            s = 0.0
            for i in range(p, n):
                s = _fma(X[i][p], X[i][q], s)
            K[p][q] = K[q][p] = s
    return K


def _corner(edge):
    """c with c * c + edge^2 + 1/4 = 1 - 2^-53, or None"""
    want = 0.75 - edge * edge - 2.0 ** -53
    c = math.sqrt(want)
    for v in (math.nextafter(c, 0), c, math.nextafter(c, 1)):
        if v * v == want:
            return v
    return None


@pytest.mark.parametrize("n_v,n_h", [(2, 2), (5, 3), (4, 5), (7, 5)])
def test_equals_the_unblocked_steps(n_v, n_h):
    n, ne = n_v * n_h, ops.n_edges(n_v, n_h)
    d = pg.rng(4).integers(1, 9, ne) / 8.0
    # the first pivot 1 - 2^-53, below it -1/4 = -(a power of two): 1 / sqrt(pivot)
    # and the quotient both lie just above the midpoint of two numbers
    edge = next(e for e in np.arange(1, 100) / 128.0 if _corner(e) is not None)
    d[0], d[n_h * (n_v - 1)] = 0.5, edge
    c = _corner(edge)
    s = Solver(n_v, n_h, levels=1)
    s.set_forward_separable(np.array([c]), np.array([1.0]))
    s.set_weights(d)
    diag = L.lcmg_get_diag(s.ctx, n)
    assert (diag == c * c).all()
    rd = torch.eye(n, dtype=torch.float64, device="cuda")
    zd = torch.empty_like(rd)
    L.lcmg_apply_vcycle_dev(s.ctx, np.ones(n), rd, zd)
    got = zd.cpu().numpy().T
    s.close()
    Lg = ops.gradient(n_v, n_h).toarray()
    G = Lg.T @ (d[:, None] ** 2 * Lg)  # dyadic: exact
    K = G.copy()
    K[np.diag_indices(n)] = [float(Fraction(G[i, i]) + Fraction(diag[i])) for i in range(n)]
    assert K[0, 0] == 1 - 2.0 ** -53 and K[1, 0] == -0.25
    assert (got == _inverse(K)).all()
