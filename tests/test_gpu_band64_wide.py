"""Separable FP64 passes of many columns: the tiles that take them (and, at 15
columns, the form with one output per thread) against the oracle's normal
operator to 1e-13, and whole solves of 32 right-hand sides against the same
systems solved one by one (relative residual 1e-12, condition numbers below
1e3: 1e-8)."""
import numpy as np
import pytest

import problemgen as pg
from oracle import operators as ops

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2306_11067_gb300 import lcmg as L  # noqa: E402
from paper_2306_11067_gb300 import Solver  # noqa: E402

SIZES = [  # n_v, n_h, r_v, r_h: whole tiles, ragged lines, ragged segments
    (128, 128, 4, 9),
    (128, 120, 15, 6),
    (120, 128, 3, 16),
]


def _solver(n_v, n_h, rv, rh, **kw):
    rng = pg.rng(5)
    fv, fh = rng.uniform(0.5, 1.5, 2 * rv + 1), rng.uniform(0.5, 1.5, 2 * rh + 1)
    fv, fh = fv / fv.sum(), fh / fh.sum()
    d = rng.uniform(0.3, 1.0, ops.n_edges(n_v, n_h))
    s = Solver(n_v, n_h, **kw)
    s.set_forward_separable(fv, fh)
    s.set_weights(d)
    return s, np.outer(fv, fh), d, rng


@pytest.mark.parametrize("n_v,n_h,rv,rh", SIZES)
@pytest.mark.parametrize("cols", [15, 32])
def test_normal_operator_of_many_columns(n_v, n_h, rv, rh, cols):
    s, psf, d, rng = _solver(n_v, n_h, rv, rh)
    x = rng.standard_normal((cols, n_v * n_h))
    lam = np.geomspace(0.1, 2.0, cols)
    xd = torch.tensor(x, device="cuda")
    yd = torch.empty_like(xd)
    L.lcmg_apply_normal_dev(s.ctx, lam, xd, yd)
    s.close()
    F, Lg = ops.ForwardPSF(psf, n_v, n_h), ops.gradient(n_v, n_h)
    for k in range(cols):
        ref = ops.normal_apply(F, Lg, d, lam[k], x[k])
        assert np.linalg.norm(yd[k].cpu().numpy() - ref) <= 1e-13 * np.linalg.norm(ref)


@pytest.mark.parametrize("n_v,n_h,rv,rh", SIZES)
def test_wide_solve_equals_single_solves(n_v, n_h, rv, rh):
    s, psf, d, rng = _solver(n_v, n_h, rv, rh, tol=1e-12)
    b = rng.standard_normal((32, n_v * n_h)) + 1.0
    wide = s.solve(np.array([1.0]), b)
    assert (wide["status"] == 0).all()
    for k in (0, 13, 31):
        one = s.solve(np.array([1.0]), b[k:k + 1])
        assert np.linalg.norm(wide["x"][k, 0] - one["x"][0, 0]) <= 1e-8 * np.linalg.norm(one["x"])
        assert abs(wide["rho"][k, 0] - one["rho"][0, 0]) <= 1e-8 * one["rho"][0, 0]
    s.close()
