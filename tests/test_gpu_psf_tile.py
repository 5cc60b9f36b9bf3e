"""The largest point-spread functions whose tile fits in shared memory (and
the first ones beyond, which run with one output per thread): the kernel's
tile and its own array of partial sums share the block's 48 KB.

The blur runs inside mixed-precision solves, whose solutions are decided by
the FP64 residual: those agree with FP64 solves to 1e-6 (both at relative
residual 1e-11, condition numbers below 1e4).
"""
import numpy as np
import pytest

import problemgen as pg
from oracle import operators as ops

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2306_11067_gb300 import lcmg as L  # noqa: E402
from paper_2306_11067_gb300 import Solver  # noqa: E402

CASES = [  # n_v, n_h, r_v, r_h: bytes of the tile
    (48, 64, 26, 40),     # tiles of 8 rows: 49120
    (64, 48, 43, 27),     # 49120
    (64, 64, 24, 39),     # 45328, a smaller one
    (32, 9728, 5, 97),    # tiles of 32 rows (304 of them): 49136
    (32, 9728, 0, 139),   # 49104
]


@pytest.mark.parametrize("n_v,n_h,rv,rh", CASES)
def test_largest_tiles_solve(n_v, n_h, rv, rh):
    rng = pg.rng(8)
    u, v = np.arange(-rv, rv + 1)[:, None], np.arange(-rh, rh + 1)[None, :]
    # of full rank or of too large a radius for the separable form
    psf = np.exp(-(0.8 * u + 0.6 * v) ** 2 / 9.0 - (0.8 * v - 0.6 * u) ** 2 / 2.0) * rng.uniform(0.7, 1.3, (2 * rv + 1, 2 * rh + 1))
    psf /= psf.sum()
    d = pg.random_weights(ops.n_edges(n_v, n_h), 4, d_min=0.05)
    b = rng.standard_normal((1, n_v * n_h)) + 1.0
    levels, a, c = 1, n_v, n_h
    while a * c > 1200 and a % 2 == 0 and c % 2 == 0:
        a, c, levels = a // 2, c // 2, levels + 1
    got = {}
    for prec in (L.PREC_FP64, L.PREC_MIXED):
        s = Solver(n_v, n_h, precision=prec, tol=1e-11, maxit=5000, levels=levels)
        s.set_forward_stencil(psf)
        assert s.forward_form() == L.FORM_PSF2D
        s.set_weights(d)
        got[prec] = s.solve(np.array([0.5]), b)
        s.close()
    a, m = got[L.PREC_FP64], got[L.PREC_MIXED]
    assert a["status"][0, 0] == 0 and m["status"][0, 0] == 0
    assert np.linalg.norm(m["x"] - a["x"]) <= 1e-6 * np.linalg.norm(a["x"])
