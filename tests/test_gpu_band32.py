"""The FP32 passes of the separable A^T A on images large enough for
k_band_line and k_band_rows (one column, more than 440 x 440 points) and for
k_band (several columns).

They run inside mixed-precision solves only.  There the answer is decided by
the FP64 residual, so a wrong coefficient would not move it: it would cost
iterations.  Against the FP64 solve of the same system the solution has to
agree to 1e-6 (both at relative residual 1e-11, condition numbers below 1e4)
and the iteration count to 15% and 12 (two reliable updates' restarts).
"""
import numpy as np
import pytest

import problemgen as pg
from oracle import operators as ops

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2306_11067_gb300 import lcmg as L  # noqa: E402
from paper_2306_11067_gb300 import Solver  # noqa: E402

CASES = [  # n_v, n_h, r_v, r_h, right-hand sides
    (512, 576, 4, 4, 1),       # 17 taps, 16-byte words, one full segment of 512, a tile of 64 rows
    (544, 640, 15, 9, 1),      # 61 and 37 taps, a segment of 32 points
    (1088, 288, 16, 12, 1),    # 65 and 49 taps, boundary rows in the third segment, 32 rows past a tile
    (288, 352, 6, 3, 3),       # 25 and 13 taps, interleaved columns, single elements
    (16, 16512, 15, 4, 1),     # lines shorter than the band, every row a boundary row
]


@pytest.mark.parametrize("n_v,n_h,rv,rh,nrhs", CASES)
def test_mixed_solve_follows_fp64(n_v, n_h, rv, rh, nrhs):
    rng = pg.rng(11)
    def taps(r):
        f = np.exp(-0.5 * (np.arange(-r, r + 1) / (0.35 * r)) ** 2) * rng.uniform(0.8, 1.2, 2 * r + 1)
        return f / f.sum()
    fv, fh = taps(rv), taps(rh)
    d = pg.random_weights(ops.n_edges(n_v, n_h), 5, d_min=0.05)
    b = rng.standard_normal((nrhs, n_v * n_h)) + 1.0
    got = {}
    for prec in (L.PREC_FP64, L.PREC_MIXED):
        s = Solver(n_v, n_h, precision=prec, tol=1e-11, maxit=5000)
        s.set_forward_separable(fv, fh)
        assert s.forward_form() == L.FORM_SEPARABLE
        s.set_weights(d)
        got[prec] = s.solve(np.array([0.5]), b)
        s.close()
    a, m = got[L.PREC_FP64], got[L.PREC_MIXED]
    assert (m["status"] == 0).all() and (a["status"] == 0).all()
    for k in range(nrhs):
        ref = a["x"][k, 0]
        assert np.linalg.norm(m["x"][k, 0] - ref) <= 1e-6 * np.linalg.norm(ref)
    ia, im = np.asarray(a["iters"]).max(), np.asarray(m["iters"]).max()
    assert im <= 1.15 * ia + 12, (ia, im)
