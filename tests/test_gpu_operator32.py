"""The FP32 operator passes output by output: banded passes of one and of
several columns on both sides of every size rule (separable.cu), tiles of the
2-D point-spread functions (psf_tile.cuh), boundary rows included.

After two PCG iterations x = a_0 p_0 + a_1 p_1, and p_1 holds M K p_0 with the
level operators in FP32, so a wrong coefficient of one row shows at the points
it touches, where the solution of a converged solve would hide it.  The same
two iterations in FP64 are the reference (their passes are compared with the
oracle elsewhere).  In a model of the FP32 operator and cycle on these
distributions (flat taps, lambda = 0.1) rounding moves x by at most 2e-7 of its
largest entry, and 2% in one coefficient of one boundary row by 1e-5 to 2e-3;
the bound is 2e-6, 32 units of FP32 rounding.  (That holds for sums of a few
hundred terms at most: the PSFs here stay small.)
"""
import numpy as np
import pytest

import problemgen as pg
from oracle import operators as ops

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2306_11067_gb300 import lcmg as L  # noqa: E402
from paper_2306_11067_gb300 import Solver  # noqa: E402


def _two_iterations(n_v, n_h, forward, form, rhs):
    rng = pg.rng(3)
    d = rng.uniform(0.3, 1.0, ops.n_edges(n_v, n_h))
    b = rng.standard_normal((rhs, n_v * n_h)) + 1.0
    x = {}
    for prec in (L.PREC_FP64, L.PREC_MIXED):
        s = Solver(n_v, n_h, precision=prec, tol=1e-15, maxit=2, smoother_fp16=0)
        forward(s)
        assert s.forward_form() == form
        s.set_weights(d)
        out = s.solve(np.array([0.1]), b)
        assert (out["iters"] == 2).all()
        x[prec] = out["x"][:, 0]
        s.close()
    for k in range(rhs):
        ref = x[L.PREC_FP64][k]
        err = np.abs(x[L.PREC_MIXED][k] - ref)
        assert err.max() <= 2e-6 * np.abs(ref).max(), (k, np.unravel_index(err.argmax(), (n_h, n_v)), err.max() / np.abs(ref).max())


@pytest.mark.parametrize("n_v,n_h,rv,rh,rhs", [
    (64, 48, 4, 4, 1),         # one output per thread, blocks of 64
    (320, 256, 9, 5, 1),       # ... of 256
    (62, 66, 15, 16, 1),       # lines of 2 mod 4 points
    (464, 432, 5, 9, 1),       # 21 (of 25) and 37 taps, ragged tiles and segments along both axes
    (464, 432, 15, 15, 1),     # 61 taps
    (464, 432, 16, 12, 1),     # 65 and 49
    (1056, 208, 3, 7, 1),      # 13 (of 17) and 29 (of 37) taps, boundary rows in the third segment
    (16, 12544, 15, 4, 1),     # every row along i a boundary row
    (12544, 16, 6, 12, 1),     # every row along j
    (96, 80, 5, 3, 3),         # several columns: one output per thread
    (160, 128, 4, 4, 4),       # tiles of 17 taps
    (160, 128, 9, 15, 4),      # of 37 and 61
    (160, 144, 6, 12, 3),      # of 25 and 49, in chunks
    (130, 66, 4, 6, 8),        # lines of 2 mod 4 points
])
def test_banded_passes(n_v, n_h, rv, rh, rhs):
    rng = pg.rng(5)
    fv, fh = rng.uniform(0.5, 1.5, 2 * rv + 1), rng.uniform(0.5, 1.5, 2 * rh + 1)
    _two_iterations(n_v, n_h, lambda s: s.set_forward_separable(fv / fv.sum(), fh / fh.sum()), L.FORM_SEPARABLE, rhs)


@pytest.mark.parametrize("n_v,n_h,rv,rh,rhs", [
    (40, 36, 1, 4, 1),     # words of taps with a remainder of three and one
    (72, 56, 7, 7, 1),     # ragged tiles
    (72, 56, 7, 6, 4),     # several columns
    (33, 27, 5, 2, 1),     # one level
    (640, 512, 2, 3, 1),   # tiles of 32 rows
])
def test_tiled_blur(n_v, n_h, rv, rh, rhs):
    psf = pg.rng(5).uniform(0.5, 1.5, (2 * rv + 1, 2 * rh + 1))
    _two_iterations(n_v, n_h, lambda s: s.set_forward_stencil(psf / psf.sum()), L.FORM_PSF2D, rhs)
