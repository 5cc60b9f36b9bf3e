"""The coarsest-level inverse (blocked, 16 x 16 tiles): with one
level the V-cycle is the exact solve K(lam)^{-1} r, compared with numpy's
dense solve.  Sizes on both sides of a tile's edge, one tile and many, one
column and several lambda at once."""
import numpy as np
import pytest

import problemgen as pg
from oracle import operators as ops

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2306_11067_gb300 import lcmg as L  # noqa: E402
from paper_2306_11067_gb300 import Solver  # noqa: E402


@pytest.mark.parametrize("n_v,n_h", [(2, 2), (3, 5), (4, 4), (17, 2), (8, 4), (7, 7), (16, 16), (31, 33)])
@pytest.mark.parametrize("lams", [[0.3], [0.05, 0.7, 4.0]])
def test_one_level_cycle_is_the_exact_solve(n_v, n_h, lams):
    n = n_v * n_h
    psf = pg.gaussian_psf(1, 0.8)
    d = pg.random_weights(ops.n_edges(n_v, n_h), 7, d_min=0.05)
    r = pg.rng(3).standard_normal((len(lams), n))
    s = Solver(n_v, n_h, levels=1)
    s.set_forward_stencil(psf)
    s.set_weights(d)
    rd = torch.from_numpy(r).cuda()
    zd = torch.empty_like(rd)
    L.lcmg_apply_vcycle_dev(s.ctx, lams, rd, zd)
    z = zd.cpu().numpy()
    diag = L.lcmg_get_diag(s.ctx, n)
    s.close()
    Lg = ops.gradient(n_v, n_h).toarray()
    G = Lg.T @ (d[:, None] ** 2 * Lg)
    for k, lam in enumerate(lams):
        K = lam * lam * G + np.diag(diag)
        ref = np.linalg.solve(K, r[k])
        # a stable inverse and its product: n eps cond(K) bounds the error
        bound = n * 2.0 ** -53 * np.linalg.cond(K) + 1e-15
        assert np.linalg.norm(z[k] - ref) <= bound * np.linalg.norm(ref)
