"""FP16 coarse levels of a cycle with two sweeps (the coefficients of a point in
one row, compact.cuh), on levels wider than a block of 64 points and with columns
interleaved, and after a cycle with one sweep on the same context (the other
layout in the same buffer): the oracle's model of the storage to 1e-5 (FP32
rounding, as on smaller grids)."""
import numpy as np
import pytest
import scipy.sparse as sp

import problemgen as pg
from oracle import multigrid as mg
from oracle import operators as ops

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2306_11067_gb300 import lcmg as L  # noqa: E402
from paper_2306_11067_gb300 import Solver  # noqa: E402


@pytest.mark.parametrize("n_v,n_h,levels,cols", [(136, 80, 3, 1), (208, 48, 4, 3), (68, 8, 2, 1)])
@pytest.mark.parametrize("smoother", [L.SMOOTH_L1_JACOBI, L.SMOOTH_JACOBI])
def test_two_sweeps_and_one(n_v, n_h, levels, cols, smoother):
    psf = pg.gaussian_psf(2, 1.0)
    s = Solver(n_v, n_h, levels=levels, smoother=smoother, nu=1, precision=L.PREC_MIXED)
    s.set_forward_stencil(psf)
    d = pg.random_weights(ops.n_edges(n_v, n_h), 9, d_min=0.02)
    s.set_weights(d)
    R = pg.rng(4).standard_normal((cols, n_v * n_h))
    rd = torch.tensor(R, device="cuda", dtype=torch.float64)
    zd = torch.empty_like(rd)
    diag = L.lcmg_get_diag(s.ctx, n_v * n_h)
    H = mg.build_hierarchy(mg.weighted_laplacian(ops.gradient(n_v, n_h), d), sp.diags(diag), n_v, n_h, levels)
    sm = "l1" if smoother == L.SMOOTH_L1_JACOBI else "jacobi"
    for nu in (1, 2, 1):
        s.set_params(nu=nu)
        L.lcmg_apply_vcycle_dev(s.ctx, np.full(cols, 0.1), rd, zd)
        V = mg.VCycle(H, 0.1, nu=nu, smoother=sm, storage="fp16")
        for k in {0, cols - 1}:
            ref = V(R[k])
            assert np.linalg.norm(zd[k].cpu().numpy() - ref) <= 1e-5 * np.linalg.norm(ref)
    s.close()
