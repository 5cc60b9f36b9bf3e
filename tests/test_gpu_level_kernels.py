"""Kernels whose tiles or strips are larger than the grids of the other tests:
the FP16 levels in strips of several rows and columns (vcoarse.cuh, vfine.cuh),
Galerkin products of several 32 x 2 tiles, the tiled blur (psf_tile.cuh).

Cycles agree with the oracle's model of the same storage to 1e-5 (FP32
rounding, as on smaller grids); Galerkin stencils with scipy's triple product
to 1e-13 of the largest entry (FP64, sums of at most 1600 positive-weight
terms); the blur runs inside mixed-precision solves, whose solutions are
decided by the FP64 residual: those agree with FP64 solves to 1e-6, and a wrong
operator would show in the iteration count (bound: 15% and 12, the restarts of
two reliable updates).
"""
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


@pytest.mark.parametrize("n_v,n_h,levels,cols", [
    (240, 512, 5, 8),   # level 1 in strips of more than one coarse row, columns interleaved
    (136, 80, 3, 1),    # 68 and 34 coarse columns: strips of 30, 28, ragged
    (640, 36, 3, 2),    # 18 and 9 coarse rows
    (68, 8, 2, 1),      # one level, 4 coarse rows
])
@pytest.mark.parametrize("smoother", [L.SMOOTH_L1_JACOBI, L.SMOOTH_JACOBI])
def test_cycle_in_strips_matches_its_model(n_v, n_h, levels, cols, smoother):
    fv, fh = pg.gaussian_psf(2, 1.0)[:, 2], pg.gaussian_psf(2, 1.0)[2, :]
    psf = np.outer(fv / fv.sum(), fh / fh.sum())
    s = Solver(n_v, n_h, levels=levels, smoother=smoother, nu=1, vfuse=2, precision=L.PREC_MIXED)
    s.set_forward_stencil(psf)
    d = pg.random_weights(ops.n_edges(n_v, n_h), 9, d_min=0.02)
    s.set_weights(d)
    R = pg.rng(4).standard_normal((cols, n_v * n_h))
    rd = torch.tensor(R, device="cuda", dtype=torch.float64)
    zd = torch.empty_like(rd)
    diag = L.lcmg_get_diag(s.ctx, n_v * n_h)
    H = mg.build_hierarchy(mg.weighted_laplacian(ops.gradient(n_v, n_h), d), sp.diags(diag), n_v, n_h, levels)
    lam = 0.1
    L.lcmg_apply_vcycle_dev(s.ctx, np.full(cols, lam), rd, zd)
    V = mg.VCycle(H, lam, nu=1, smoother="l1" if smoother == L.SMOOTH_L1_JACOBI else "jacobi", storage="fp16")
    for k in {0, cols - 1}:
        ref = V(R[k])
        assert np.linalg.norm(zd[k].cpu().numpy() - ref) <= 1e-5 * np.linalg.norm(ref)
    s.close()


@pytest.mark.parametrize("n_v,n_h,levels,cols", [(512, 384, 6, 1), (256, 176, 5, 2), (20, 12, 2, 1)])
def test_fp64_cycle_in_tiles_of_every_size(n_v, n_h, levels, cols):
    """k_vdown64 / k_vup64 with 8, 4 and 2 coarse points a side, against the oracle's
    cycle to 1e-12 (FP64 rounding, summed in other orders)."""
    s = Solver(n_v, n_h, levels=levels, nu=1)
    s.set_forward_stencil(pg.gaussian_psf(2, 1.0))
    d = pg.random_weights(ops.n_edges(n_v, n_h), 9, d_min=0.05)
    s.set_weights(d)
    R = pg.rng(4).standard_normal((cols, n_v * n_h))
    rd = torch.tensor(R, device="cuda", dtype=torch.float64)
    zd = torch.empty_like(rd)
    diag = L.lcmg_get_diag(s.ctx, n_v * n_h)
    H = mg.build_hierarchy(mg.weighted_laplacian(ops.gradient(n_v, n_h), d), sp.diags(diag), n_v, n_h, levels)
    L.lcmg_apply_vcycle_dev(s.ctx, np.full(cols, 0.3), rd, zd)
    for k in range(cols):
        ref = mg.VCycle(H, 0.3, nu=1)(R[k])
        assert np.linalg.norm(zd[k].cpu().numpy() - ref) <= 1e-12 * np.linalg.norm(ref)
    s.close()


@pytest.mark.parametrize("n_v,n_h,levels", [(140, 72, 3), (12, 10, 2), (4, 130, 2), (256, 6, 2)])
def test_galerkin_tiles(n_v, n_h, levels):
    s = Solver(n_v, n_h, levels=levels)
    s.set_forward_stencil(pg.gaussian_psf(2, 1.0))
    d = pg.random_weights(ops.n_edges(n_v, n_h), 5, d_min=0.05)
    s.set_weights(d)
    z = torch.zeros(1, n_v * n_h, device="cuda", dtype=torch.float64)
    L.lcmg_apply_vcycle_dev(s.ctx, np.array([0.3]), z, torch.empty_like(z))  # builds the hierarchy
    diag = L.lcmg_get_diag(s.ctx, n_v * n_h)
    H = mg.build_hierarchy(mg.weighted_laplacian(ops.gradient(n_v, n_h), d), sp.diags(diag), n_v, n_h, levels)
    for k in range(1, levels):
        nv, nh, gl, ga = L.lcmg_get_level(s.ctx, k)
        for got, ref in ((gl, H.G_L[k]), (ga, H.G_A[k])):
            ref = ref.tocsr()
            n = nv * nh
            i, j = np.arange(n) % nv, np.arange(n) // nv
            acc = sp.csr_matrix((n, n))
            for o in range(25):
                di, dj = o % 5 - 2, o // 5 - 2
                ok = (i + di >= 0) & (i + di < nv) & (j + dj >= 0) & (j + dj < nh)
                assert (np.asarray(got[o])[~ok] == 0).all()
                p = np.arange(n)[ok]
                acc = acc + sp.csr_matrix((np.asarray(got[o])[ok], (p, p + di + dj * nv)), shape=(n, n))
            assert abs(acc - ref).max() <= 1e-13 * abs(ref).max()
    s.close()


@pytest.mark.parametrize("n_v,n_h,kv,kh", [
    (40, 36, 1, 4),     # 3 and 9 taps: words of taps with a remainder of three and one
    (72, 56, 7, 7),     # ragged tiles
    (33, 27, 5, 2),     # one level
    (80, 96, 34, 34),   # too large for the tiles: one output per thread
    (640, 512, 2, 3),   # tiles of 32 rows
])
def test_mixed_blur_follows_fp64(n_v, n_h, kv, kh):
    rng = pg.rng(5)
    u, v = np.arange(-kv, kv + 1)[:, None], np.arange(-kh, kh + 1)[None, :]
    psf = np.exp(-(0.8 * u + 0.6 * v) ** 2 / 9.0 - (0.8 * v - 0.6 * u) ** 2 / 2.0) * rng.uniform(0.7, 1.3, (2 * kv + 1, 2 * kh + 1))
    psf /= psf.sum()
    d = pg.random_weights(ops.n_edges(n_v, n_h), 4, d_min=0.05)
    b = rng.standard_normal((1, n_v * n_h)) + 1.0
    got = {}
    for prec in (L.PREC_FP64, L.PREC_MIXED):
        s = Solver(n_v, n_h, precision=prec, tol=1e-11, maxit=5000)
        s.set_forward_stencil(psf)
        assert s.forward_form() == L.FORM_PSF2D
        s.set_weights(d)
        got[prec] = s.solve(np.array([0.5]), b)
        s.close()
    a, m = got[L.PREC_FP64], got[L.PREC_MIXED]
    assert a["status"][0, 0] == 0 and m["status"][0, 0] == 0
    assert np.linalg.norm(m["x"] - a["x"]) <= 1e-6 * np.linalg.norm(a["x"])
    assert m["iters"][0, 0] <= 1.15 * a["iters"][0, 0] + 12, (a["iters"], m["iters"])
