"""The work that is timed: what a program has this library do, over its range of sizes.

A case names an entry point of ``lcmg`` and a problem: the operator
application that needs no context (``operator``), solves of

    (A^T A + lambda^2 L^T D^2 L) x = A^T b

for a list of lambda (``solve``), Algorithm 2 from end to end (``lcurve``),
and a new weight vector followed by an application of the preconditioner
(``precond``, for a program that runs a Krylov method of its own).  The
forward operator A is a ray-length matrix (``ct``), a blur as a sparse
matrix (``blur_csr``), a blur given by its 1-D factors (``sep``) or a blur
whose point-spread function has no such factors (``psf``).

The lambda are those where the L-curve bends and above, and the tolerances
are tight enough for the answer to be determined by the system: at a loose
tolerance the result is a matter of where the iteration stopped.  Iteration
counts are left out of the outputs for the same reason.
"""
import functools
import math

import numpy as np
import torch

from paper_2306_11067_gb300 import lcmg

DEV = "cuda:0"


# ---------------------------------------------------------------------------
# The cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # One application of the operator, nothing allocated: the inner call
        # of a caller's own iteration on the smallest grid; all latency.
        dict(name="operator32", what="operator", n_v=32, n_h=32, fwd="blur_csr", r_v=4, r_h=4, s_v=1.5, s_h=1.5,
             cols=1, weights="edges"),
        # The smallest solve, from host arrays to host arrays: a 32 x 32 blur
        # as a sparse matrix in FP64 (the default precision), one lambda.
        dict(name="solve32", what="solve", n_v=32, n_h=32, fwd="blur_csr", r_v=4, r_h=4, s_v=1.5, s_h=1.5, mixed=False,
             batched=False, levels=3, lam_lo=0.05, lam_hi=0.05, n_lam=1, rhs=1, tol=1e-12, weights="ones", host=True),
        # A grid of odd sides, which cannot be coarsened: a crop as it comes.
        dict(name="odd27x21", what="solve", n_v=27, n_h=21, fwd="sep", r_v=4, r_h=4, s_v=1.5, s_h=1.5, mixed=False,
             batched=False, levels=0, lam_lo=0.1, lam_hi=1.0, n_lam=2, rhs=1, tol=1e-12, weights="edges", host=True),
        # Algorithm 2 end to end on a small image: the call most programs make.
        dict(name="lcurve64", what="lcurve", n_v=64, n_h=64, fwd="sep", r_v=9, r_h=9, s_v=3.0, s_h=3.0, mixed=False,
             batched=False, levels=3, lam_lo=0.05, lam_hi=1.0, n_lam=12, rhs=1, tol=1e-12, weights="ones", outer=3),
        # Limited-angle CT, all lambda of a window advanced as one batch.
        dict(name="ct128_batched", what="solve", n_v=128, n_h=128, fwd="ct", angles=66, bins=183, mixed=True,
             batched=True, levels=0, lam_lo=0.5, lam_hi=4.0, n_lam=10, rhs=1, tol=1e-13, weights="edges", host=False),
        # 256 x 256 CT, the warm-start chain over lambda in mixed precision:
        # the operator is a streamed sparse matrix of 15M nonzeros.
        dict(name="ct256", what="solve", n_v=256, n_h=256, fwd="ct", angles=180, bins=363, mixed=True,
             batched=False, levels=0, lam_lo=0.5, lam_hi=4.0, n_lam=4, rhs=1, tol=1e-13, weights="edges", host=False),
        # The anisotropic blur of the deblurring experiment on a grid that is
        # not square, FP64 chain.
        dict(name="aniso240x176", what="solve", n_v=240, n_h=176, fwd="sep", r_v=6, r_h=7, s_v=4.7, s_h=4.1, mixed=False,
             batched=False, levels=0, lam_lo=0.1, lam_hi=1.0, n_lam=4, rhs=1, tol=1e-12, weights="edges", host=False),
        # A motion blur (a tilted ridge, no 1-D factors), mixed chain.
        dict(name="motion200x152", what="solve", n_v=200, n_h=152, fwd="psf", r_v=7, r_h=7, s_v=3.0, s_h=1.0, mixed=True,
             batched=False, levels=0, lam_lo=0.1, lam_hi=1.0, n_lam=3, rhs=1, tol=1e-12, weights="edges", host=False),
        # Four images of one camera: their chains share each lambda.
        dict(name="deblur512_rhs4", what="solve", n_v=512, n_h=512, fwd="sep", r_v=9, r_h=9, s_v=3.0, s_h=3.0, mixed=True,
             batched=False, levels=6, lam_lo=0.1, lam_hi=1.0, n_lam=3, rhs=4, tol=1e-12, weights="edges", host=False),
        # New weights (the Galerkin hierarchy is rebuilt) and one FP64 cycle
        # on two vectors, as preconditioner of a caller's own method.
        dict(name="weights512x320", what="precond", n_v=512, n_h=320, fwd="sep", r_v=9, r_h=9, s_v=3.0, s_h=3.0,
             mixed=False, levels=0, lam_lo=0.1, lam_hi=1.0, n_lam=2, weights="edges"),
        # A large image in FP64, one lambda.
        dict(name="deblur1024_fp64", what="solve", n_v=1024, n_h=1024, fwd="sep", r_v=15, r_h=15, s_v=5.0, s_h=5.0,
             mixed=False, batched=False, levels=0, lam_lo=0.3, lam_hi=0.3, n_lam=1, rhs=1, tol=1e-12, weights="edges",
             host=False),
        # 2048 x 2048 deblurring with the weights of the second outer
        # iteration, mixed precision, three lambda of its window.
        dict(name="deblur2048", what="solve", n_v=2048, n_h=2048, fwd="sep", r_v=15, r_h=15, s_v=5.0, s_h=5.0, mixed=True,
             batched=False, levels=10, lam_lo=0.2, lam_hi=1.0, n_lam=3, rhs=1, tol=1e-12, weights="edges", host=False),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _side(rng, lo, hi):
    """A side that coarsens to at most 20 or so: an odd number or twice one, times a power of two."""
    s = _log(rng, lo, hi)
    k = max(0, round(math.log2(s / 14)))
    return max(8, round(s / 2 ** k)) * 2 ** k


def _sides(rng, lo, hi):
    a = _side(rng, lo, hi)
    return dict(n_v=a, n_h=_side(rng, max(lo, a / 2), min(hi, 2 * a)))


def draw(rng):
    """One more case of the same ranges."""
    kind = rng.choice(["operator", "small", "odd", "lcurve", "ct", "sep", "sep", "psf", "rhs", "precond", "large"])
    c = dict(what="solve", batched=False, levels=0, rhs=1, tol=1e-12, weights=rng.choice(["ones", "edges"]), host=False,
             mixed=rng.random() < 0.5)

    def blur(r_hi):
        for a in "vh":
            r = max(2, round(_log(rng, 2, r_hi)))
            c["r_" + a], c["s_" + a] = r, round(r / rng.uniform(2.4, 3.2), 2)

    def lams(lo, n):
        c["lam_lo"], c["n_lam"] = round(_log(rng, lo, 3 * lo), 3), n
        c["lam_hi"] = c["lam_lo"] if n == 1 else round(c["lam_lo"] * _log(rng, 2, 8), 3)

    if kind == "operator":
        blur(5)
        c = dict(what="operator", n_v=rng.randrange(9, 90), n_h=rng.randrange(9, 90), fwd="blur_csr", cols=rng.choice([1, 1, 2, 5]),
                 weights=c["weights"], **{k: c[k] for k in ("r_v", "r_h", "s_v", "s_h")})
    elif kind == "small":
        c.update(**_sides(rng, 16, 72), fwd="blur_csr", host=True)
        blur(4)
        lams(0.05, rng.choice([1, 2]))
    elif kind == "odd":
        c.update(n_v=rng.randrange(15, 35, 2), n_h=rng.randrange(15, 29, 2), fwd="sep", host=True)
        blur(5)
        lams(0.1, rng.choice([1, 2]))
    elif kind == "lcurve":
        c.update(what="lcurve", **_sides(rng, 32, 128), fwd="sep", weights="ones", n_lam=rng.randrange(10, 14),
                 lam_lo=0.05, lam_hi=1.0, outer=2)
        blur(9)
    elif kind == "ct":
        s = _side(rng, 48, 224)
        c.update(n_v=s, n_h=s, fwd="ct", angles=rng.randrange(s // 2, s), bins=2 * math.ceil(0.71 * s) - 1, mixed=True,
                 batched=rng.random() < 0.4, tol=1e-13)
        lams(0.5, rng.randrange(2, 7))
    elif kind == "sep":
        c.update(**_sides(rng, 100, 1000), fwd="sep")
        blur(15)
        lams(0.1, rng.choice([1, 2, 3]) if c["n_v"] * c["n_h"] < 3e5 or c["mixed"] else 1)
    elif kind == "psf":
        c.update(**_sides(rng, 60, 200), fwd="psf", mixed=True, r_v=rng.randrange(3, 9),
                 r_h=rng.randrange(3, 9), s_v=3.0, s_h=1.0)
        lams(0.1, rng.choice([1, 2]))
    elif kind == "rhs":
        c.update(**_sides(rng, 100, 600), fwd="sep", mixed=True, rhs=rng.choice([2, 3, 4]))
        blur(12)
        lams(0.1, rng.choice([1, 2]))
    elif kind == "precond":
        c = dict(what="precond", **_sides(rng, 60, 800), fwd="sep", mixed=False, levels=0,
                 weights="edges")
        blur(12)
        lams(0.1, rng.choice([1, 2]))
    else:
        c.update(**_sides(rng, 1000, 1900), fwd="sep", mixed=True)
        blur(15)
        lams(0.2, rng.choice([1, 2]))
    return c


# ---------------------------------------------------------------------------
# Inputs.  An image is a tensor [n_h, n_v]: pixel (i, j) at [j, i], so that
# its flat index is i + j n_v.
# ---------------------------------------------------------------------------
def _gauss(r, s):
    u = torch.arange(-r, r + 1, dtype=torch.float64)
    f = torch.exp(-u * u / (2 * s * s))
    return f / f.sum()


def _ridge(case):
    """A tilted anisotropic Gaussian: a point-spread function of full rank."""
    u = torch.arange(-case["r_v"], case["r_v"] + 1, dtype=torch.float64)[:, None]
    v = torch.arange(-case["r_h"], case["r_h"] + 1, dtype=torch.float64)[None, :]
    a, b = 0.8 * u + 0.6 * v, -0.6 * u + 0.8 * v
    f = torch.exp(-a * a / (2 * case["s_v"] ** 2) - b * b / (2 * case["s_h"] ** 2))
    return f / f.sum()


def _correlate(x, f, dim):
    """sum_u f[u + r] x(. + u) along dim, zero outside."""
    r, n, out = len(f) // 2, x.shape[dim], torch.zeros_like(x)
    for u in range(-min(r, n - 1), min(r, n - 1) + 1):
        k = n - abs(u)
        out.narrow(dim, max(0, -u), k).add_(x.narrow(dim, max(0, u), k), alpha=float(f[u + r]))
    return out


@functools.lru_cache(maxsize=4)
def _ct(n, angles, bins):
    """Ray lengths of an n x n image for parallel beams over 180 degrees: CSR in FP32 (host) of exact intersections."""
    half, dt = n / 2.0, dict(dtype=torch.float64, device=DEV)
    th = torch.arange(angles, **dt) * (math.pi / angles)
    c, s = torch.cos(th)[:, None].clone(), torch.sin(th)[:, None].clone()
    off = torch.arange(bins, **dt)[None, :] - (bins - 1) / 2.0
    px, py = (off * c).reshape(-1, 1), (off * s).reshape(-1, 1)
    dx, dy = (-s).expand(-1, bins).reshape(-1, 1).clone(), c.expand(-1, bins).reshape(-1, 1).clone()
    dx[dx.abs() < 1e-9] = 1e-9
    dy[dy.abs() < 1e-9] = 1e-9
    lines = torch.arange(n + 1, **dt)[None, :] - half
    tx, ty = (lines - px) / dx, (lines - py) / dy
    t0 = torch.maximum(torch.minimum(tx[:, :1], tx[:, -1:]), torch.minimum(ty[:, :1], ty[:, -1:]))
    t1 = torch.minimum(torch.maximum(tx[:, :1], tx[:, -1:]), torch.maximum(ty[:, :1], ty[:, -1:]))
    t = torch.cat([tx, ty], 1)
    t = torch.minimum(torch.maximum(t, t0), torch.maximum(t0, t1)).sort(1).values
    length, mid = t.diff(dim=1), 0.5 * (t[:, 1:] + t[:, :-1])
    col, row = torch.floor(px + mid * dx + half).long(), torch.floor(half - (py + mid * dy)).long()
    ok = (length > 1e-6) & (col >= 0) & (col < n) & (row >= 0) & (row < n)
    ptr = torch.zeros(angles * bins + 1, dtype=torch.int64)
    ptr[1:] = ok.sum(1).cumsum(0).cpu()
    return ptr.numpy(), (row + col * n)[ok].to(torch.int32).cpu().numpy(), length[ok].float().cpu().numpy()


@functools.lru_cache(maxsize=8)
def _blur_csr(n_v, n_h, r_v, r_h, s_v, s_h):
    """The blur with zero boundary as a CSR matrix in FP64 (host)."""
    fv, fh = _gauss(r_v, s_v).numpy(), _gauss(r_h, s_h).numpy()
    j, i, v, u = np.meshgrid(np.arange(n_h), np.arange(n_v), np.arange(-r_h, r_h + 1), np.arange(-r_v, r_v + 1), indexing="ij")
    ok = (i + u >= 0) & (i + u < n_v) & (j + v >= 0) & (j + v < n_h)
    ptr = np.zeros(n_v * n_h + 1, np.int64)
    ptr[1:] = np.cumsum(ok.reshape(n_v * n_h, -1).sum(1))
    return ptr, ((i + u) + (j + v) * n_v)[ok].astype(np.int32), (fv[u + r_v] * fh[v + r_h])[ok]


def _csr(case):
    if case["fwd"] == "ct":
        return _ct(case["n_v"], case["angles"], case["bins"])
    return _blur_csr(*(case[k] for k in ("n_v", "n_h", "r_v", "r_h", "s_v", "s_h")))


def _transposed(ptr, col, val, n):
    """The CSR arrays of the transpose (rows of A in increasing order)."""
    order = np.argsort(col, kind="stable")
    tptr = np.zeros(n + 1, np.int64)
    tptr[1:] = np.cumsum(np.bincount(col, minlength=n))
    rows = np.repeat(np.arange(len(ptr) - 1, dtype=np.int32), np.diff(ptr))
    return tptr, rows[order], val[order]


class _Forward:
    """A and A^T in plain torch, FP64, on vectors of the flat image."""

    def __init__(self, case):
        self.case, self.shape = case, (case["n_h"], case["n_v"])
        if case["fwd"] in ("ct", "blur_csr"):
            ptr, col, val = _csr(case)
            n = case["n_v"] * case["n_h"]

            def up(p, c, v, cols):
                return torch.sparse_csr_tensor(torch.from_numpy(p), torch.from_numpy(c.astype(np.int64)),
                                               torch.from_numpy(v.astype(np.float64)), size=(len(p) - 1, cols), device=DEV)
            self.a, self.at = up(ptr, col, val, n), up(*_transposed(ptr, col, val, n), len(ptr) - 1)
            self.diag = torch.mv(up(*_transposed(ptr, col, val.astype(np.float64) ** 2, n), len(ptr) - 1),
                                 torch.ones(len(ptr) - 1, dtype=torch.float64, device=DEV))
            self.apply, self.transpose = (lambda x: torch.mv(self.a, x)), (lambda y: torch.mv(self.at, y))
        elif case["fwd"] == "sep":
            fv, fh = _gauss(case["r_v"], case["s_v"]), _gauss(case["r_h"], case["s_h"])

            def both(x, gv, gh):
                return _correlate(_correlate(x.reshape(self.shape), gv, 1), gh, 0).reshape(-1)
            self.apply = lambda x: both(x, fv, fh)
            self.transpose = lambda y: both(y, fv.flip(0), fh.flip(0))
            one = torch.ones(self.shape[0] * self.shape[1], dtype=torch.float64, device=DEV)
            self.diag = both(one, fv.flip(0) ** 2, fh.flip(0) ** 2)
        else:
            psf = _ridge(case)
            pad = (case["r_h"], case["r_v"])

            def conv(x, f):  # f[u, v]: u along i (the last axis of an image), v along j
                return torch.nn.functional.conv2d(x.reshape(1, 1, *self.shape), f.T[None, None].contiguous().to(DEV), padding=pad).reshape(-1)
            self.apply, self.transpose = (lambda x: conv(x, psf)), (lambda y: conv(y, psf.flip(0, 1)))
            self.diag = conv(torch.ones(self.shape[0] * self.shape[1], dtype=torch.float64, device=DEV), psf.flip(0, 1) ** 2)


def _image(case, gen):
    """Piecewise constant: rectangles and ellipses, later ones over earlier ones."""
    nv, nh = case["n_v"], case["n_h"]
    i = torch.arange(nv, dtype=torch.float64, device=DEV)[None, :] + 0.5
    j = torch.arange(nh, dtype=torch.float64, device=DEV)[:, None] + 0.5
    img = torch.zeros(nh, nv, dtype=torch.float64, device=DEV)
    for k in range(14):
        p = torch.rand(6, generator=gen, dtype=torch.float64).tolist()
        di, dj = (i - p[0] * nv) / (nv * (1 + 3 * p[2]) / 16), (j - p[1] * nh) / (nh * (1 + 3 * p[3]) / 16)
        inside = torch.maximum(di.abs(), dj.abs()) <= 1 if k % 2 else di ** 2 + dj ** 2 <= 1
        img = torch.where(inside, 0.1 + 0.9 * p[4], img)
    return img


def _grad(x, shape):
    x = x.reshape(shape)
    return torch.cat([(x[:, 1:] - x[:, :-1]).reshape(-1), (x[1:] - x[:-1]).reshape(-1)])


def _grad_t(e, shape):
    nh, nv = shape
    a, b = e[:nh * (nv - 1)].reshape(nh, nv - 1), e[nh * (nv - 1):].reshape(nh - 1, nv)
    out = torch.zeros(shape, dtype=e.dtype, device=e.device)
    out[:, 1:] += a
    out[:, :-1] -= a
    out[1:] += b
    out[:-1] -= b
    return out.reshape(-1)


def _next_weights(d, x, shape):
    """The weight update after a solution x, from d: large weighted differences lose their weight."""
    v = (d * _grad(x, shape)).abs()
    return torch.clamp(1 - (v / v.max()) ** 2, min=1e-3) * d


def _lambdas(case):
    n = case["n_lam"]
    return np.array([case["lam_lo"]]) if n == 1 else np.geomspace(case["lam_lo"], case["lam_hi"], n)


def _inputs(case, seed):
    """Images, data b [rhs, m] with 1% noise, edge weights d, a random vector per column."""
    gen = torch.Generator().manual_seed(1000003 * seed + 17)
    A, shape = _Forward(case), (case["n_h"], case["n_v"])
    rows = []
    for _ in range(case.get("rhs", 1)):
        img = _image(case, gen)
        b = A.apply(img.reshape(-1))
        e = torch.randn(b.numel(), generator=gen, dtype=torch.float64).to(DEV)
        rows.append(b + 0.01 * b.norm() * e / e.norm())
    d = torch.ones(_grad(img, shape).numel(), dtype=torch.float64, device=DEV)
    if case["weights"] == "edges":  # of a first, blurred reconstruction
        f = _gauss(2, 1.0)
        d = _next_weights(d, _correlate(_correlate(img, f, 0), f, 1).reshape(-1), shape)
    cols = case.get("cols", case.get("n_lam", 1))
    v = torch.randn(cols, img.numel(), generator=gen, dtype=torch.float64).to(DEV) + 1.0
    return A, torch.stack(rows), d, v


# ---------------------------------------------------------------------------
# What a program has in hand, and the call
# ---------------------------------------------------------------------------
class _Csr:
    def __init__(self, ptr, col, val, n):
        self.m, self.n, self.row_ptr, self.col, self.val = len(ptr) - 1, n, ptr, col, val


def prepare(case, seed):
    _, b, d, v = _inputs(case, seed)
    n = case["n_v"] * case["n_h"]
    st = dict(case=case, lam=_lambdas(case) if "n_lam" in case else np.geomspace(0.1, 1.0, case["cols"]), b=b, d=d, v=v)
    if case["what"] == "operator":
        ptr, col, val = _csr(case)
        st["csr"] = [torch.from_numpy(a).to(DEV) for a in (ptr, col, val, *_transposed(ptr, col, val, n))]
        st["out"] = torch.empty_like(v)
        return st
    s = lcmg.Solver(case["n_v"], case["n_h"], levels=case["levels"], tol=case.get("tol", 1e-6), maxit=20000,
                    precision=lcmg.PREC_MIXED if case["mixed"] else lcmg.PREC_FP64,
                    mode=lcmg.MODE_BATCHED if case.get("batched") else lcmg.MODE_SEQUENTIAL)
    if case["fwd"] in ("ct", "blur_csr"):
        s.set_forward_csr(_Csr(*_csr(case), n))
    elif case["fwd"] == "sep":
        s.set_forward_separable(_gauss(case["r_v"], case["s_v"]).numpy(), _gauss(case["r_h"], case["s_h"]).numpy())
    else:
        s.set_forward_stencil(_ridge(case).numpy())
    st["solver"] = s
    if case["what"] == "solve":
        lcmg.lcmg_set_weights_dev(s.ctx, d, d.numel())
        shape = (case["rhs"], case["n_lam"])
        st["x"] = torch.empty(*shape, n, dtype=torch.float64, device=DEV)
        st["rho"], st["eta"] = (torch.empty(shape, dtype=torch.float64, device=DEV) for _ in range(2))
        st["status"] = torch.empty(shape, dtype=torch.int32, device=DEV)
    elif case["what"] == "precond":
        st["out"] = torch.empty_like(v)
    if case.get("host") or case["what"] == "lcurve":
        st["b"] = b.cpu().numpy()
    return st


def run(st):
    case = st["case"]
    if case["what"] == "operator":
        lcmg.lcmg_apply_normal_noalloc(0, None, case["n_v"], case["n_h"], st["csr"][0].numel() - 1, *st["csr"], st["d"],
                                       st["lam"], st["v"], st["out"])
        return st["out"]
    s = st["solver"]
    if case["what"] == "lcurve":
        r = s.lcurve_run(st["lam"], st["b"][0], max_outer=case["outer"])
        return r["x"], np.array(r["history"]), r["n_solves"], r["n_converged"]
    if case["what"] == "precond":
        lcmg.lcmg_set_weights_dev(s.ctx, st["d"], st["d"].numel())
        lcmg.lcmg_apply_vcycle_dev(s.ctx, st["lam"], st["v"], st["out"])
        return st["out"]
    if case["host"]:
        r = s.solve(st["lam"], st["b"])
        return r["x"], r["rho"], r["eta"], r["status"]
    lcmg.lcmg_solve_dev(s.ctx, st["lam"], st["b"], st["x"], rho_dev=st["rho"], eta_dev=st["eta"], status_dev=st["status"])
    return st["x"], st["rho"], st["eta"], st["status"]


def work(case):
    """The operator and the weights read once, each vector in and out once; for each column one application of the
    operator (how many a solve takes is the method's business)."""
    n = case["n_v"] * case["n_h"]
    m = n
    if case["fwd"] == "ct":
        m = case["angles"] * case["bins"]
        nnz = int(m * 0.9 * case["n_v"])
        op, fl = 8 * nnz, 4 * nnz
    elif case["fwd"] == "blur_csr":
        nnz = n * (2 * case["r_v"] + 1) * (2 * case["r_h"] + 1)
        op, fl = 12 * nnz, 4 * nnz
    else:
        taps = (2 * case["r_v"] + 1, 2 * case["r_h"] + 1)
        op, fl = 8 * (sum(taps) if case["fwd"] == "sep" else taps[0] * taps[1]), 4 * n * (sum(taps) if case["fwd"] == "sep" else taps[0] * taps[1])
    cols = case["cols"] if case["what"] == "operator" else case["n_lam"] * case.get("rhs", 1)
    outs = 1 if case["what"] == "lcurve" else cols
    ins = cols * n if case["what"] in ("operator", "precond") else case.get("rhs", 1) * m
    return {"bytes": op + 16 * n + 8 * ins + 8 * outs * n, "flops": cols * (fl + 12 * n)}


# ---------------------------------------------------------------------------
# The same in 64 bits, from plain torch
# ---------------------------------------------------------------------------
def _normal(A, d, lam, x, shape):
    return A.transpose(A.apply(x)) + lam * lam * _grad_t(d * d * _grad(x, shape), shape)


def _solve64(A, d, lam, c, x, shape):
    """Conjugate gradients with the diagonal as preconditioner, restarted until the true residual is at rounding."""
    w = d * d
    nh, nv = shape
    dl = torch.zeros(shape, dtype=torch.float64, device=DEV)
    a, b = w[:nh * (nv - 1)].reshape(nh, nv - 1), w[nh * (nv - 1):].reshape(nh - 1, nv)
    dl[:, 1:] += a
    dl[:, :-1] += a
    dl[1:] += b
    dl[:-1] += b
    inv = 1 / (A.diag + lam * lam * dl.reshape(-1))
    for goal in (1e-13, 3e-15):
        r = c - _normal(A, d, lam, x, shape)
        z = inv * r
        p, rz = z.clone(), r @ z
        stop = goal * float(c.norm())
        for it in range(6000):
            q = _normal(A, d, lam, p, shape)
            al = rz / (p @ q)
            x = x + al * p
            r = r - al * q
            if it % 10 == 9 and float(r.norm()) <= stop:
                break
            z = inv * r
            rz, old = r @ z, rz
            p = z + (rz / old) * p
    return x


def _corner(rho, eta):
    """The interior point of largest positive Menger curvature of the log-log curve."""
    u, v = np.log10(rho), np.log10(eta)
    kap = np.full(len(u), -np.inf)
    for i in range(1, len(u) - 1):
        a, b = np.array([u[i] - u[i - 1], v[i] - v[i - 1]]), np.array([u[i + 1] - u[i], v[i + 1] - v[i]])
        kap[i] = 2 * (a[0] * b[1] - a[1] * b[0]) / (np.hypot(*a) * np.hypot(*b) * np.hypot(*(a + b)))
    return int(np.argmax(kap))


def _sweep64(A, d, lams, b, x, shape):
    c, xs = A.transpose(b), [None] * len(lams)
    for k in reversed(range(len(lams))):
        x = xs[k] = _solve64(A, d, float(lams[k]), c, x, shape)
    rho = [(A.apply(x) - b).norm() for x in xs]
    eta = [(d * _grad(x, shape)).norm() for x in xs]
    return torch.stack(xs), torch.stack(rho), torch.stack(eta)


def _interp(n):
    """Cell-centred linear interpolation from n / 2 to n points, a missing neighbour's weight going to the parent."""
    a = torch.arange(n)
    near = a // 2
    far = near + torch.where(a % 2 == 1, 1, -1)
    ok = (far >= 0) & (far < n // 2)
    rows, cols = torch.cat([a, a[ok]]), torch.cat([near, far[ok]])
    vals = torch.cat([torch.where(ok, 0.75, 1.0).double(), torch.full((int(ok.sum()),), 0.25, dtype=torch.float64)])
    return torch.sparse_coo_tensor(torch.stack([rows, cols]), vals, (n, n // 2)).to_dense().to(DEV)


def _kron(ph, pv):
    """P_h (x) P_v of two sparse-in-fact matrices, as a sparse one."""
    h, v = ph.nonzero(), pv.nonzero()
    r = (h[:, :1] * pv.shape[0] + v[None, :, 0]).reshape(-1)
    c = (h[:, 1:] * pv.shape[1] + v[None, :, 1]).reshape(-1)
    w = (ph[h[:, 0], h[:, 1]][:, None] * pv[v[:, 0], v[:, 1]][None, :]).reshape(-1)
    return torch.sparse_coo_tensor(torch.stack([r, c]), w, (ph.shape[0] * pv.shape[0], ph.shape[1] * pv.shape[1])).coalesce()


def _vcycle64(A, d, lam, r, shape):
    """V(1,1) with l1-Jacobi and an exact coarsest solve on lam^2 L^T D^2 L + diag(A^T A), Galerkin coarse operators."""
    nh, nv = shape
    w = lam * lam * d * d
    q = torch.arange(nh * nv, device=DEV).reshape(shape)
    s, t = torch.cat([q[:, :-1].reshape(-1), q[:-1].reshape(-1)]), torch.cat([q[:, 1:].reshape(-1), q[1:].reshape(-1)])
    f = q.reshape(-1)
    idx = torch.stack([torch.cat([s, t, s, t, f]), torch.cat([t, s, s, t, f])])
    K = torch.sparse_coo_tensor(idx, torch.cat([-w, -w, w, w, A.diag]), (nh * nv, nh * nv)).coalesce()
    levels = []
    while (nv > 16 or nh > 16) and nv % 2 == 0 and nh % 2 == 0:
        P = _kron(_interp(nh), _interp(nv))
        l1 = torch.zeros(nh * nv, dtype=torch.float64, device=DEV).index_add_(0, K.indices()[0], K.values().abs())
        levels.append((K, P, 1 / l1))
        K = torch.sparse.mm(torch.sparse.mm(P.t().coalesce(), K), P).coalesce()
        nv, nh = nv // 2, nh // 2
    K = K.to_dense()

    def cycle(k, r):
        if k == len(levels):
            return torch.linalg.solve(K, r)
        M, P, di = levels[k]
        mul = lambda S, x: torch.sparse.mm(S, x[:, None])[:, 0]  # noqa: E731
        z = di * r
        z = z + mul(P, cycle(k + 1, mul(P.t(), r - mul(M, z))))
        return z + di * (r - mul(M, z))
    return cycle(0, r)


def exact(case, seed):
    A, b, d, v = _inputs(case, seed)
    shape, n = (case["n_h"], case["n_v"]), case["n_v"] * case["n_h"]
    zero = torch.zeros(n, dtype=torch.float64, device=DEV)
    if case["what"] == "operator":
        return torch.stack([_normal(A, d, float(x), v[k], shape) for k, x in enumerate(np.geomspace(0.1, 1.0, case["cols"]))])
    lams = _lambdas(case)
    if case["what"] == "precond":
        return torch.stack([_vcycle64(A, d, float(x), v[k], shape) for k, x in enumerate(lams)])
    if case["what"] == "solve":
        per = [_sweep64(A, d, lams, b[k], zero, shape) for k in range(case["rhs"])]
        return (*(torch.stack([p[q] for p in per]) for q in range(3)), None)
    # Algorithm 2: sweep, corner, weights, a window of ten lambda around the
    # corner; the stop after three equal selections ends a run after the third
    x, lo, hi = zero, 0, len(lams)
    m, hist = len(lams), []
    for ell in range(case["outer"]):
        xs, rho, eta = _sweep64(A, d, lams[lo:hi], b[0], x, shape)
        k = _corner(rho.cpu().numpy(), eta.cpu().numpy())
        x = xs[k]
        hist.append(lo + k + 1)
        if ell + 1 < case["outer"]:
            d = _next_weights(d, x, shape)
            lo, hi = max(min(hist[-1] - 2, m - 9), 1) - 1, min(max(hist[-1] + 7, 10), m)
    return x, None, None, None
