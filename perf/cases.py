"""Performance cases of the BSPAI-GMRES-IR framework: what its users have it do.

Every case is one call sequence through the public entry points
(paper_2307_03914_gb300.bspai, .autograd) on seeded synthetic systems of the
kinds the framework's own workloads use: convection-diffusion on 2D and 3D
grids, random sparse matrices with log-normal entries, diffusion with a
log-normal coefficient field, and batches of small 2D systems.  A case is a
dict of plain values; its kinds are

  apply     y = M x by the adaptive-precision product, M given by the caller
  residual  r = b - A x in u_r ~ u^2
  spai      the fixed-pattern sparse approximate inverse of A
  adaptive  the adaptive (growing-pattern) sparse approximate inverse
  solve     one refinement solve with A, M and the buckets kept by the caller
  step      the whole path on a new matrix: build, bucketing and solve
  batch     many independent systems, several right-hand sides each
  adjoint   a differentiable solve: forward and both gradients

Matrices and right-hand sides are generated on the GPU from the seed.
"""
import math

import numpy as np
import torch

from paper_2307_03914_gb300 import autograd as AG
from paper_2307_03914_gb300 import bspai as B

BUCKETS3 = "fp64,fp32,fp16"
BUCKETS4 = "fp64,fp32,fp16,e4m3"
BUCKETSR = "fp64,fp32,fp16,bf16"
BUCKETSD = "fp32,fp16,drop"


def listed():
    return [
        # the smallest product: the preconditioner of a 32 x 32 problem applied in a
        # caller's own Krylov loop, where the call and one launch are all there is
        dict(name="apply_2d_32", kind="apply", mat="cd2", gx=32, gy=32, gz=1, precs=BUCKETS3, eps=2.0 ** -16,
             io="fp64"),
        # the bucketed product of the 128^3 workload (fp16 + e4m3 buckets), as inside GMRES
        dict(name="apply_3d_128", kind="apply", mat="cd3", gx=128, gy=128, gz=128, precs=BUCKETS4, eps=2.0 ** -10,
             io="fp32"),
        # the compensated residual of the 128^3 workload near the solution
        dict(name="residual_3d_128", kind="residual", mat="cd3", gx=128, gy=128, gz=128),
        # the preconditioner of the 128^3 workload: a new matrix on a known pattern
        dict(name="spai_3d_128", kind="spai", mat="cd3", gx=128, gy=128, gz=128, u_f="fp32"),
        # the growing-pattern build on a ragged 3D grid (spai_eps 0.3, alpha 3, beta 8)
        dict(name="adaptive_3d_63", kind="adaptive", mat="cd3", gx=63, gy=64, gz=65, alpha=3, beta=8),
        # the smallest solve: 32 x 32 convection-diffusion, where launches and waits count
        dict(name="solve_2d_32", kind="solve", mat="cd2", gx=32, gy=32, gz=1, precs=BUCKETS3, eps=2.0 ** -37,
             u_f="fp32", u="fp64", u_r="dd", u_g="fp32", tol=1e-4),
        # a solve wholly in double, the setting users compare the mixed ones with
        dict(name="solve_fp64_3d_64", kind="solve", mat="cd3", gx=64, gy=64, gz=64, precs="fp64", eps=2.0 ** -37,
             u_f="fp32", u="fp64", u_r="dd", u_g="fp64", tol=1e-8),
        # the (half, single, double) setting on a ragged 3D grid, single-precision result
        dict(name="solve_half_3d_95", kind="solve", mat="cd3", gx=95, gy=96, gz=97, precs=BUCKETSD, eps=2.0 ** -18,
             u_f="fp16", u="fp32", u_r="fp64", u_g="fp32", tol=1e-4),
        # the random workload from its CSR on: wide SPAI blocks, irregular gathers
        dict(name="step_random_65536", kind="step", mat="rnd", gx=65536, gy=1, gz=1, precs=BUCKETSR, eps=2.0 ** -37),
        # the 128^3 workload from its CSR on: the framework's headline step
        dict(name="step_3d_128", kind="step", mat="cd3", gx=128, gy=128, gz=128, precs=BUCKETS4, eps=2.0 ** -10),
        # a batch of small and mid-size systems, several right-hand sides each
        dict(name="batch_96x4", kind="batch", nsys=96, nrhs=4, nmin=1000, nmax=16000, sizes=7),
        # a differentiable solve with eight right-hand sides (forward and backward)
        dict(name="adjoint_96x8", kind="adjoint", gx=96, nrhs=8),
    ]


def draw(rng):
    def log_int(a, b):
        return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))

    def grid3(a, b):
        g = log_int(a, b)
        return dict(mat="cd3", gx=g, gy=max(2, g + rng.randint(-2, 2)), gz=max(2, g + rng.randint(-2, 2)))

    def grid2(a, b):
        g = log_int(a, b)
        return dict(mat="cd2", gx=g, gy=max(2, g + rng.randint(-3, 3)), gz=1)

    kind = rng.choice(["apply", "residual", "spai", "adaptive", "solve", "solve", "solve", "step", "batch", "adjoint"])
    if kind == "apply":
        precs, eps = rng.choice([(BUCKETS3, 2.0 ** -16), (BUCKETS4, 2.0 ** -10), (BUCKETSR, 2.0 ** -16), ("fp32", 2.0 ** -16)])
        return dict(kind=kind, **(grid3(12, 126) if rng.random() < 0.7 else grid2(32, 1000)), precs=precs, eps=eps,
                    io=rng.choice(["fp64", "fp32"]))
    if kind == "residual":
        return dict(kind=kind, **(grid3(12, 126) if rng.random() < 0.7 else grid2(32, 1000)))
    if kind == "spai":
        g = grid3(12, 126) if rng.random() < 0.7 else dict(mat="rnd", gx=log_int(1000, 30000), gy=1, gz=1)
        return dict(kind=kind, **g, u_f="fp32")
    if kind == "adaptive":
        return dict(kind=kind, **grid3(10, 62), alpha=rng.choice([1, 2, 3]), beta=8)
    if kind == "solve":
        g = rng.choice([grid3(10, 110), grid2(24, 400), dict(mat="rnd", gx=log_int(1000, 30000), gy=1, gz=1)])
        mode = rng.choice(["mixed", "mixed", "mixed", "double", "single"])
        base = dict(kind=kind, **g)
        if mode == "double":
            return dict(base, precs="fp64", eps=2.0 ** -37, u_f="fp32", u="fp64", u_r="dd", u_g="fp64", tol=1e-8)
        if mode == "single":
            return dict(base, precs=BUCKETSD, eps=2.0 ** -18, u_f="fp32", u="fp32", u_r="fp64", u_g="fp32", tol=1e-4)
        precs, eps = rng.choice([(BUCKETS3, 2.0 ** -16), (BUCKETS3, 2.0 ** -37), ("fp32", 2.0 ** -16)])
        return dict(base, precs=precs, eps=eps, u_f="fp32", u="fp64", u_r="dd", u_g="fp32", tol=1e-4)
    if kind == "step":
        if rng.random() < 0.3:
            return dict(kind=kind, mat="rnd", gx=log_int(1000, 60000), gy=1, gz=1, precs=BUCKETSR, eps=2.0 ** -37)
        return dict(kind=kind, **grid3(12, 126), precs=BUCKETS4, eps=2.0 ** -10)
    if kind == "batch":
        return dict(kind=kind, nsys=log_int(4, 96), nrhs=rng.choice([1, 2, 3, 4]), nmin=1000,
                    nmax=log_int(2000, 16000), sizes=rng.randint(0, 999))
    return dict(kind=kind, gx=log_int(16, 96), nrhs=rng.choice([1, 2, 4, 8]))


# ------------------------------------------------------------------ matrices
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) & 0x7FFFFFFF)


def _unit(seed):
    return float(np.random.default_rng(int(seed) & 0x7FFFFFFF).uniform(-1.0, 1.0))


class _Table:
    """A sparse matrix as an (n, w) table: columns ascending, -1 for an absent entry."""

    def __init__(self, cols, vals):
        self.cols, self.vals, self.n, self.w = cols, vals, cols.shape[0], cols.shape[1]

    def csr(self):
        mask = self.cols >= 0
        row_ptr = torch.zeros(self.n + 1, dtype=torch.int32, device="cuda")
        row_ptr[1:] = torch.cumsum(mask.sum(dim=1), 0).to(torch.int32)
        return B.DeviceCSR(self.n, row_ptr, self.cols[mask].to(torch.int32), self.vals[mask])

    def pattern(self):
        c = self.csr()
        return B.DeviceCSR(c.n, c.row_ptr, c.col)

    def mul(self, x):
        y = torch.zeros_like(x)
        for t in range(self.w):
            c = self.cols[:, t]
            y += torch.where(c >= 0, self.vals[:, t] * x[..., c.clamp(min=0)], torch.zeros((), dtype=x.dtype, device="cuda"))
        return y


def _stencil(n, entries):
    """entries: (column offset, mask of the rows that have it, value), ascending offsets."""
    r = torch.arange(n, device="cuda")
    absent = torch.full((), -1, device="cuda", dtype=torch.int64)
    cols = torch.stack([torch.where(m, r + o, absent) for o, m, _ in entries], dim=1)
    vals = torch.stack([torch.where(m, torch.full((), 1.0, dtype=torch.float64, device="cuda") * v, torch.zeros((), dtype=torch.float64, device="cuda"))
                        for _, m, v in entries], dim=1)
    return _Table(cols, vals)


def _convdiff3d(gx, gy, gz, peclet, eps=(1.0, 10.0, 100.0)):
    n = gx * gy * gz
    r = torch.arange(n, device="cuda")
    ix, iy, iz = r % gx, (r // gx) % gy, r // (gx * gy)
    ex, ey, ez = eps
    lo, hi, every = 1.0 + peclet, 1.0 - peclet, r >= 0
    return _stencil(n, [(-gx * gy, iz > 0, -ez * lo), (-gx, iy > 0, -ey * lo), (-1, ix > 0, -ex * lo),
                        (0, every, 2.0 * (ex + ey + ez)), (1, ix < gx - 1, -ex * hi), (gx, iy < gy - 1, -ey * hi),
                        (gx * gy, iz < gz - 1, -ez * hi)])


def _convdiff2d(gx, gy, px, py):
    n = gx * gy
    r = torch.arange(n, device="cuda")
    ix, iy = r % gx, r // gx
    return _stencil(n, [(-gx, iy > 0, -(1.0 + py)), (-1, ix > 0, -(1.0 + px)), (0, r >= 0, 4.0),
                        (1, ix < gx - 1, -(1.0 - px)), (gx, iy < gy - 1, -(1.0 - py))])


def _convdiff2d_9pt(g, px, py):
    n = g * g
    r = torch.arange(n, device="cuda")
    ix, iy = r % g, r // g
    edge = {(-1, 0): -(1.0 + px), (1, 0): -(1.0 - px), (0, -1): -(1.0 + py), (0, 1): -(1.0 - py), (0, 0): 8.0}
    out = []
    for dy in (-1, 0, 1):
        for dx in (-1, 0, 1):
            m = (ix + dx >= 0) & (ix + dx < g) & (iy + dy >= 0) & (iy + dy < g)
            out.append((dx + g * dy, m, edge.get((dx, dy), -1.0)))
    return _stencil(n, out)


def _random(n, seed, k=16, sigma=2.0, delta=-0.35):
    """k distinct off-diagonal columns per row, values sign * exp(N(0, sigma)), the
    diagonal (1 + delta) times the row's absolute sum."""
    g = _gen(seed)
    cols = torch.randint(0, n - 1, (n, k), generator=g, device="cuda")
    while True:
        cols = cols.sort(dim=1).values
        bad = (cols[:, 1:] == cols[:, :-1]).any(dim=1).nonzero()[:, 0]
        if bad.numel() == 0:
            break
        cols[bad] = torch.randint(0, n - 1, (bad.numel(), k), generator=g, device="cuda")
    rows = torch.arange(n, device="cuda")[:, None]
    cols = torch.where(cols >= rows, cols + 1, cols)
    mag = torch.exp(sigma * torch.randn((n, k), generator=g, device="cuda", dtype=torch.float64))
    off = torch.where(torch.rand((n, k), generator=g, device="cuda") < 0.5, -mag, mag)
    allc = torch.cat([cols, rows], dim=1)
    allv = torch.cat([off, (1.0 + delta) * mag.sum(dim=1, keepdim=True)], dim=1)
    allc, order = allc.sort(dim=1)
    return _Table(allc, allv.gather(1, order))


def _pattern_power(A, keep=24):
    """Pattern of |A||A| thinned to the `keep` largest entries of each row, the diagonal always kept."""
    rows = torch.arange(A.n, device="cuda")[:, None]
    cc = A.cols[A.cols].reshape(A.n, -1)
    vv = (A.vals.abs()[:, :, None] * A.vals.abs()[A.cols]).reshape(A.n, -1)
    cc, order = cc.sort(dim=1, stable=True)
    cum = torch.cumsum(vv.gather(1, order), dim=1)
    last = torch.ones_like(cc, dtype=torch.bool)
    last[:, :-1] = cc[:, 1:] != cc[:, :-1]
    # a run's sum: the running sum at its last entry less that at the run before
    at = torch.where(last, cum, torch.zeros((), dtype=cum.dtype, device="cuda")).cummax(dim=1).values
    before = torch.zeros_like(cum)
    before[:, 1:] = at[:, :-1]
    total = torch.where(last, cum - before, torch.full((), -1.0, dtype=cum.dtype, device="cuda"))
    total = torch.where(last & (cc == rows), torch.full((), math.inf, dtype=cum.dtype, device="cuda"), total)
    top = total.topk(min(keep, total.shape[1]), dim=1).indices
    cols = cc.gather(1, top)
    return _Table(cols.sort(dim=1).values, torch.zeros(cols.shape, dtype=torch.float64, device="cuda"))


def _in_units(A, seed):
    """The rows of A in other units (powers of two): the column scaling of the build takes
    them out again, so the pattern that grows, and with it the result's shape, is the same."""
    exps = torch.randint(-3, 4, (A.n,), generator=_gen(seed), device="cuda")
    rows = torch.repeat_interleave(torch.arange(A.n, device="cuda"), A.row_ptr.diff())
    return B.DeviceCSR(A.n, A.row_ptr, A.col, torch.ldexp(A.val, exps[rows]))


def _matrix(case, seed):
    """(A, its pattern of M) of a case; the coefficients move a little with the seed
    (not where they decide the shape of what comes back)."""
    u = _unit(seed) if case["kind"] != "adaptive" else 0.0
    if case["mat"] == "cd3":
        A = _convdiff3d(case["gx"], case["gy"], case["gz"], 0.8 + 0.02 * u)
        return A, A
    if case["mat"] == "cd2":
        A = _convdiff2d(case["gx"], case["gy"], 0.5 + 0.02 * u, 0.5 - 0.02 * u)
        return A, A
    A = _random(case["gx"], seed)
    return A, _pattern_power(A)


def _uniform(shape, seed):
    return 2.0 * torch.rand(shape, generator=_gen(seed + 77), device="cuda", dtype=torch.float64) - 1.0


def _neumann(A):
    """A sparse approximate inverse on A's own pattern: D^-1 (2 I - A D^-1)."""
    r = torch.arange(A.n, device="cuda")[:, None]
    diag = torch.where(A.cols == r, A.vals, torch.zeros((), dtype=torch.float64, device="cuda")).sum(dim=1)
    at = diag[A.cols.clamp(min=0)]
    one = (A.cols == r).to(torch.float64)
    return _Table(A.cols, (2.0 * one - A.vals / at) / diag[:, None])


def _lognormal(g, seed, corr=8.0):
    """exp of a unit Gaussian field with squared-exponential correlation of `corr` cells."""
    w = torch.randn((g, g), generator=_gen(seed + 7), device="cuda", dtype=torch.float64)
    k = torch.fft.fftfreq(g, dtype=torch.float64, device="cuda")
    k2 = k[:, None] ** 2 + k[None, :] ** 2
    f = torch.fft.ifft2(torch.fft.fft2(w) * torch.exp(-(2 * math.pi) ** 2 * k2 * corr ** 2 / 4.0)).real
    return torch.exp((f - f.mean()) / f.std())


def _diffusion2d(g, seed):
    """-div(kappa grad u), 5-point finite volumes with harmonic face coefficients (symmetric)."""
    kap = _lognormal(g, seed).reshape(-1)
    n = g * g
    r = torch.arange(n, device="cuda")
    ix, iy = r % g, r // g
    diag = torch.zeros(n, dtype=torch.float64, device="cuda")
    face = {}
    for o, m in ((-g, iy > 0), (-1, ix > 0), (1, ix < g - 1), (g, iy < g - 1)):
        other = kap[torch.where(m, r + o, r)]
        t = torch.where(m, 2.0 * kap * other / (kap + other), 2.0 * kap)
        diag = diag + t
        face[o] = (m, -t)
    return _stencil(n, [(-g, *face[-g]), (-1, *face[-1]), (0, r >= 0, diag), (1, *face[1]), (g, *face[g])])


def _batch(case, seed):
    """The systems' tables; their orders and stencils belong to the case, the coefficients to the seed."""
    shape = np.random.default_rng(case["sizes"])
    values = np.random.default_rng(int(seed) & 0x7FFFFFFF)
    out = []
    for _ in range(case["nsys"]):
        g = int(round(math.sqrt(math.exp(shape.uniform(math.log(case["nmin"]), math.log(case["nmax"]))))))
        five, (px, py) = shape.random() < 0.5, values.uniform(0.1, 1.0, 2)
        out.append(_convdiff2d(g, g, px, py) if five else _convdiff2d_9pt(g, px, py))
    return out


def _stack(mats, align=32):
    """Block-diagonal CSR, every system padded with empty rows to a multiple of `align`."""
    off = [0]
    for m in mats:
        off.append(off[-1] + -(-m.n // align) * align)
    lens = torch.zeros(off[-1], dtype=torch.int64, device="cuda")
    cols, vals = [], []
    for m, o in zip(mats, off):
        mask = m.cols >= 0
        lens[o:o + m.n] = mask.sum(dim=1)
        cols.append((m.cols[mask] + o).to(torch.int32))
        vals.append(m.vals[mask])
    row_ptr = torch.zeros(off[-1] + 1, dtype=torch.int32, device="cuda")
    row_ptr[1:] = torch.cumsum(lens, 0).to(torch.int32)
    return B.DeviceCSR(off[-1], row_ptr, torch.cat(cols), torch.cat(vals)), off


def _batch_x(mats, off, nrhs, seed):
    X = torch.zeros((nrhs, off[-1]), dtype=torch.float64, device="cuda")
    for s, (m, o) in enumerate(zip(mats, off)):
        X[:, o:o + m.n] = _uniform((nrhs, m.n), seed + 1000 * s)
    return X


# ------------------------------------------------------------------ the calls
def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        mats = _batch(case, seed)
        A, off = _stack(mats)
        P = B.DeviceCSR(A.n, A.row_ptr, A.col)
        X = _batch_x(mats, off, case["nrhs"], seed)
        b = torch.zeros_like(X)
        for m, o in zip(mats, off):
            b[:, o:o + m.n] = m.mul(X[:, o:o + m.n])
        row_off = torch.tensor(off, dtype=torch.int32, device="cuda")
        M, _ = B.bspai_build(A, P, 0.3)
        BM, _ = B.bspai_bucket_batched(M, row_off, 2.0 ** -16, BUCKETS3.split(","))
        return dict(kind=kind, Ah=B.matrix_create(A), M=M, BM=BM, row_off=row_off, nrhs=case["nrhs"],
                    b=b.reshape(-1), x=torch.zeros_like(b).reshape(-1))
    if kind == "adjoint":
        T = _diffusion2d(case["gx"], seed)
        A = T.csr()
        x = _uniform((case["nrhs"], A.n), seed)
        return dict(kind=kind, a=A.val.clone().requires_grad_(True), b=T.mul(x).requires_grad_(True),
                    row_ptr=A.row_ptr, col=A.col, pattern=B.DeviceCSR(A.n, A.row_ptr, A.col),
                    target=_uniform(tuple(x.shape), seed + 1))
    T, Pt = _matrix(case, seed)
    if kind == "apply":
        Mt = _neumann(T).csr()
        M = B.M_create(Mt)
        BM, _ = B.bspai_bucket(M, case["eps"], case["precs"].split(","))
        dt = torch.float64 if case["io"] == "fp64" else torch.float32
        x = _uniform(T.n, seed).to(dt)
        return dict(kind=kind, BM=BM, x=x, y=torch.empty_like(x))
    A = T.csr()
    x = _uniform(T.n, seed)
    if kind == "residual":
        b = T.mul(x)
        return dict(kind=kind, Ah=B.matrix_create(A), b=b, x=x * (1.0 + 1e-5 * _uniform(T.n, seed + 1)),
                    r=torch.empty_like(b))
    if kind == "spai":
        return dict(kind=kind, A=A, P=Pt.pattern(), u_f=case["u_f"])
    if kind == "adaptive":
        return dict(kind=kind, A=_in_units(A, seed), alpha=case["alpha"], beta=case["beta"])
    b = T.mul(x)
    out = torch.zeros_like(b)
    if kind == "step":
        return dict(kind=kind, A=A, P=Pt.pattern(), b=b, x=out, precs=case["precs"].split(","), eps=case["eps"])
    M, _ = B.bspai_build(A, Pt.pattern(), 0.3, u_f=case["u_f"])
    BM, _ = B.bspai_bucket(M, case["eps"], case["precs"].split(","))
    return dict(kind=kind, Ah=B.matrix_create(A), M=M, BM=BM, b=b, x=out, u=case["u"], u_r=case["u_r"],
                u_g=case["u_g"], tol=case["tol"])


def run(s):
    kind = s["kind"]
    if kind == "apply":
        return B.apply(s["BM"], s["x"], s["y"])
    if kind == "residual":
        return B.residual(s["Ah"], s["x"], s["b"], s["r"])
    if kind == "spai":
        M, info = B.bspai_build(s["A"], s["P"], 0.3, u_f=s["u_f"])
        _, _, val, resid = B.M_export(M, s["P"].n, s["P"].nnz)
        return dict(val=val, resid=resid)
    if kind == "adaptive":
        M, info = B.bspai_build_adaptive(s["A"], 0.3, s["alpha"], s["beta"])
        row_ptr, col, val, resid = B.M_export(M, s["A"].n, int(info["nnz"]))
        return dict(row_ptr=row_ptr, col=col, val=val, resid=resid)
    if kind == "solve":
        B.gmres_ir_solve(s["Ah"], s["b"], s["BM"], s["M"], s["x"], u=s["u"], u_r=s["u_r"], u_g=s["u_g"], u_p=s["u_g"],
                         tol=s["tol"])
        # a single-precision solve leaves single-precision values in its double buffer
        return s["x"].float() if s["u"] == "fp32" else s["x"]
    if kind == "step":
        M, _ = B.bspai_build(s["A"], s["P"], 0.3)
        BM, _ = B.bspai_bucket(M, s["eps"], s["precs"])
        B.gmres_ir_solve(s["A"], s["b"], BM, M, s["x"], tol=1e-4)
        return s["x"]
    if kind == "batch":
        B.gmres_ir_solve_batched(s["Ah"], s["row_off"], s["nrhs"], s["b"], s["BM"], s["M"], s["x"], tol=1e-4)
        return s["x"]
    x = AG.solve(s["a"], s["b"], s["row_ptr"], s["col"], s["pattern"])
    da, db = torch.autograd.grad((x - s["target"]).square().sum(), (s["a"], s["b"]))
    return dict(x=x.detach(), da=da, db=db)


# ------------------------------------------------------------------ the work
def _entries(case):
    """(rows, entries of A, entries of M) of a single-system case."""
    n = case["gx"] * case["gy"] * case["gz"]
    if case["mat"] == "rnd":
        return n, 17 * n, 24 * n
    nnz = 7 * n - 2 * (case["gx"] * case["gy"] + case["gy"] * case["gz"] + case["gx"] * case["gz"]) \
        if case["mat"] == "cd3" else 5 * n - 2 * (case["gx"] + case["gy"])
    return n, nnz, nnz


def work(case):
    """Each input read once and each output written once (CSR with 4-byte columns, a
    bucketed M as it is stored);
    operations: of one product per matrix for the products, of the least-squares
    solves for the builds, and for the solves of the Arnoldi steps that systems of
    their kind take (two products and the orthogonalisation of each step)."""
    kind = case["kind"]
    if kind == "batch":
        n = sum(m * m for m in _batch_orders(case))
        nnz, rhs = 7 * n, case["nrhs"]
        steps = 200
        return dict(bytes=12 * nnz + 4 * nnz + 4 * nnz + 16 * n * rhs, flops=rhs * steps * (4 * nnz + 2 * 50 * 2 * n))
    if kind == "adjoint":
        n, rhs = case["gx"] ** 2, case["nrhs"]
        nnz = 5 * n
        return dict(bytes=12 * nnz + 4 * nnz + 32 * n * rhs + 8 * nnz, flops=rhs * 1200 * (4 * nnz + 2 * 150 * 2 * n))
    n, na, nm = _entries(case)
    if kind == "apply":
        size = dict(fp64=8, fp32=4)[case["io"]]
        # 16-bit entries and column differences, as the mixes that are used come to on average
        return dict(bytes=nm * (2 + 2) + 2 * size * n, flops=2 * nm)
    if kind == "residual":
        return dict(bytes=na * 12 + 24 * n, flops=2 * na)
    rows = na / n
    cols = nm / n
    spai = nm * (2 * cols * rows * cols * 0.6 + 4 * rows)
    if kind == "spai":
        return dict(bytes=na * 12 + nm * 4 + 4 * nm + 4 * n, flops=spai)
    if kind == "adaptive":
        return dict(bytes=na * 12 + 8 * nm + 4 * n, flops=case["alpha"] * spai)
    steps = 120 if case["mat"] == "rnd" else 300
    krylov = steps * (2 * na + 2 * nm + 2 * (steps // 8) * 2 * n)
    both = na * 12 + nm * 4 + 16 * n
    return dict(bytes=both + (nm * 4 if kind == "step" else 0), flops=krylov + (spai if kind == "step" else 0))


def _batch_orders(case):
    shape = np.random.default_rng(case["sizes"])
    out = []
    for _ in range(case["nsys"]):
        out.append(int(round(math.sqrt(math.exp(shape.uniform(math.log(case["nmin"]), math.log(case["nmax"])))))))
        shape.random()
    return out


# ------------------------------------------------------------------ 64-bit values
def _exact_spai(A, P, chunk):
    """Rows of M = M'^T D in 64 bits: for every k the least-squares solution of
    B(:, J_k) m = e_k on B = A^T D (D: the reciprocal of each row's largest entry of
    A), by Gram-Schmidt applied twice; and its residual norm."""
    d = 1.0 / A.vals.abs().max(dim=1).values
    vals, resid = [], []
    for k0 in range(0, A.n, chunk):
        J = P.cols[k0:k0 + chunk]
        m, w = J.shape
        have = J >= 0
        rows = A.cols[J.clamp(min=0)]                         # row indices of B's column j: the columns of row j of A
        rows = torch.where(have[:, :, None], rows, torch.full((), -1, device="cuda"))
        entry = torch.where(rows >= 0, A.vals[J.clamp(min=0)] * d[J.clamp(min=0)][:, :, None],
                            torch.zeros((), dtype=torch.float64, device="cuda"))
        flat = rows.reshape(m, -1)
        srt, order = flat.sort(dim=1, stable=True)
        new = torch.ones_like(srt, dtype=torch.int64)
        new[:, 1:] = (srt[:, 1:] != srt[:, :-1]).to(torch.int64)
        rank_sorted = torch.cumsum(new, dim=1) - 1
        rank = torch.empty_like(rank_sorted).scatter_(1, order, rank_sorted).reshape(m, w, -1)
        height = int(rank.max()) + 1
        Q = torch.zeros((m, w, height), dtype=torch.float64, device="cuda").scatter_(2, rank, entry)
        Ab = Q.clone()
        k = torch.arange(k0, k0 + m, device="cuda")[:, None]
        e = torch.zeros((m, height), dtype=torch.float64, device="cuda")
        hit = (srt == k).to(torch.float64)
        e = e.scatter_reduce(1, rank_sorted, hit, "amax")
        R = torch.zeros((m, w, w), dtype=torch.float64, device="cuda")
        y = torch.zeros((m, w), dtype=torch.float64, device="cuda")
        res = e.clone()
        for j in range(w):
            q = Q[:, j]
            for _ in range(2):
                if j:
                    c = torch.einsum("mih,mh->mi", Q[:, :j], q)
                    q = q - torch.einsum("mi,mih->mh", c, Q[:, :j])
                    R[:, :j, j] += c
            norm = q.norm(dim=1)
            R[:, j, j] = torch.where(norm > 0, norm, torch.ones((), dtype=torch.float64, device="cuda"))
            Q[:, j] = q / R[:, j, j][:, None]
            y[:, j] = (Q[:, j] * res).sum(dim=1)
            res = res - y[:, j][:, None] * Q[:, j]
        mk = torch.linalg.solve_triangular(R, y[:, :, None], upper=True)[:, :, 0]
        s = torch.einsum("mw,mwh->mh", mk, Ab) - e
        vals.append((mk * d[J.clamp(min=0)])[have])
        resid.append(s.norm(dim=1))
    return torch.cat(vals), torch.cat(resid)


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        mats = _batch(case, seed)
        off = [0]
        for m in mats:
            off.append(off[-1] + -(-m.n // 32) * 32)
        return _batch_x(mats, off, case["nrhs"], seed).reshape(-1)  # b = A x
    if kind == "adjoint":
        T = _diffusion2d(case["gx"], seed)
        x = _uniform((case["nrhs"], T.n), seed)
        g = 2.0 * (x - _uniform(tuple(x.shape), seed + 1))
        dense = torch.zeros((T.n, T.n), dtype=torch.float64, device="cuda")
        r = torch.arange(T.n, device="cuda")[:, None].expand_as(T.cols)
        mask = T.cols >= 0
        dense[r[mask], T.cols[mask]] = T.vals[mask]
        lam = torch.linalg.solve(dense.T, g.T).T
        da = torch.zeros_like(T.vals)
        for q in range(case["nrhs"]):
            da -= lam[q][:, None] * x[q][T.cols.clamp(min=0)]
        return dict(x=x, da=da[mask], db=lam)
    if kind == "adaptive":
        return None  # the pattern itself is chosen by the computation
    T, Pt = _matrix(case, seed)
    if kind == "apply":
        Mt = _neumann(T)
        Mt.vals = Mt.vals.float().double()
        return Mt.mul(_uniform(T.n, seed).to(torch.float64 if case["io"] == "fp64" else torch.float32).double())
    x = _uniform(T.n, seed)
    if kind == "residual":
        # b - A x_near with b = fl(A x): the products' differences are formed before they are added
        near = x * (1.0 + 1e-5 * _uniform(T.n, seed + 1))
        b = T.mul(x)
        r = b.clone()
        for t in range(T.w):
            c = T.cols[:, t]
            r -= torch.where(c >= 0, T.vals[:, t] * near[c.clamp(min=0)], torch.zeros((), dtype=torch.float64, device="cuda"))
        return r
    if kind == "spai":
        val, resid = _exact_spai(T, Pt, 1024 if case["mat"] == "rnd" else 131072)
        return dict(val=val, resid=resid)
    return x  # solves: b = A x
