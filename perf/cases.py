"""The work that users of this library have it do, as measurable cases.

Every case goes through the public Python entry points (``Matrix``, ``Split``, ``Batch``,
``spmv``, ``cg``, ``ir_cg``).  Matrices have the shapes of the library's own workloads: 2D
5-point and 3D 7-point Laplacians, the 27-point pattern with free values, and the symmetric
Hamiltonian-like pattern (half of a row's entries within 64 columns of the diagonal, half
anywhere).  They are drawn here with torch on the GPU, so that inputs are made quickly.

``listed()`` gives the fixed cases, ``draw(rng)`` one more of the same ranges, ``prepare``
what a program holds before the call, ``run`` one pass, ``work`` the bytes and operations a
pass cannot do without, and ``exact`` the same results in 64-bit torch without the library.
"""
from __future__ import annotations

import math
import random

import torch

from paper_1106_5908_gb300.torch_api import Batch, Matrix, cg, ir_cg, spmv

_DEV = "cuda"
_DT = {"f64": torch.float64, "f32": torch.float32}


# --------------------------------------------------------------------------------------
# The cases
# --------------------------------------------------------------------------------------

def listed():
    return [
        # A small 2D Poisson operator: one product is a few microseconds, so the call itself
        # and its launch are what a time stepper or a small Krylov solver waits for.
        dict(name="apply-lap2d-256", kind="apply", pattern="lap2d", n=256, dtype="f64", alpha=1.0, beta=0.0),
        # The paper's workload: the plain product of a large scattered symmetric matrix.
        dict(name="apply-ham-4m", kind="apply", pattern="ham", n=4_194_304, dtype="f64", alpha=1.0, beta=0.0),
        # The same product with FP32-stored values and vectors.
        dict(name="apply-ham-4m-f32", kind="apply", pattern="ham", n=4_194_304, dtype="f32", alpha=1.0, beta=0.0),
        # The paper's local/nonlocal split over 8 row blocks, the halo gathered on a second stream.
        dict(name="split-ham-1m", kind="split", pattern="ham", n=1_048_576, blocks=8),
        # Block vectors on a scattered matrix: block Krylov and Chebyshev methods.
        dict(name="spmm16-ham-2m", kind="spmm", pattern="ham", n=2_097_152, nrhs=16),
        # An odd number of right-hand sides on a stencil-like matrix of odd size.
        dict(name="spmm5-sten27-101", kind="spmm", pattern="stencil27", n=101, nrhs=5),
        # A training step over the matrix values: new values, forward, both gradients.
        dict(name="train-sten27-128", kind="train", pattern="stencil27", n=128, dtype="f64"),
        # Reverse passes on values that stay: an adjoint solver with FP32 storage.
        dict(name="grad-sten27-96-f32", kind="grad", pattern="stencil27", n=96, dtype="f32"),
        # Many uneven matrices applied together: half 5-point grids, half scattered.
        dict(name="batch-64", kind="batch", count=64, lo=1000, hi=200_000, dtype="f64"),
        # FP64 CG on a small grid: latency of the iteration.
        dict(name="cg-lap2d-256", kind="cg", pattern="lap2d", n=256, tol=1e-12),
        # The mixed-precision solver on a 3D Poisson problem, to its default 1e-12.
        dict(name="ircg-poisson7-128", kind="ir_cg", pattern="poisson7", n=128, tol=1e-12),
        # A symmetric matrix given by its upper triangle.
        dict(name="sym-ham-1m", kind="sym", pattern="ham", n=1_048_576, dtype="f64"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


# grid edges or orders of each pattern: from calls of a few microseconds to the largest listed
_RANGE = {"lap2d": (60, 2000), "poisson7": (16, 160), "stencil27": (12, 128), "ham": (3_000, 4_194_304)}


def draw(rng):
    kind = rng.choice(["apply", "apply", "apply", "split", "spmm", "spmm", "train", "grad", "batch", "cg", "ir_cg",
                       "sym"])
    pattern = rng.choice(["lap2d", "poisson7", "stencil27", "ham"])
    lo, hi = _RANGE[pattern]
    dtype = rng.choice(["f64", "f64", "f32"])
    if kind == "apply":
        alpha, beta = rng.choice([(1.0, 0.0), (1.0, 0.0), (-0.75, 0.5)])
        return dict(kind=kind, pattern=pattern, n=_log_int(rng, lo, hi), dtype=dtype, alpha=alpha, beta=beta)
    if kind == "split":
        return dict(kind=kind, pattern="ham", n=_log_int(rng, 20_000, 1_048_576), blocks=rng.choice([2, 4, 8]))
    if kind == "spmm":
        nrhs = _log_int(rng, 2, 32)
        # at most the work of the largest listed block product
        top = {"ham": 2_097_152 * 16 // nrhs, "lap2d": 1400, "poisson7": 112, "stencil27": 72}[pattern]
        return dict(kind=kind, pattern=pattern, n=_log_int(rng, lo, max(2 * lo, min(hi, top))), nrhs=nrhs)
    if kind in ("train", "grad"):
        top = {"lap2d": 2000, "poisson7": 160, "stencil27": 112, "ham": 1_500_000}[pattern]
        return dict(kind=kind, pattern=pattern, n=_log_int(rng, lo, top), dtype=dtype)
    if kind == "batch":
        return dict(kind=kind, count=rng.randint(5, 64), lo=1000, hi=_log_int(rng, 5_000, 200_000), dtype=dtype)
    if kind == "cg":
        pattern = rng.choice(["lap2d", "poisson7"])
        return dict(kind=kind, pattern=pattern, n=_log_int(rng, 40 if pattern == "lap2d" else 16,
                                                           300 if pattern == "lap2d" else 96), tol=1e-12)
    if kind == "ir_cg":
        return dict(kind=kind, pattern="poisson7", n=_log_int(rng, 24, 128), tol=1e-12)
    return dict(kind=kind, pattern="ham", n=_log_int(rng, 5_000, 1_048_576), dtype=dtype)


# --------------------------------------------------------------------------------------
# Matrices and vectors: sizes and patterns by the case, values and vectors by the seed
# --------------------------------------------------------------------------------------

def _gen(seed):
    return torch.Generator(device=_DEV).manual_seed(seed)


def _uniform(g, *shape):
    return torch.rand(*shape, dtype=torch.float64, device=_DEV, generator=g) * 2.0 - 1.0


def _normal(g, *shape):
    return torch.randn(*shape, dtype=torch.float64, device=_DEV, generator=g)


def _stencil(dims, n, offsets):
    """CRS pattern of a truncated stencil on an n^dims grid, first axis fastest."""
    size = n ** dims
    idx = torch.arange(size, device=_DEV, dtype=torch.int32)
    coord = [idx // n ** d % n for d in range(dims)]
    ok = torch.empty(size, len(offsets), dtype=torch.bool, device=_DEV)
    col = torch.empty(size, len(offsets), dtype=torch.int32, device=_DEV)
    for m, off in enumerate(offsets):
        inside = torch.ones(size, dtype=torch.bool, device=_DEV)
        for d in range(dims):
            c = coord[d] + off[d]
            inside &= (c >= 0) & (c < n)
        ok[:, m] = inside
        col[:, m] = idx + sum(off[d] * n ** d for d in range(dims))
    return _row_ptr(ok.sum(1)), col[ok]


def _row_ptr(counts):
    rp = torch.zeros(counts.numel() + 1, dtype=torch.int32, device=_DEV)
    rp[1:] = counts.cumsum(0)
    return rp


def _hamiltonian_upper(n):
    """Sorted distinct (row, column) keys of the strictly upper triangle.  The pattern of an order
    is always the same one (as a program's grid or lattice is): a seed draws its values."""
    g = _gen(2201 + n)
    i = torch.arange(n, device=_DEV)
    length = torch.poisson(torch.full((n,), 6.0, device=_DEV), generator=g).clamp_(2, 16).long()
    near = (length + 1) // 2
    keys = []
    for m in range(8):
        at = i[near > m]
        keys.append(at * n + at + torch.randint(1, 65, (at.numel(),), device=_DEV, generator=g))
        at = i[(length - near > m) & (i + 65 < n)]
        far = (torch.rand(at.numel(), dtype=torch.float64, device=_DEV, generator=g) * (n - at - 65)).long()
        keys.append(at * n + at + 65 + torch.minimum(far, n - at - 66))
    keys = torch.cat(keys)
    # a near column past the last one falls into the next row: drop it
    row = keys // n
    reach = torch.cat([(i[near > m] if f == 0 else i[(length - near > m) & (i + 65 < n)])
                       for m in range(8) for f in (0, 1)])
    return torch.unique(keys[row == reach])


def _hamiltonian(g, n, upper_only=False):
    keys = _hamiltonian_upper(n)
    i = torch.arange(n, device=_DEV)
    v, diag = _normal(g, keys.numel()), _normal(g, n)
    parts, vals = [keys, i * n + i], [v, diag]
    if not upper_only:
        parts.append((keys % n) * n + keys // n)
        vals.append(v)
    keys, order = torch.sort(torch.cat(parts))
    val = torch.cat(vals)[order]
    row = keys // n
    return _row_ptr(torch.bincount(row, minlength=n)), (keys - row * n).to(torch.int32), val


_CROSS2 = [(0, -1), (-1, 0), (0, 0), (1, 0), (0, 1)]
_CROSS3 = [(0, 0, -1), (0, -1, 0), (-1, 0, 0), (0, 0, 0), (1, 0, 0), (0, 1, 0), (0, 0, 1)]
_CUBE3 = [(a, b, c) for c in (-1, 0, 1) for b in (-1, 0, 1) for a in (-1, 0, 1)]


def _matrix(pattern, n, g, upper_only=False):
    """(row_ptr, col, val FP64, order) on the GPU."""
    if pattern == "ham":
        rp, col, val = _hamiltonian(g, n, upper_only)
        return rp, col, val, n
    dims, offsets = {"lap2d": (2, _CROSS2), "poisson7": (3, _CROSS3), "stencil27": (3, _CUBE3)}[pattern]
    rp, col = _stencil(dims, n, offsets)
    if pattern == "stencil27":
        return rp, col, _normal(g, col.numel()), n ** dims
    val = torch.where(col == _rows(rp, col), 2.0 * dims, -1.0).double()
    return rp, col, val, n ** dims


def _rows(rp, col):
    return torch.repeat_interleave(torch.arange(rp.numel() - 1, device=_DEV), (rp[1:] - rp[:-1]).long(),
                                   output_size=col.numel())


def _members(case, g):
    """The batch's matrices: even ones 5-point grids, odd ones scattered, orders uniform."""
    orders = random.Random(4402)
    for m in range(case["count"]):
        n = orders.randint(case["lo"], case["hi"])
        yield _matrix("ham", n, g) if m % 2 else _matrix("lap2d", max(2, math.isqrt(n)), g)


def _inputs(case, seed):
    """Everything a case draws: plain tensors, the same for ``prepare`` and ``exact``."""
    g = _gen(seed)
    kind = case["kind"]
    dt = _DT[case.get("dtype", "f64")]
    if kind == "batch":
        mats = [(rp, col, val.to(dt), n, _uniform(g, n).to(dt)) for rp, col, val, n in _members(case, g)]
        return dict(mats=mats)
    rp, col, val, n = _matrix(case["pattern"], case["n"], g, upper_only=kind == "sym")
    s = dict(rp=rp, col=col, val=val.to(dt), n=n)
    if kind == "spmm":
        s["x"] = _uniform(g, n, case["nrhs"])
    else:
        s["x"] = _uniform(g, n).to(dt)
    if kind in ("train", "grad"):
        s["g"] = _uniform(g, n).to(dt)
    if kind == "apply" and case["beta"] != 0.0:
        s["y"] = _uniform(g, n).to(dt)
    return s


def prepare(case, seed):
    s = _inputs(case, seed)
    s["case"] = case
    kind = case["kind"]
    if kind == "batch":
        mats = s.pop("mats")
        s["xs"] = [m[4] for m in mats]
        s["ys"] = [torch.empty_like(x) for x in s["xs"]]
        s["A"] = [Matrix.from_csr(rp, col, val, n) for rp, col, val, n, _ in mats]
        s["batch"] = Batch(s["A"])
        return s
    rp, col, val = s.pop("rp"), s.pop("col"), s.pop("val")
    if kind == "sym":
        s["A"] = Matrix.from_symmetric_upper(rp.cpu().numpy(), col.cpu().numpy(), val.cpu().numpy())
        return s
    s["A"] = Matrix.from_csr(rp, col, val, s["n"])
    if kind == "train":
        s["val"] = val.requires_grad_(True)
        s["x"].requires_grad_(True)
    if kind == "split":
        s["split"] = s["A"].split(case["blocks"])
        s["comm"] = torch.cuda.Stream()
        s["y"] = torch.empty_like(s["x"])
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "apply":
        if case["beta"] == 0.0:
            return s["A"].apply(s["x"], alpha=case["alpha"])
        return s["A"].apply(s["x"], s["y"], alpha=case["alpha"], beta=case["beta"])
    if kind == "sym":
        return s["A"].apply(s["x"])
    if kind == "split":
        return s["split"].apply(s["x"], s["y"], s_comm=s["comm"])
    if kind == "spmm":
        return s["A"].spmm(s["x"])
    if kind == "train":
        y = spmv(s["A"], s["val"], s["x"])
        gx, gv = torch.autograd.grad(y, (s["x"], s["val"]), s["g"])
        return dict(y=y, grad_x=gx, grad_val=gv)
    if kind == "grad":
        gx, gv = s["A"].backward(s["g"], s["x"])
        return dict(grad_x=gx, grad_val=gv)
    if kind == "batch":
        s["batch"].apply(s["xs"], s["ys"])
        return s["ys"]
    if kind == "cg":
        return cg(s["A"], s["x"], tol=case["tol"])[0]
    return ir_cg(s["A"], s["x"], outer_tol=case["tol"])[0]


# --------------------------------------------------------------------------------------
# Work and exact results
# --------------------------------------------------------------------------------------

def _shape(case, pattern=None, n=None):
    """(order, entries) of a case's matrix (the scattered pattern: its mean)."""
    pattern, n = pattern or case["pattern"], n or case["n"]
    if pattern == "ham":
        return n, int(12.85 * n)
    if pattern == "lap2d":
        return n * n, 5 * n * n - 4 * n
    if pattern == "poisson7":
        return n ** 3, 7 * n ** 3 - 6 * n * n
    return n ** 3, (3 * n - 2) ** 3


def work(case):
    kind = case["kind"]
    vb = 8 if case.get("dtype", "f64") == "f64" else 4
    if kind == "batch":
        mean = (case["lo"] + case["hi"]) // 2
        half = case["count"] / 2
        (na, ea), (nb, eb) = _shape(case, "lap2d", math.isqrt(mean)), _shape(case, "ham", mean)
        nnz, n = half * (ea + eb), half * (na + nb)
        return dict(bytes=(vb + 4) * nnz + (4 + 2 * vb) * n, flops=2 * nnz)
    n, nnz = _shape(case)
    matrix = (vb + 4) * nnz + 4 * n  # values, column indices, row pointers, each once
    if kind == "apply":
        return dict(bytes=matrix + (2 if case["beta"] == 0.0 else 3) * vb * n, flops=2 * nnz)
    if kind == "split":
        return dict(bytes=matrix + 2 * vb * n, flops=2 * nnz)
    if kind == "sym":
        return dict(bytes=(vb + 4) * (nnz + n) / 2 + 4 * n + 2 * vb * n, flops=2 * nnz)
    if kind == "spmm":
        r = case["nrhs"]
        return dict(bytes=matrix + 2 * vb * n * r, flops=2 * nnz * r)
    if kind == "train":  # new values in, y, grad_x and grad_val out, the pattern read once
        return dict(bytes=(vb + 4) * nnz + 4 * n + vb * nnz + 4 * vb * n, flops=5 * nnz)
    if kind == "grad":
        return dict(bytes=(vb + 4) * nnz + 4 * n + vb * nnz + 3 * vb * n, flops=3 * nnz)
    # solvers: about 1.8 (2D) or 2.5 (3D) iterations per grid point of an edge to reach 1e-12 (the
    # mixed solver a third more, in FP32); each reads the matrix and moves the four CG vectors
    if kind == "cg":
        its = int((3.0 if case["pattern"] == "lap2d" else 4.5) * case["n"])
        return dict(bytes=its * (matrix + 9 * 8 * n), flops=its * (2 * nnz + 10 * n))
    its = int(6.0 * case["n"])
    return dict(bytes=its * (8 * nnz + 4 * n + 9 * 4 * n), flops=its * (2 * nnz + 10 * n))


def _product(rp, col, val, x):
    """A x in 64 bits (x: a vector or the columns of a block)."""
    row = _rows(rp, col)
    val, x, col = val.double(), x.double(), col.long()
    if x.dim() == 1:
        return torch.zeros(rp.numel() - 1, dtype=torch.float64, device=_DEV).index_add_(0, row, val * x[col])
    return torch.stack([_product(rp, col, val, x[:, r].contiguous()) for r in range(x.shape[1])], 1)


def _poisson_solve(dims, n, b):
    """A^-1 b of the 5- or 7-point Laplacian by its sine eigenvectors, in 64 bits."""
    k = torch.arange(1, n + 1, dtype=torch.float64, device=_DEV)
    s = torch.sin(math.pi / (n + 1) * k[:, None] * k[None, :]) * math.sqrt(2.0 / (n + 1))
    lam = 2.0 - 2.0 * torch.cos(math.pi / (n + 1) * k)
    u = b.view(*[n] * dims)
    for d in range(dims):
        u = torch.movedim(torch.tensordot(s, u, dims=([1], [d])), 0, d)
    u = u / sum(lam.view(*[-1 if e == d else 1 for e in range(dims)]) for d in range(dims))
    for d in range(dims):
        u = torch.movedim(torch.tensordot(s, u, dims=([1], [d])), 0, d)
    return u.reshape(-1)


def exact(case, seed):
    kind = case["kind"]
    s = _inputs(case, seed)
    if kind == "batch":
        return [_product(rp, col, val, x) for rp, col, val, _, x in s["mats"]]
    if kind in ("cg", "ir_cg"):
        return _poisson_solve(2 if case["pattern"] == "lap2d" else 3, case["n"], s["x"])
    rp, col, val, x = s["rp"], s["col"], s["val"], s["x"]
    if kind == "sym":
        row = _rows(rp, col)
        y = _product(rp, col, val, x)
        off = (col != row).double() * val.double() * x.double()[row]
        return y.index_add_(0, col.long(), off)
    if kind in ("train", "grad"):
        row, g = _rows(rp, col), s["g"].double()
        gx = torch.zeros(s["n"], dtype=torch.float64, device=_DEV).index_add_(0, col.long(), val.double() * g[row])
        out = dict(grad_x=gx, grad_val=g[row] * x.double()[col.long()])
        return dict(y=_product(rp, col, val, x), **out) if kind == "train" else out
    y = _product(rp, col, val, x)
    if kind == "apply":
        y = case["alpha"] * y + (case["beta"] * s["y"].double() if case["beta"] else 0.0)
    return y
