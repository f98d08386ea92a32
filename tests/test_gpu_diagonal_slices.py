"""The row-slice kernel on diagonal slices (slot rows whose 64 entries lie on one
diagonal need no column indices) against the oracle, at the edges of its range:
widths around its blocks of 8 slot rows and its 4 diagonals per load, orders around
a slice of 64 rows, slices broken by irregular, empty and long rows."""
import numpy as np
import pytest

import oracle
from paper_1106_5908_gb300 import workloads as W
from tests.gpu_util import assert_bitexact, assert_within, dev, host, need_gpu

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _gpu():
    need_gpu()


def banded(n, width, seed, broken=0, long_rows=0, integer=False):
    """n x n matrix with `width` diagonals (cut at the edges); `broken` rows get
    their columns shifted by one, `broken` more are empty, `long_rows` have 200."""
    rng = np.random.default_rng(seed)
    offs = np.sort(rng.choice(np.arange(-3 * width, 3 * width + 1), width, replace=False))
    rows = []
    for i in range(n):
        c = i + offs
        rows.append(c[(c >= 0) & (c < n)])
    pick = rng.permutation(n)
    for i in pick[:broken]:
        rows[i] = np.minimum(rows[i] + 1, n - 1)
    for i in pick[broken:2 * broken]:
        rows[i] = rows[i][:0]
    for i in pick[2 * broken:2 * broken + long_rows]:
        rows[i] = rng.integers(0, n, 200)
    rp = np.zeros(n + 1, np.int32)
    rp[1:] = np.cumsum([len(r) for r in rows])
    col = np.concatenate(rows).astype(np.int32)
    val = rng.integers(-4, 5, col.size).astype(np.float64) if integer else rng.standard_normal(col.size)
    return W.CRS(rp, col, val, n)


@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("n,width,broken,long_rows", [
    (63, 1, 0, 0), (64, 1, 0, 0), (65, 3, 0, 0), (5000, 1, 0, 0), (5000, 4, 3, 0), (5000, 5, 0, 2), (9000, 7, 5, 1),
    (4097, 8, 2, 0), (8191, 9, 0, 0), (20000, 12, 10, 3), (20000, 16, 0, 0), (9000, 17, 4, 0), (6000, 33, 2, 2),
    (5000, 128, 0, 0), (70000, 5, 7, 3)])
def test_diagonal_slices_match_the_oracle(n, width, broken, long_rows, dtype):
    from paper_1106_5908_gb300 import Matrix
    tol = 1e-13 if dtype == "f64" else 1e-6  # the library's bounds for FP64 and FP32 storage
    ft = np.float64 if dtype == "f64" else np.float32
    A = banded(n, width, seed=n + width, broken=broken, long_rows=long_rows)
    val, x, y0 = A.val.astype(ft), W.uniform(n, 1).astype(ft), W.uniform(n, 2).astype(ft)
    M = Matrix.from_csr(A.row_ptr, A.col_idx, val, n)
    M.set_plan(5, 0)
    for alpha, beta in ((1.0, 0.0), (-0.5, 0.0), (1.0, 1.0), (2.0, -0.75)):
        ref, bound = oracle.spmv(A.row_ptr, A.col_idx, val.astype(np.float64), x.astype(np.float64), with_bound=True)
        want = alpha * ref + beta * y0.astype(np.float64)
        lim = abs(alpha) * bound + abs(beta) * np.abs(y0).astype(np.float64)
        y = torch.full((n,), float("nan"), device="cuda", dtype=torch.float64 if ft is np.float64 else torch.float32)
        if beta:
            y = dev(y0)
        assert_within(host(M.apply(dev(x), y, alpha, beta)), want, lim, tol, f"{n} {width} {alpha} {beta}")
    # new values, integers: exact sums
    B = banded(n, width, seed=n + width, broken=broken, long_rows=long_rows, integer=True)
    M.set_values(dev(B.val.astype(ft)))
    xi = W.integers(n, 3)
    assert_bitexact(host(M.apply(dev(xi.astype(ft)))).astype(np.float64), oracle.spmv(*B.astuple(), xi), "integers")


@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("n,width,broken", [(65, 3, 0), (5000, 4, 3), (9000, 7, 5), (70, 10, 0), (8191, 9, 0),
                                            (5003, 12, 40), (4097, 16, 3), (9001, 32, 2), (6000, 33, 2), (3000, 70, 1)])
def test_training_steps_match_the_oracle(n, width, broken, dtype):
    """New values, the forward product and reverse passes on them (the first reads
    A's slices through positions, the second A^T's own copy), each against the oracle."""
    from paper_1106_5908_gb300 import Matrix
    ft, tt = (np.float64, torch.float64) if dtype == "f64" else (np.float32, torch.float32)
    tol = 1e-13 if dtype == "f64" else 1e-6
    A = banded(n, width, seed=3 * n + width, broken=broken)
    M = Matrix.from_csr(A.row_ptr, A.col_idx, A.val.astype(ft), n)
    M.set_plan(5, 0)
    x, g = W.uniform(n, 1).astype(ft), W.uniform(n, 2).astype(ft)
    xd, gd = x.astype(np.float64), g.astype(np.float64)
    M.apply(dev(x))
    for step, alpha in enumerate((1.0, -0.5, 1.0)):
        # values of the other type every second step: converted as they are set
        raw = np.random.default_rng(step).standard_normal(A.nnz).astype(np.float32)
        M.set_values(dev(raw) if step % 2 else dev(raw.astype(ft)))
        val = raw.astype(np.float64)
        if step == 2:
            M.set_plan(5, 256)  # other slices: the positions of the values change
        ref, bound = oracle.spmv(A.row_ptr, A.col_idx, val, xd, with_bound=True)
        assert_within(host(M.apply(dev(x), alpha=alpha)), alpha * ref, abs(alpha) * bound, tol, f"forward {step}")
        rgx, rgv, gbound = oracle.backward(A.row_ptr, A.col_idx, val, n, gd, xd, with_bound=True)
        for rep in range(3):
            gx, gv = M.backward(dev(g), dev(x), alpha)
            assert gx.dtype == tt and gv.dtype == tt
            assert_within(host(gx), alpha * rgx, abs(alpha) * gbound, tol, f"grad_x {step} {rep}")
            assert_within(host(gv), alpha * rgv, np.abs(alpha * rgv), 1e-6 if dtype == "f32" else 1e-15, f"grad_val {step} {rep}")


def test_tuner_takes_grid_stencils():
    """FP64 stencils on a grid of at least 16,384 points run on the row slices
    whatever their row length; a banded matrix without diagonals does not."""
    from paper_1106_5908_gb300 import Matrix
    A = W.laplace2d(128)
    M = Matrix.from_csr(A.row_ptr, A.col_idx, A.val, A.n_cols)
    assert M.info()["family"] == 5
    xi = W.integers(A.n_rows, 4)
    assert_bitexact(host(M.apply(dev(xi))), oracle.spmv(*A.astuple(), xi), "5-point integers")
    rng = np.random.default_rng(5)
    n = 20000
    col = np.sort(np.clip(np.arange(n)[:, None] + rng.integers(-6, 7, (n, 5)), 0, n - 1), axis=1)
    M = Matrix.from_csr(np.arange(0, 5 * n + 1, 5, dtype=np.int32), col.reshape(-1).astype(np.int32),
                        rng.standard_normal(5 * n), n)
    assert M.info()["family"] == 4


@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("others", [0, 3])
def test_batch_members_on_diagonal_slices(others, dtype):
    """Large grid stencils of a batch run on their diagonal slices beside (or without)
    chunk members, follow new values and keep their own copy of them."""
    from paper_1106_5908_gb300 import Batch, Matrix
    ft, tol = (np.float64, 1e-13) if dtype == "f64" else (np.float32, 1e-6)
    As = [W.laplace2d(200, 190), W.laplace3d(33), W.laplace2d(181)]
    As += [W.hamiltonian_like(5000, seed=3), W.laplace2d(60), W.random_csr(700, 700, seed=4, max_len=4)][:others]
    mats = [Matrix.from_csr(A.row_ptr, A.col_idx, A.val.astype(ft), A.n_cols) for A in As]
    B = Batch(mats)
    assert B.info()["member_E"][:3] == [0, 0, 9]  # the last has 32,761 rows
    xs = [W.uniform(A.n_cols, 50 + m).astype(ft) for m, A in enumerate(As)]
    y0 = [W.uniform(A.n_rows, 80 + m).astype(ft) for m, A in enumerate(As)]
    vals = [A.val.astype(ft) for A in As]
    for rep, (alpha, beta) in enumerate(((1.0, 0.0), (1.0, 0.0), (-1.5, 0.5))):
        if rep:
            vals[0] = W.uniform(As[0].nnz, 90 + rep).astype(ft)
            mats[0].set_values(dev(vals[0]))
        xd, yd = [dev(x) for x in xs], [dev(y) for y in y0]
        B.apply(xd, yd, alpha, beta)
        for m, A in enumerate(As):
            ref, bound = oracle.spmv(A.row_ptr, A.col_idx, vals[m].astype(np.float64), xs[m].astype(np.float64), alpha,
                                     beta, y0[m].astype(np.float64), with_bound=True)
            assert_within(host(yd[m]), ref, bound, tol, f"member {m} rep {rep}")
