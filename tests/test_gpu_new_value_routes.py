"""New values, products and reverse passes in any order: each sees the last values set,
whichever copy they went to (with the CRS copy in one pass, or laid out by the call that
needs them)."""
import random

import numpy as np
import pytest

import oracle
from paper_1106_5908_gb300 import workloads as W
from gpu_util import assert_within, dev, host, need_gpu

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _gpu():
    need_gpu()


# below and above the entries from which the reverse passes read A's slices
@pytest.mark.parametrize("kind,n", [("5-point", 131), ("5-point", 290), ("7-point", 27), ("7-point", 39), ("27-point", 26),
                                    ("27-point", 44)])
@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("seed", [1, 2])
def test_any_order(kind, n, dtype, seed):
    from paper_1106_5908_gb300 import Matrix
    A = {"5-point": W.laplace2d, "7-point": W.laplace3d, "27-point": W.stencil27}[kind](n)
    ft, tol = (np.float64, 1e-13) if dtype == "f64" else (np.float32, 1e-6)
    T = oracle.transpose(A.row_ptr, A.col_idx, A.n_cols)
    rows = np.repeat(np.arange(A.n_rows), np.diff(A.row_ptr.astype(np.int64)))
    x, g = W.uniform(A.n_cols, 3).astype(ft), W.uniform(A.n_rows, 4).astype(ft)
    xd, gd = dev(x), dev(g)
    val = A.val.astype(ft)
    M = Matrix.from_csr(A.row_ptr, A.col_idx, val, A.n_cols)
    rng = random.Random(seed)
    for step in range(40):
        op = rng.choice(["set", "set", "set_apply", "apply", "backward", "backward"])
        if op.startswith("set"):
            val = W.uniform(A.nnz, 100 + step).astype(ft)
        v64 = val.astype(np.float64)
        if op == "set":
            M.set_values(dev(val))
        elif op == "backward":
            gx, gv = M.backward(gd, xd)
            ref, bound = oracle.spmv(T[0], T[1], v64[T[2]], g.astype(np.float64), with_bound=True)
            assert_within(host(gx), ref, bound, tol, f"{step}")
            assert np.array_equal(host(gv), g[rows] * x[A.col_idx])
        else:
            y = M.apply(xd) if op == "apply" else M.set_values_apply(dev(val), xd)
            ref, bound = oracle.spmv(A.row_ptr, A.col_idx, v64, x.astype(np.float64), with_bound=True)
            assert_within(host(y), ref, bound, tol, f"{step}")
