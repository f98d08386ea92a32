"""Calls captured right after new values: what the capture records runs with the graph
only, so a call beside it, before its first run, uses the new values all the same; and
nothing is built while a stream is captured."""
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


def _matrix(kind):
    if kind == "grid":
        return W.laplace3d(28)  # 21,952 rows: diagonal slices
    if kind == "27-point":
        return W.stencil27(26)
    return W.hamiltonian_like(20000, seed=4)


@pytest.mark.parametrize("kind,plan", [("scattered", None), ("grid", None), ("scattered", (5, 4096)), ("scattered", (6, 9)),
                                       ("scattered", (0, 15))])
def test_apply_captured_on_new_values(kind, plan):
    from paper_1106_5908_gb300 import Matrix
    A = _matrix(kind)
    M = Matrix.from_csr(A.row_ptr, A.col_idx, A.val, A.n_cols)
    if plan:
        M.set_plan(*plan)
    x = dev(W.uniform(A.n_cols, 3))
    y = torch.zeros_like(x)
    M.apply(x)
    val = W.uniform(A.nnz, 6)
    M.set_plan(4, 9)  # leaves the copies of the matrix's own plan behind: they have to be laid out anew
    M.apply(x)
    M.set_values(dev(val))
    if plan or kind == "grid":
        M.set_plan(*(plan or (5, 4096)))
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        M.apply(x, y)
        M.apply(x, y, alpha=1.0, beta=1.0)
    ref, bound = oracle.spmv(A.row_ptr, A.col_idx, val, host(x), with_bound=True)
    assert_within(host(M.apply(x)), ref, bound, 1e-13, "before the graph's first run")
    for _ in range(2):
        g.replay()
        assert_within(host(y), 2 * ref, 3 * bound, 1e-13, "replayed")
    assert_within(host(M.apply(x)), ref, bound, 1e-13, "after the graph")


@pytest.mark.parametrize("applies", [0, 1, 2])
def test_symmetric_apply_captured_on_new_values(applies):
    from paper_1106_5908_gb300 import Matrix
    U = W.random_symmetric_upper(20000, seed=5, max_len=9)
    M = Matrix.from_symmetric_upper(U.row_ptr, U.col_idx, U.val)
    x = dev(W.uniform(U.n_rows, 3))
    y = torch.zeros_like(x)
    M.apply(x)
    val = W.uniform(U.nnz, 6)
    M.set_values(dev(val))
    for _ in range(applies):
        M.apply(x)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        M.apply(x, y)
    ref, bound = oracle.spmv_sym(U.row_ptr, U.col_idx, val, host(x), with_bound=True)
    for _ in range(3):
        assert_within(host(M.apply(x)), ref, bound, 1e-13, "before the graph's first run")
    y.zero_()
    g.replay()
    assert_within(host(y), ref, bound, 1e-13, "replayed")
    assert_within(host(M.apply(x)), ref, bound, 1e-13, "after the graph")


@pytest.mark.parametrize("kind", ["27-point", "scattered"])
@pytest.mark.parametrize("new_values", [False, True])
def test_reverse_pass_captured(kind, new_values):
    """The reverse passes build copies of A^T on the way; captured, they take what is
    there, with the values laid out once more by the next pass beside the graph."""
    from paper_1106_5908_gb300 import Matrix
    A = _matrix(kind)
    M = Matrix.from_csr(A.row_ptr, A.col_idx, A.val, A.n_cols)
    x, g = dev(W.uniform(A.n_cols, 3)), dev(W.uniform(A.n_rows, 4))
    M.backward(g, x)
    M.backward(g, x)
    val, vd = A.val, dev(W.uniform(A.nnz, 8))
    torch.cuda.synchronize()
    if new_values:
        val = host(vd)
        M.set_values(vd)
        M.backward(g, x)
        torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        gx, gv = M.backward(g, x)
        if not new_values:  # and a first pass on values set in the graph
            M.set_values(vd)
            gx2, gv2 = M.backward(g, x)
    T = oracle.transpose(A.row_ptr, A.col_idx, A.n_cols)

    def check(got, v, what):
        ref, bound = oracle.spmv(T[0], T[1], v[T[2]], host(g), with_bound=True)
        assert_within(host(got[0]), ref, bound, 1e-13, what)
        rows = np.repeat(np.arange(A.n_rows), np.diff(A.row_ptr.astype(np.int64)))
        assert np.array_equal(host(got[1]), host(g)[rows] * host(x)[A.col_idx]), what

    check(M.backward(g, x), val, "before the graph's first run")
    graph.replay()
    check((gx, gv), val, "replayed")
    if not new_values:
        check((gx2, gv2), host(vd), "replayed, new values")
    M.set_values(vd)
    check(M.backward(g, x), host(vd), "after the graph")


def test_captured_reverse_pass_outlives_its_plan():
    """A first reverse pass on new values reads positions that belong to the window of A's
    slices; a pass on another window beside the graph leaves the graph's alone."""
    from paper_1106_5908_gb300 import Matrix
    A = W.stencil27(26)
    M = Matrix.from_csr(A.row_ptr, A.col_idx, A.val, A.n_cols)
    x, g, source = dev(W.uniform(A.n_cols, 3)), dev(W.uniform(A.n_rows, 4)), dev(A.val)
    T = oracle.transpose(A.row_ptr, A.col_idx, A.n_cols)

    def step():
        M.set_values(source)
        M.apply(x)
        return M.backward(g, x)[0]

    for _ in range(2):
        step()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        gx = step()
    for turn, window in enumerate((64, 4096, 1024)):
        val = W.uniform(A.nnz, 30 + turn)
        source.copy_(dev(val))
        ref, bound = oracle.spmv(T[0], T[1], val[T[2]], host(g), with_bound=True)
        M.set_plan(5, window)
        for _ in range(2):
            assert_within(host(step()), ref, bound, 1e-13, f"{window}")
        gx.zero_()
        graph.replay()
        assert_within(host(gx), ref, bound, 1e-13, f"replayed after {window}")


@pytest.mark.parametrize("dtype", ["f64", "f32"])
def test_first_reverse_pass_captured_on_short_rows(dtype):
    """On large grids of short rows a first reverse pass takes A's slices when a product has
    laid them out and the permutation when not: a capture of the one that has not run yet
    builds nothing either."""
    from paper_1106_5908_gb300 import Matrix
    A = W.laplace2d(290)  # 419,340 entries
    ft, tol = (np.float64, 1e-13) if dtype == "f64" else (np.float32, 1e-6)
    M = Matrix.from_csr(A.row_ptr, A.col_idx, A.val.astype(ft), A.n_cols)
    x, g = dev(W.uniform(A.n_cols, 3).astype(ft)), dev(W.uniform(A.n_rows, 4).astype(ft))
    source = dev(A.val.astype(ft))
    T = oracle.transpose(A.row_ptr, A.col_idx, A.n_cols)
    M.apply(x)
    for _ in range(2):  # on the slices
        M.set_values_apply(source, x)
        M.backward(g, x)
    M.set_values(source)
    M.backward(g, x)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        M.set_values(source)  # nothing has read the slices since the last values
        gx, gv = M.backward(g, x)
    for seed in (5, 6):
        val = W.uniform(A.nnz, seed).astype(ft)
        source.copy_(dev(val))
        graph.replay()
        ref, bound = oracle.spmv(T[0], T[1], val[T[2]].astype(np.float64), host(g).astype(np.float64), with_bound=True)
        assert_within(host(gx), ref, bound, tol, f"replayed {seed}")
