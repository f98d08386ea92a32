"""A symmetric handle sums in one order: the same values and x give the same bits from
the first apply on, after new values, captured or not, on any stream.  A handle whose first
apply is captured keeps to the two passes."""
import pytest

import oracle
from paper_1106_5908_gb300 import workloads as W
from gpu_util import assert_within, dev, host, need_gpu

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _gpu():
    need_gpu()


def _upper(kind):
    if kind == "scattered":
        return W.upper_triangle(W.hamiltonian_like(30000, seed=4))
    if kind == "grid":
        return W.upper_triangle(W.laplace3d(28))
    if kind == "27-point":
        return W.upper_triangle(W.stencil27(20))
    return W.random_symmetric_upper(20000, seed=5, max_len=40)  # rows of all lengths, empty ones too


def _sym(U, dtype):
    from paper_1106_5908_gb300 import Matrix
    return Matrix.from_symmetric_upper(U.row_ptr, U.col_idx, U.val, dtype=dtype)


def _captured(M, x):
    y = torch.empty_like(x)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        M.apply(x, y)
    g.replay()
    return y


@pytest.mark.parametrize("kind", ["scattered", "grid", "27-point", "uneven"])
@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
def test_same_bits(kind, dtype):
    U = _upper(kind)
    M = _sym(U, dtype)
    tol = 1e-13 if dtype == torch.float64 else 1e-6
    x = dev(W.uniform(U.n_rows, 3), dtype)
    other = torch.cuda.Stream()
    val = dev(U.val, dtype)
    for seed in (None, 8, 9, None):
        val = dev(U.val if seed is None else W.uniform(U.nnz, seed), dtype)
        M.set_values(val)
        first = M.apply(x)
        other.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(other):
            elsewhere = M.apply(x)
        torch.cuda.current_stream().wait_stream(other)
        for y in (M.apply(x), elsewhere, _captured(M, x)):
            assert torch.equal(first, y), seed
        ref, bound = oracle.spmv_sym(U.row_ptr, U.col_idx, host(val.double()), host(x.double()), with_bound=True)
        assert_within(host(first), ref, bound, tol, f"{kind} {seed}")
        M.set_values(val)
        assert torch.equal(first, _captured(M, x)) and torch.equal(first, M.apply(x))


def test_one_apply_of_the_first_values_then_new_ones():
    """The same bits as a handle created with those values."""
    U = _upper("scattered")
    M = _sym(U, torch.float64)
    x = dev(W.uniform(U.n_rows, 3))
    M.apply(x)
    U.val[:] = W.uniform(U.nnz, 21)
    M.set_values(dev(U.val))
    assert torch.equal(M.apply(x), _sym(U, torch.float64).apply(x))


@pytest.mark.parametrize("kind", ["scattered", "grid", "uneven"])
@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
def test_first_new_values_captured(kind, dtype):
    """The first values after the ones of creation are filled in by a graph; then graph and
    handle take new values in turn."""
    U = _upper(kind)
    tol = 1e-13 if dtype == torch.float64 else 1e-6
    M = _sym(U, dtype)
    x = dev(W.uniform(U.n_rows, 3), dtype)
    y = torch.empty_like(x)
    M.apply(x)
    source = torch.empty(U.nnz, dtype=dtype, device="cuda")
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        M.set_values(source)
        M.apply(x, y)
        M.apply(x, y, alpha=1.0, beta=1.0)

    def check(got, val, times, what):
        ref, bound = oracle.spmv_sym(U.row_ptr, U.col_idx, host(val.double()), host(x.double()), with_bound=True)
        assert_within(host(got), times * ref, (2 * times - 1) * bound, tol, f"{kind} {what}")

    for turn in range(4):
        val = dev(W.uniform(U.nnz, 40 + turn), dtype)
        if turn % 2:
            M.set_values(val)
            check(M.apply(x), val, 1, turn)
        val = dev(W.uniform(U.nnz, 50 + turn), dtype)
        source.copy_(val)
        g.replay()
        check(y, val, 2, turn)


@pytest.mark.parametrize("kind", ["scattered", "uneven"])
def test_fp32_sums_out_of_range_follow_new_values(kind):
    """Products below 2^-100 are summed again in FP64, from the values of U."""
    U = _upper(kind)
    M = _sym(U, torch.float32)
    x = dev(W.uniform(U.n_rows, 3) * 2.0 ** -40, torch.float32)
    M.apply(x)
    for seed in (8, 9, 10):
        val = dev(W.uniform(U.nnz, seed) * 2.0 ** -70, torch.float32)
        M.set_values(val)
        ref, bound = oracle.spmv_sym(U.row_ptr, U.col_idx, host(val.double()), host(x.double()), with_bound=True)
        for _ in range(2):
            y = M.apply(x)
            assert_within(host(y), ref, bound, 2.0 ** -23, f"{kind} {seed}")  # the store's rounding alone


def test_first_apply_captured():
    U = _upper("grid")
    M = _sym(U, torch.float64)
    x = dev(W.uniform(U.n_rows, 3))
    y = torch.empty_like(x)
    ref, bound = oracle.spmv_sym(*U.astuple(), host(x), with_bound=True)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, capture_error_mode="relaxed"):  # the chunk tables are uploaded meanwhile
        M.apply(x, y)
    assert_within(host(M.apply(x)), ref, bound, 1e-13, "before the graph's first run")
    g.replay()
    assert_within(host(y), ref, bound, 1e-13, "replayed")
    assert torch.equal(M.apply(x), M.apply(x))
