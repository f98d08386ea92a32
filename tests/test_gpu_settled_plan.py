"""A matrix whose rows look like a stencil's to the tuner but whose slices are not
diagonal: 63 of 64 rows lie on three diagonals, the 64th on others.  The first call finds
out: the handle reports and runs the slot-major kernel, and keeps no row slices."""
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


def _broken_band(n):
    i = np.arange(n)
    col = np.stack([i, (i + 1) % n, np.where(i % 64 == 10, (i + 3) % n, (i + 2) % n)], 1).astype(np.int32)
    return np.arange(0, 3 * n + 1, 3, dtype=np.int32), col.ravel(), W.uniform(3 * n, 4), n


def _matrix(args):
    from paper_1106_5908_gb300 import Matrix
    return Matrix.from_csr(*args)


@pytest.mark.parametrize("n", [16384, 30001])
@pytest.mark.parametrize("first", ["apply", "info", "cg"])
def test_falls_back_to_the_chunks(n, first):
    from paper_1106_5908_gb300 import cg
    args = _broken_band(n)
    M, N = _matrix(args), _matrix(args)
    N.set_plan(4, 7)
    x = dev(W.uniform(n, 5))
    if first == "apply":
        M.apply(x)
    elif first == "cg":
        cg(M, x, max_iter=3)
        M.apply(x)
    assert (M.info()["family"], M.info()["E"]) == (4, 7)
    for seed in (None, 8):
        if seed is not None:
            val = W.uniform(3 * n, seed)
            M.set_values(dev(val)), N.set_values(dev(val))
            args = (*args[:2], val, n)
        ref, bound = oracle.spmv(*args[:3], host(x), with_bound=True)
        y = M.apply(x)
        assert_within(host(y), ref, bound, 1e-13, first)
        assert torch.equal(y, N.apply(x))


def test_keeps_no_slices():
    n = 2_000_000
    args = [dev(a) for a in _broken_band(n)[:3]] + [n]
    x = torch.rand(n, dtype=torch.float64, device="cuda")
    y = torch.empty_like(x)
    _matrix(args).apply(x, y)  # the library's and torch's own first allocations
    used = []
    for plan in (None, (4, 7)):
        M = _matrix(args)
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        if plan:
            M.set_plan(*plan)
        M.apply(x, y)
        M.set_values(args[2])
        M.apply(x, y)
        torch.cuda.synchronize()
        used.append(before - torch.cuda.mem_get_info()[0])
        M.close()
    assert used[0] <= used[1] + (8 << 20), used  # the slices take 80 MB


def test_diagonal_ones_stay():
    A = W.laplace2d(140)
    M = _matrix((A.row_ptr, A.col_idx, A.val, A.n_cols))
    assert M.info()["family"] == 5
    x = dev(W.uniform(A.n_cols, 5))
    M.apply(x)
    assert M.info()["family"] == 5
