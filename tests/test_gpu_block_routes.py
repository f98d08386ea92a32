"""Block vectors on each of their routes: lanes across the right-hand sides (no long
rows), two rows per lane in groups of 4 (long rows), and the tile kernel (2 or 3
right-hand sides on few rows), on both sides of the sizes where the route changes."""
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


def _matrix(n, kind, lens):
    rng = np.random.default_rng(n)
    rp = np.zeros(n + 1, np.int32)
    rp[1:] = np.cumsum(lens)
    row = np.repeat(np.arange(n), lens)
    at = np.arange(rp[-1]) - rp[row]
    col = (row + at) % n if kind == "stencil" else rng.integers(0, n, rp[-1])
    return W.CRS(rp, col.astype(np.int32), rng.standard_normal(rp[-1]), n)


def _check(A, nrhs, plan=None):
    from paper_1106_5908_gb300 import Matrix
    M = Matrix.from_csr(A.row_ptr, A.col_idx, A.val, A.n_cols)
    X, Y0 = W.uniform(A.n_cols * nrhs, 3).reshape(-1, nrhs), W.uniform(A.n_rows * nrhs, 4).reshape(-1, nrhs)
    for alpha, beta in ((1.0, 0.0), (-0.75, 0.5)):
        Y = dev(Y0)
        M.spmm(dev(X), Y, alpha=alpha, beta=beta)
        ref, bound = oracle.spmm(*A.astuple(), X, alpha, beta, Y0, with_bound=True)
        assert_within(host(Y), ref, bound, 1e-13, f"{A.n_rows} {nrhs}")
    M.close()


@pytest.mark.parametrize("kind", ["stencil", "scattered"])
@pytest.mark.parametrize("nrhs", list(range(2, 35)) + [64])
@pytest.mark.parametrize("longest", [0, 129, 900])
def test_every_width(kind, nrhs, longest):
    rng = np.random.default_rng(12)
    lens = rng.integers(6, 8, 1000)
    lens[:64] = 0
    lens[64:128] = np.arange(64) % 5 + 1
    if longest:
        lens[500] = lens[999] = longest
    _check(_matrix(1000, kind, lens), nrhs)


@pytest.mark.parametrize("kind,n", [("stencil", 65535), ("stencil", 65536), ("scattered", 262143), ("scattered", 262144)])
@pytest.mark.parametrize("nrhs", [2, 3, 4])
def test_few_right_hand_sides_at_the_edges(kind, n, nrhs):
    _check(_matrix(n, kind, np.full(n, 5)), nrhs)
