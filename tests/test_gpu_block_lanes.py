"""Block vectors with lanes across the right-hand sides: every width of a pass (each
number of right-hand sides per lane, full and partly filled last lanes, idle lanes),
odd leading dimensions and unaligned blocks, row lengths around the blocks of loads,
empty and long rows, against the oracle."""
import numpy as np
import pytest

import oracle
from paper_1106_5908_gb300 import workloads as W
from gpu_util import assert_bitexact, assert_within, dev, host, need_gpu

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _gpu():
    need_gpu()


def matrix(kind, integer=False):
    """Rows of nearly equal length, so the slices pad little; `stencil` keeps its
    columns near the diagonal, `scattered` does not."""
    rng = np.random.default_rng(11)
    n = 1000
    lens = rng.integers(6, 8, n)
    lens[:64] = 0
    lens[64:128] = np.arange(64) % 5 + 1  # one slice of short rows
    lens[500] = 300                       # a long row
    rows = []
    for i in range(n):
        if kind == "stencil":
            rows.append(np.clip(i - lens[i] // 2 + np.arange(lens[i]), 0, n - 1))
        else:
            rows.append(rng.integers(0, n, lens[i]))
    rp = np.zeros(n + 1, np.int32)
    rp[1:] = np.cumsum(lens)
    col = np.concatenate(rows).astype(np.int32)
    val = rng.integers(-4, 5, col.size).astype(np.float64) if integer else rng.standard_normal(col.size)
    return W.CRS(rp, col, val, n)


@pytest.mark.parametrize("kind", ["stencil", "scattered"])
@pytest.mark.parametrize("nrhs", list(range(2, 34)) + [48, 63, 64])
def test_every_width(kind, nrhs):
    from paper_1106_5908_gb300 import Matrix
    A = matrix(kind)
    M = Matrix.from_csr(A.row_ptr, A.col_idx, A.val, A.n_cols)
    X, Y0 = W.uniform(0, 1, shape=(A.n_cols, nrhs)), W.uniform(0, 2, shape=(A.n_rows, nrhs))
    ref, bound = oracle.spmm(*A.astuple(), X, with_bound=True)
    for alpha, beta in ((1.0, 0.0), (-0.5, 0.75)):
        Y = dev(Y0) if beta else torch.full((A.n_rows, nrhs), float("nan"), dtype=torch.float64, device="cuda")
        M.spmm(dev(X), Y, alpha, beta)
        assert_within(host(Y), alpha * ref + beta * Y0, abs(alpha) * bound + abs(beta) * np.abs(Y0), 1e-13,
                      f"{kind} {nrhs} {alpha} {beta}")


@pytest.mark.parametrize("nrhs", [2, 4, 8, 16])
def test_unaligned_blocks(nrhs):
    """X and Y 8 bytes off a 16-byte boundary; integers, so the sums are exact."""
    from paper_1106_5908_gb300 import Matrix
    A = matrix("scattered", integer=True)
    M = Matrix.from_csr(A.row_ptr, A.col_idx, A.val, A.n_cols)
    X = W.integers(A.n_cols * nrhs, 5).reshape(A.n_cols, nrhs)
    buf = torch.zeros(A.n_cols * nrhs + 1, dtype=torch.float64, device="cuda")
    buf[1:] = dev(X).reshape(-1)
    Xo = buf[1:].view(A.n_cols, nrhs)
    Yo = torch.zeros(A.n_rows * nrhs + 1, dtype=torch.float64, device="cuda")[1:].view(A.n_rows, nrhs)
    assert Xo.data_ptr() % 16 == 8 and Yo.data_ptr() % 16 == 8
    M.spmm(Xo, Yo)
    assert_bitexact(host(Yo), oracle.spmm(*A.astuple(), X), f"unaligned {nrhs}")
