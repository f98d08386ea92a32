"""CG as one cooperative kernel (matrices on diagonal row slices): solutions against
the matrix they solve, at the edges of its range: fewer rows than a slice, one CTA
and many, rows on either side of 8 and 11 entries, the matrix values in shared
memory and not, iteration caps between two convergence tests."""
import numpy as np
import pytest

import oracle
from paper_1106_5908_gb300 import workloads as W
from gpu_util import dev, host, need_gpu

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _gpu():
    need_gpu()


def band(n, half):
    """Symmetric positive definite Toeplitz band: -1 on `half` diagonals either
    side, 2*half + 0.1 on the diagonal."""
    offs = np.arange(-half, half + 1)
    col = np.arange(n)[:, None] + offs[None, :]
    ok = (col >= 0) & (col < n)
    val = np.where(offs == 0, 2 * half + 0.1, -1.0)[None, :].repeat(n, 0)
    rp = np.zeros(n + 1, np.int32)
    rp[1:] = np.cumsum(ok.sum(1))
    return W.CRS(rp, col[ok].astype(np.int32), val[ok], n)


def cases():
    for n, half in ((40, 1), (64, 1), (65, 2), (1000, 1), (5000, 3), (30000, 5), (30000, 6), (20000, 16)):
        yield pytest.param(lambda n=n, half=half: band(n, half), id=f"band-{n}-{half}")
    yield pytest.param(lambda: W.laplace2d(101), id="5-point-101")
    yield pytest.param(lambda: W.laplace3d(88), id="7-point-88")  # values stay in L2 in FP64


@pytest.mark.parametrize("make", list(cases()))
def test_solves(make):
    from paper_1106_5908_gb300 import Matrix, cg, ir_cg
    A = make()
    M = Matrix.from_csr(A.row_ptr, A.col_idx, A.val, A.n_cols)
    b = W.uniform(A.n_rows, 7)
    nb = np.linalg.norm(b)
    x, st = cg(M, dev(b), tol=1e-12)
    assert st["converged"], st
    # the recursive residual stops at 1e-12; its gap to the true one is of order
    # iterations * u (2.2e-16)
    assert np.linalg.norm(oracle.residual(*A.astuple(), b, host(x))) <= (1e-12 + st["inner"] * 2.3e-16 * 4) * nb, st
    assert st["inner"] % 8 == 0
    x, st = ir_cg(M, dev(b))
    assert st["converged"], st
    assert np.linalg.norm(oracle.residual(*A.astuple(), b, host(x))) <= 1.5e-12 * nb, st
    M.check_device_error()


@pytest.mark.parametrize("cap", [0, 1, 7, 8, 13])
def test_iteration_caps(cap):
    """A capped solve takes exactly `cap` steps of textbook CG and reports that it
    has not converged."""
    from paper_1106_5908_gb300 import Matrix, cg
    A = W.laplace2d(70)
    M = Matrix.from_csr(A.row_ptr, A.col_idx, A.val, A.n_cols)
    b = W.uniform(A.n_rows, 9)
    x, st = cg(M, dev(b), tol=1e-12, max_iter=cap)
    assert not st["converged"] and st["inner"] == cap
    want, r, p = np.zeros_like(b), b.copy(), b.copy()
    rho = r @ r
    for _ in range(cap):
        q = oracle.spmv(*A.astuple(), p)
        a = rho / (p @ q)
        want += a * p
        r -= a * q
        rho, old = r @ r, rho
        p = r + rho / old * p
    assert np.linalg.norm(host(x) - want) <= 1e-12 * max(1.0, np.linalg.norm(want))


def test_zero_right_hand_side_and_new_values():
    from paper_1106_5908_gb300 import Matrix, cg
    A = W.laplace2d(64)
    M = Matrix.from_csr(A.row_ptr, A.col_idx, A.val, A.n_cols)
    x, st = cg(M, torch.zeros(A.n_rows, dtype=torch.float64, device="cuda"))
    assert st["converged"] and st["inner"] == 0 and not host(x).any()
    b = W.uniform(A.n_rows, 3)
    x1, _ = cg(M, dev(b))
    M.set_values(dev(2.0 * A.val))
    x2, st = cg(M, dev(b))
    assert st["converged"]
    assert np.linalg.norm(2.0 * host(x2) - host(x1)) <= 1e-9 * np.linalg.norm(host(x1))


@pytest.mark.parametrize("kind", ["grid", "scattered"])
def test_solvers_follow_new_values(kind):
    """Both solvers after spmv_set_values, on the one-kernel path and (scattered
    columns) on the captured iterations, into the same x as before."""
    from paper_1106_5908_gb300 import Matrix, _abi
    if kind == "grid":
        A = W.laplace2d(80)
        val2 = A.val * 3.0
    else:
        H = W.hamiltonian_like(6000, seed=21)
        rows = np.repeat(np.arange(H.n_rows), np.diff(H.row_ptr.astype(np.int64)))
        off = rows != H.col_idx
        rowabs = np.bincount(rows[off], weights=np.abs(H.val[off]), minlength=H.n_rows)
        v = H.val.copy()
        v[~off] = rowabs[rows[~off]] + 1.0  # diagonally dominant: SPD
        A = W.CRS(H.row_ptr, H.col_idx, v, H.n_cols)
        val2 = A.val.copy()
        val2[~off] += 40.0  # another matrix, not a multiple of the first
    M = Matrix.from_csr(A.row_ptr, A.col_idx, A.val, A.n_cols)
    b, x = dev(W.uniform(A.n_rows, 5)), torch.empty(A.n_rows, dtype=torch.float64, device="cuda")
    st = np.zeros(4)
    for val in (A.val, val2):
        M.set_values(dev(val))
        for solve in (lambda: _abi.spmv_cg(M.handle, b.data_ptr(), x.data_ptr(), 1e-12, 5000, st.ctypes.data, None),
                      lambda: _abi.spmv_ir_cg(M.handle, b.data_ptr(), x.data_ptr(), 1e-12, 20, 1e-3, 500, st.ctypes.data,
                                              None)):
            torch.cuda.synchronize()
            assert solve() == _abi.SPMV_OK
            r = oracle.residual(A.row_ptr, A.col_idx, val, host(b), host(x))
            assert np.linalg.norm(r) <= 2e-12 * np.linalg.norm(host(b)), (kind, st)
