"""A plan that spmv_set_plan refuses changes nothing: the plan reported, the bits of a
product and of a solve, and the kernels behind them stay those of before."""
import pytest

from paper_1106_5908_gb300 import workloads as W
from gpu_util import dev, host, need_gpu

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

REFUSED = [(-1, 0), (7, 0), (0, 9), (0, -7), (1, 3), (1, 64), (2, 4), (2, 33), (3, 9), (4, 8), (4, -9), (5, 48), (5, 16),
           (5, 1 << 21), (6, 11), (6, 15)]


@pytest.fixture(autouse=True)
def _gpu():
    need_gpu()


def _refuse_all(M, plans=REFUSED):
    from paper_1106_5908_gb300 import _abi
    before = M.info()
    for family, param in plans:
        assert _abi.spmv_set_plan(M.handle, family, param) == _abi.SPMV_ERR_INVALID_ARG, (family, param)
    assert M.info() == before


def test_solver_keeps_its_kernel():
    from paper_1106_5908_gb300 import Matrix, cg
    A = W.laplace2d(96)
    b = dev(W.uniform(A.n_rows, 5))
    M, N = (Matrix.from_csr(A.row_ptr, A.col_idx, A.val, A.n_cols) for _ in range(2))
    _refuse_all(N)
    (x, st), (y, su) = cg(M, b), cg(N, b)
    assert st["inner"] == su["inner"] and torch.equal(x, y)


def test_symmetric_keeps_the_expanded_product():
    from paper_1106_5908_gb300 import Matrix
    U = W.upper_triangle(W.hamiltonian_like(20000, seed=4))
    x = dev(W.uniform(U.n_rows, 5))
    M, N = (Matrix.from_symmetric_upper(U.row_ptr, U.col_idx, U.val) for _ in range(2))
    _refuse_all(N)
    assert torch.equal(M.apply(x), N.apply(x))
    N.set_plan(4, 9)
    assert not torch.equal(M.apply(x), N.apply(x))  # the two passes round otherwise


@pytest.mark.parametrize("dtype,plans", [("f64", [(0, 0), (0, 7), (1, 4), (2, 0), (3, 0), (4, 0), (5, 0), (5, 64), (6, 0), (6, 7)]),
                                         ("f32", [(0, 15), (4, 0), (5, 1 << 20), (6, 0), (6, 15)])])
def test_accepted_plans_are_reported(dtype, plans):
    from paper_1106_5908_gb300 import Matrix
    A = W.hamiltonian_like(5000, seed=4)
    val = A.val if dtype == "f64" else A.val.astype("float32")
    M = Matrix.from_csr(A.row_ptr, A.col_idx, val, A.n_cols)
    default = {0: 16, 2: 15, 3: 7, 4: 9 if dtype == "f64" else 15, 5: 4096, 6: 9}
    for family, param in plans:
        M.set_plan(family, param)
        info = M.info()
        assert info["family"] == family
        if family == 1:
            assert info["T"] == param
        else:
            assert info["E"] == (param or default[family])
        _refuse_all(M, [p for p in REFUSED if dtype == "f64" or p != (6, 15)])
