"""alpha and beta of Matrix.apply: anything float() takes."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("make", [float, int, np.float32, np.int64, torch.tensor])
def test_apply_scalars(make):
    from paper_1106_5908_gb300 import Matrix

    rp, col = (torch.tensor(a, dtype=torch.int32, device="cuda") for a in ([0, 1, 2], [1, 0]))
    A = Matrix.from_csr(rp, col, torch.tensor([3.0, 5.0], dtype=torch.float64, device="cuda"), 2)
    x = torch.tensor([1.0, 2.0], dtype=torch.float64, device="cuda")
    y = torch.tensor([10.0, 20.0], dtype=torch.float64, device="cuda")
    A.apply(x, y, alpha=make(2), beta=make(3))
    assert y.tolist() == [42.0, 70.0]
    A.close()
