"""FP32 batch members on diagonal slices are no less exact than in chunks: the rounding
error of a batch against that of the same matrices on the slot-major kernel, whose lanes
sum up to 9 entries of a row in a run, as in a batch's chunks.  The norm over 400,000 rows
of independent rounding errors varies by 0.2 %."""
import numpy as np
import pytest

from gpu_util import need_gpu

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("offsets", [(-1, 0, 1), (-600, -1, 0, 1, 600), (-900, -30, -1, 0, 1, 30, 900),
                                     (-4, -3, -2, -1, 0, 1, 2, 3, 4), tuple(range(-5, 6))])
def test_no_less_exact_than_chunks(offsets):
    from paper_1106_5908_gb300 import Batch, Matrix
    need_gpu()
    n, members = 40000, 10
    rng = np.random.default_rng(len(offsets))
    i = np.arange(n)[:, None] + np.array(offsets)[None, :]
    ok = (i >= 0) & (i < n)
    rp = np.concatenate([[0], np.cumsum(ok.sum(1))]).astype(np.int32)
    col = i[ok].astype(np.int32)
    mats, xs, want, err = [], [], [], {"batch": 0.0, "chunks": 0.0}
    for _ in range(members):
        val, x = rng.standard_normal(col.size).astype(np.float32), rng.uniform(-1, 1, n).astype(np.float32)
        M = Matrix.from_csr(rp, col, val, n)
        mats.append(M)
        xs.append(torch.from_numpy(x).cuda())
        want.append(np.add.reduceat(val.astype(np.float64) * x[col].astype(np.float64), rp[:-1]))
    ys = [torch.empty_like(x) for x in xs]
    B = Batch(mats)
    assert set(B.info()["member_E"]) == {0}  # on the slices
    B.apply(xs, ys)
    for M, x, y, w in zip(mats, xs, ys, want):
        M.set_plan(4, 9)
        for name, got in (("batch", y), ("chunks", M.apply(x))):
            err[name] += float(((got.cpu().numpy().astype(np.float64) - w) ** 2).sum())
    assert err["batch"] <= err["chunks"] * 1.02 ** 2, {k: np.sqrt(v) for k, v in err.items()}
