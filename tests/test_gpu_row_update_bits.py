"""FP32 rows, y = alpha*A*x + beta*y with all 53 bits of alpha and beta: terms that cancel
to 2^-24 of themselves show every bit below, where FP64 arithmetic keeps 2^-53 of the
terms and the store half an ulp of the result."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("plan", [(4, 7), (4, 9), (4, 11), (4, 15), (5, 4096), (0, 0)])
@pytest.mark.parametrize("alpha,beta", [(1 / 3, -0.7), (-np.pi, np.e), (1e5 / 7, 1e-3 / 11), (2.0 ** -19 / 3, -1.0), (-1.0, 1.0),
                                        (1 / 3, 0.0)])
@pytest.mark.parametrize("entries", [1, 2])
def test_cancelling_terms(plan, alpha, beta, entries):
    from paper_1106_5908_gb300 import Matrix

    n = 17000
    rng = np.random.default_rng(7)
    # one entry per row with an exact product, or two that leave an exact sum of 2 x 22 bits
    v = rng.integers(1, 2048, (n, entries)).astype(np.float64)
    x = rng.integers(1, 2048, n) * 2.0 ** rng.integers(-30, 30)
    if entries == 2:
        v[:, 1] *= 2.0 ** -22
        x = rng.integers(1, 2048, n) * 2.0
    col = np.stack([rng.permutation(n)] * entries, 1)
    ax = (v * x[col]).sum(1)  # 46 bits at most
    y = (-(alpha / beta) * ax if beta else rng.uniform(-1, 1, n)).astype(np.float32)
    y[::5] = (y * (1.0 + rng.integers(-3, 4, n) * 2.0 ** -20))[::5].astype(np.float32)
    t = np.longdouble(alpha) * ax.astype(np.longdouble)
    u = np.longdouble(beta) * y.astype(np.longdouble)
    want = t + u
    # FP64: one rounding of beta*y and one of the sum; the store: half an ulp.  Runs of
    # FP32 round a row sum of more than 24 bits themselves.
    exact_sum = entries == 1 or plan in ((4, 15),)
    tol = np.abs(want) * 2.0 ** -24 * (1 + 2.0 ** -20) + (np.abs(t) + np.abs(u)) * (2.0 ** -52 if exact_sum else 2.0 ** -22)
    assert entries == 2 or beta == 0 or np.median(np.abs(want) / np.abs(t)) < 2.0 ** -20  # they do cancel
    rp = np.arange(0, n * entries + 1, entries, dtype=np.int32)
    A = Matrix.from_csr(*(torch.from_numpy(a).cuda() for a in (rp, col.ravel().astype(np.int32), v.ravel().astype(np.float32))), n)
    if plan != (0, 0):
        A.set_plan(*plan)
    yd = torch.from_numpy(y).cuda()
    A.apply(torch.from_numpy(x.astype(np.float32)).cuda(), yd, alpha=alpha, beta=beta)
    got = yd.cpu().numpy().astype(np.longdouble)
    bad = np.abs(got - want) > tol
    assert not bad.any(), (bad.sum(), np.flatnonzero(bad)[:5], got[bad][:5], want[bad][:5])
    A.close()
