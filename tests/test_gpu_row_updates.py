"""y = alpha*A*x + beta*y.  FP64: each form of the update (plain, scaled, added,
subtracted, general) over chunk and slice edges, exact on small whole numbers.

FP32: the update runs in pairs of floats inside its range and in FP64 outside it.  One entry per row with an exact product, so the row
sum is exact and only the update rounds: half an ulp of the result, plus what 48-bit
alpha and beta and the dropped low products leave out (below 2^-44 of the terms)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("plan", [(4, 7), (4, 11), (4, 15), (5, 4096), (0, 0)])
@pytest.mark.parametrize("alpha,beta", [(-0.75, 0.5), (-1.0, 1.0), (1.0, 1.0), (1 / 3, 0.0), (1 / 3, -1.7),
                                        (0.0, 0.5), (2.0 ** 21, 1.0), (1e-9, 3.0), (-0.0, 1.0), (0.7, -0.0)])
def test_update_rounds_once(plan, alpha, beta):
    from paper_1106_5908_gb300 import Matrix

    n = 17000
    rng = np.random.default_rng(5)
    v = rng.integers(1, 2048, n).astype(np.float64) * rng.choice([-1.0, 1.0], n)
    x = rng.integers(1, 2048, n) * 2.0 ** rng.integers(-80, 60, n)
    y = rng.uniform(-1.0, 1.0, n) * 2.0 ** rng.integers(-80, 60, n)
    near = rng.random(n) < 0.5  # terms of like size, many of them nearly cancelling
    y[near] = -(v * x)[near] * (1.0 + rng.integers(-3, 4, near.sum()) * 2.0 ** -20)
    y[:: 7] = 0.0
    x[:: 11] = 0.0
    v, x, y = (a.astype(np.float32) for a in (v, x, y))
    rp = np.arange(n + 1, dtype=np.int32)
    col = rng.permutation(n).astype(np.int32)
    with np.errstate(over="ignore", invalid="ignore"):
        t = np.longdouble(alpha) * (v.astype(np.longdouble) * x[col].astype(np.longdouble))
        u = np.longdouble(beta) * y.astype(np.longdouble)
    want = t + u
    tol = np.abs(want) * 2.0 ** -24 * (1 + 2.0 ** -20) + (np.abs(t) + np.abs(u)) * 2.0 ** -44 + 2.0 ** -149
    A = Matrix.from_csr(*(torch.from_numpy(a).cuda() for a in (rp, col, v)), n)
    if plan != (0, 0):
        A.set_plan(*plan)
    yd = torch.from_numpy(y).cuda()
    A.apply(torch.from_numpy(x).cuda(), yd, alpha=alpha, beta=beta)
    got = yd.cpu().numpy().astype(np.longdouble)
    bad = np.abs(got - want) > tol
    assert not bad.any(), (np.flatnonzero(bad)[:5], got[bad][:5], want[bad][:5])
    A.close()


@pytest.mark.parametrize("plan", [(4, 7), (4, 9), (4, 11), (4, 15), (5, 4096), (0, 0)])
@pytest.mark.parametrize("n", [1, 33, 1000, 20011])
def test_fp64_forms_exact(plan, n):
    from paper_1106_5908_gb300 import Matrix

    rng = np.random.default_rng(n)
    width = rng.choice([0, 1, 2, 5, 30, 70], n, p=[0.1, 0.3, 0.2, 0.3, 0.08, 0.02])
    rp = np.concatenate([[0], np.cumsum(width)]).astype(np.int32)
    col = rng.integers(0, n, rp[-1]).astype(np.int32)
    val = rng.integers(-8, 9, rp[-1]).astype(np.float64)
    x = rng.integers(-8, 9, n).astype(np.float64)
    y = rng.integers(-8, 9, n).astype(np.float64)
    ax = np.zeros(n)
    np.add.at(ax, np.repeat(np.arange(n), width), val * x[col])
    A = Matrix.from_csr(*(torch.from_numpy(a).cuda() for a in (rp, col, val)), n)
    if plan != (0, 0):
        A.set_plan(*plan)
    for alpha, beta in ((1.0, 0.0), (-0.75, 0.0), (1.0, 1.0), (-1.0, 1.0), (-0.75, 0.5), (0.0, 2.0)):
        yd = torch.from_numpy(y).cuda() if beta else torch.full((n,), float("nan"), dtype=torch.float64).cuda()
        A.apply(torch.from_numpy(x).cuda(), yd, alpha=alpha, beta=beta)
        want = alpha * ax + (beta * y if beta else 0.0)
        assert np.array_equal(yd.cpu().numpy(), want), (alpha, beta)
    A.close()
