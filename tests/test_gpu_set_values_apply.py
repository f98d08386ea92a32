"""New values and the product in one pass: the same bits as one after the other, and
the copies that follow (CRS, slices, reverse pass) hold the new values."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _stencil(shape, offsets):
    """CRS of a grid stencil with the offsets that stay inside the grid."""
    idx = np.arange(np.prod(shape)).reshape(shape)
    rows, cols = [], []
    for o in offsets:
        src = tuple(slice(max(0, -d), n - max(0, d)) for d, n in zip(o, shape))
        dst = tuple(slice(max(0, d), n - max(0, -d)) for d, n in zip(o, shape))
        rows.append(idx[src].ravel())
        cols.append(idx[dst].ravel())
    rows, cols = np.concatenate(rows), np.concatenate(cols)
    order = np.lexsort((cols, rows))
    rp = np.concatenate([[0], np.cumsum(np.bincount(rows, minlength=idx.size))]).astype(np.int32)
    return rp, cols[order].astype(np.int32), idx.size


def _grid3(reach):
    return [(a, b, c) for a in (-1, 0, 1) for b in (-1, 0, 1) for c in (-1, 0, 1) if abs(a) + abs(b) + abs(c) <= reach]


CASES = {
    "5-point": ((131, 133), [(0, 0), (0, 1), (0, -1), (1, 0), (-1, 0)]),
    "7-point": ((27, 26, 29), _grid3(1)),
    "27-point": ((26, 27, 28), _grid3(3)),
    "line": ((20001,), [(0,), (1,)]),
}


@pytest.mark.parametrize("name", CASES)
@pytest.mark.parametrize("vt,st,xt", [("f64", "f64", "f64"), ("f32", "f32", "f32"), ("f32", "f64", "f32"),
                                      ("f64", "f32", "f64")])
def test_same_as_two_calls(name, vt, st, xt):
    from paper_1106_5908_gb300 import Matrix

    dt = dict(f64=torch.float64, f32=torch.float32)
    rp, col, n = _stencil(*CASES[name])
    g = torch.Generator().manual_seed(3)
    val = (torch.rand(len(col), generator=g, dtype=torch.float64) - 0.5).cuda()
    x = (torch.rand(n, generator=g, dtype=torch.float64) - 0.5).to(dt[xt]).cuda()
    x[::977] *= 2.0 ** -126  # FP32: sums outside the range of float pairs
    rpd, cold = (torch.from_numpy(a).cuda() for a in (rp, col))
    A, B = (Matrix.from_csr(rpd, cold, val.to(dt[vt]), n) for _ in range(2))
    for step, alpha in enumerate((1.0, -0.75, 1.0, 2.0)):
        new = (val * (step + 0.3)).to(dt[st])
        new[:: 131] *= 2.0 ** -120
        y = A.set_values_apply(new, x, alpha)
        B.set_values(new)
        assert torch.equal(y, B.apply(x, alpha=alpha))
        assert torch.equal(A.apply(x), B.apply(x))
        if step:
            for a, b in zip(A.backward(x, x), B.backward(x, x)):
                assert torch.equal(a, b)
        A.set_plan(4, 7), B.set_plan(4, 7)  # from the CRS copy
        assert torch.equal(A.apply(x), B.apply(x))
        A.set_plan(5, 4096), B.set_plan(5, 4096)
    A.close(), B.close()
