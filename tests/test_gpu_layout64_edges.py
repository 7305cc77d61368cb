"""The FP64 layout (inverse by 64-blocks, 64 x 64 pass tiles) at the edges of
its tiles against numpy: one and a few updates of Eq. (10) from the same X."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import paper_2112_14944_gb300 as P
    c = P.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("iters", [1, 3])
@pytest.mark.parametrize("k", [1, 2, 3, 63, 64, 65, 127, 129, 192, 321])
def test_fp64_layout_updates(ctx, k, iters):
    """Forward error of an update: the solve's ~ k cond(A) 2^-53 of the layout's
    size, the pass's a few roundings per pair; a later update carries the error
    of the one before by at most cond(A)."""
    import paper_2112_14944_gb300 as P
    rng = np.random.default_rng(k)
    delta = rng.uniform(2.0, 14.0, (k, k))
    delta = (delta + delta.T) / 2
    np.fill_diagonal(delta, 0.0)
    x0 = rng.uniform(-1.0, 1.0, (k, 2))
    if k > 3:
        x0[1] = x0[0]           # coincident points: their term is 0
        x0[2] = x0[0] + 1e-160  # a distance whose square is not a normal number
    x, _ = ctx.layout(delta, x0, iters, precision=P.FP64)
    w = np.zeros((k, k))
    off = ~np.eye(k, dtype=bool)
    w[off] = 1.0 / delta[off]
    a = 1.0 / k - w * w
    a[~off] = (w * w).sum(1) + 1.0 / k
    cond = np.linalg.cond(a)
    y = x0.copy()
    for _ in range(iters):
        df = y[:, None, :] - y[None, :, :]
        d = np.hypot(df[..., 0], df[..., 1])
        c = np.divide(w, d, out=np.zeros_like(w), where=d > 0)
        b = (c[..., None] * df).sum(1)
        y = np.linalg.solve(a, b)
    y -= y.mean(0)
    tol = 64 * k * 2.0 ** -53 * cond ** iters * max(1.0, np.abs(y).max())
    assert np.abs(x - y).max() <= tol
