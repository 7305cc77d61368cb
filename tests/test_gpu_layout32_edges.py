"""The FP32 layout (inverse by 128-blocks) at the edges of its blocks against
numpy in FP64: one update of Eq. (10)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import paper_2112_14944_gb300 as P
    c = P.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("k", [1, 2, 5, 127, 128, 129, 255, 257, 384, 513, 608, 609, 1217, 1999, 2048, 2049])
def test_fp32_layout_update(ctx, k):
    """Views that stay in the shared memories (up to about 2,000 nodes: 4, 8 and
    16 rows per block) and one beyond. Forward error of one update: 1/Delta and the squares are rounded once, the
    inverse errs by a small multiple of 2^-22 cond(A) (3xTF32 products) and the
    passes by a few float roundings of sums of k terms."""
    rng = np.random.default_rng(k)
    delta = rng.uniform(2.0, 14.0, (k, k)).astype(np.float32)
    delta = np.triu(delta, 1)
    delta = delta + delta.T
    x0 = rng.uniform(-1.0, 1.0, (k, 2)).astype(np.float32)
    x, _ = ctx.layout(delta, x0, 1)
    w = np.zeros((k, k))
    off = ~np.eye(k, dtype=bool)
    w[off] = 1.0 / delta[off].astype(np.float64)
    a = 1.0 / k - w * w
    a[~off] = (w * w).sum(1) + 1.0 / k
    df = x0[:, None, :].astype(np.float64) - x0[None, :, :].astype(np.float64)
    d = np.hypot(df[..., 0], df[..., 1])
    c = np.divide(w, d, out=np.zeros_like(w), where=d > 0)
    b = (c[..., None] * df).sum(1)
    y = np.linalg.solve(a, b)
    y -= y.mean(0)
    # |M| |c| bounds the sums that the passes round
    ev = np.linalg.eigvalsh(a)
    cond = ev[-1] / ev[0]
    size = np.abs(np.linalg.inv(a)) @ np.abs(c[..., None] * df).sum(1)
    tol = 2.0 ** -22 * (8.0 * cond * np.abs(y).max() + 4.0 * size.max())
    assert np.abs(x - y).max() <= tol
