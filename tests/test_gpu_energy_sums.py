"""Gradient sums of the stress energy, against the same gradient in more
precision: a row's sum is no further off (root mean square) than plain sums in
the result's own type, with one fused multiply-add per term in 32 interleaved
partial sums, which are then added pairwise. Both have the same terms, so what
is compared is what adding them up loses."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import paper_2112_14944_gb300 as P
    c = P.Context(0)
    yield c
    c.close()


def inputs(k, seed, dtype):
    """Distances spread as a view's PDist, coordinates uniform in [-5, 5]^2."""
    rng = np.random.default_rng(seed)
    r = rng.normal(size=(k, k))
    delta = np.clip(7.0 + 1.5 * (r + r.T) / np.sqrt(2.0), 2.0, 12.0).astype(dtype)
    np.fill_diagonal(delta, 0)
    return delta, rng.uniform(-5.0, 5.0, (k, 2)).astype(dtype)


def terms(delta, x, i, t):
    """Coefficients and coordinate differences of row i in type t (0 for i itself)."""
    u = x[i].astype(t) - x.astype(t)
    d = np.sqrt((u * u).sum(1))
    d[i] = 1
    w = delta[i].astype(t)
    w[i] = 1
    c = t(-2) * (t(1) - d * (t(1) / w)) * (t(1) / w) / d
    c[i] = 0
    return c, u


def gradient(delta, x, wide):
    g = np.zeros((len(x), 2), wide)
    for i in range(len(x)):
        c, u = terms(delta, x, i, wide)
        g[i] = (c[:, None] * u).sum(0)
    return g


def plain_gradient(delta, x, wide):
    k, t = len(x), delta.dtype.type
    g = np.zeros((k, 2), t)
    for i in range(k):
        c, u = terms(delta, x, i, t)
        pad = -k % 32
        c, u = np.pad(c, (0, pad)).reshape(-1, 32), np.pad(u, ((0, pad), (0, 0))).reshape(-1, 32, 2)
        acc = np.zeros((32, 2), t)
        for q in range(len(c)):  # one rounding per term
            acc = (acc.astype(wide) + c[q][:, None].astype(wide) * u[q].astype(wide)).astype(t)
        while len(acc) > 1:
            acc = acc[: len(acc) // 2] + acc[len(acc) // 2:]
        g[i] = acc[0]
    return g


@pytest.mark.parametrize("k,dtype,seeds", [(200, np.float32, 8), (255, np.float32, 8), (1000, np.float32, 3),
                                           (2500, np.float32, 1), (200, np.float64, 8), (600, np.float64, 2)])
def test_gradient_sums_lose_no_more_than_plain_sums(ctx, k, dtype, seeds):
    wide = np.float64 if dtype == np.float32 else np.longdouble
    if np.finfo(wide).eps > 2.0 ** -10 * np.finfo(dtype).eps:
        pytest.skip("no wider type here")
    err = plain = 0.0
    for seed in range(seeds):
        delta, x = inputs(k, seed, dtype)
        _, gx, _ = ctx.energy(delta, x, grad_x=True)
        g = gradient(delta, x, wide)
        err += float(((gx.astype(wide) - g) ** 2).sum())
        plain += float(((plain_gradient(delta, x, wide).astype(wide) - g) ** 2).sum())
    assert err <= plain, (np.sqrt(err), np.sqrt(plain))
