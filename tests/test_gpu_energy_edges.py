"""The energy pass at the sizes where its row groups, column chunks and block
loop end, and on values outside the range of its fast formulas, against the
same formulas in FP64."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

U = 2.0 ** -24  # rounding unit of float


@pytest.fixture(scope="module")
def ctx():
    import paper_2112_14944_gb300 as P
    c = P.Context(0)
    yield c
    c.close()


def reference(delta, x):
    """(E, grad_x, grad_pdist, first-order error scales of the two gradients), FP64."""
    delta, x = delta.astype(np.float64), x.astype(np.float64)
    k = len(x)
    gx, sx = np.zeros((k, 2)), np.zeros((k, 1))
    gd, sd = np.zeros((k, k)), np.zeros((k, k))
    e_sum = 0.0
    for i in range(k):
        dx = x[i] - x
        d = np.sqrt((dx * dx).sum(1))
        u = np.zeros(k)
        off = np.arange(k) != i
        u[off] = 1.0 / delta[i, off]
        e = np.where(off, 1.0 - d * u, 0.0)
        e_sum += (e * e).sum()
        c = np.divide(-2.0 * e * u, d, out=np.zeros(k), where=d > 0)
        gx[i] = (c[:, None] * dx).sum(0)
        sx[i] = (2.0 * (1.0 + d * u) * u).sum()
        gd[i] = e * d * u * u
        sd[i] = (1.0 + d * u) * d * u * u
    return 0.5 * e_sum, gx, gd, sx, sd


@pytest.mark.parametrize("special", [False, True])
@pytest.mark.parametrize("k", [1, 2, 3, 4, 5, 255, 257, 1026, 2433, 2436])
def test_energy_row_groups_and_ranges(ctx, k, special):
    """Each term has fewer than 16 roundings of values bounded by its scale
    ((1 - d u) counted as 1 + d u), a row sum at most 8 + k / 256 more per
    thread and 16 across threads; the energy's terms (1 - d u)^2 err by at most
    16 U (1 + d u)^2 each and their sum is exact beside that."""
    rng = np.random.default_rng(k)
    delta = rng.uniform(2.0, 18.0, (k, k)).astype(np.float32)  # not symmetric
    x = rng.uniform(-6.0, 6.0, (k, 2)).astype(np.float32)
    if special and k > 3:
        x[1] = x[0]                      # coincident
        x[2] = x[0] + np.float32(1e-6)   # a few ulps apart
        x[3] = (1e-16, 0.0)
        x[k // 2] = (0.0, 0.0) if k > 8 else x[k // 2]
        delta[0, k - 1] = 1e-8           # outside the fast range
        delta[k - 1, 0] = 1e20
    np.fill_diagonal(delta, 0.0)
    e, gx, gd = ctx.energy(delta, x, grad_scale=1.0, grad_x=True, grad_pdist=True)
    e_ref, gx_ref, gd_ref, sx, sd = reference(delta, x)
    scale = 0.0
    for i in range(k):
        d = np.sqrt(((x[i].astype(np.float64) - x) ** 2).sum(1))
        off = np.arange(k) != i
        scale += ((1.0 + d[off] / delta[i, off].astype(np.float64)) ** 2).sum()
    assert abs(e - e_ref) <= 0.5 * 32 * U * scale
    assert (np.abs(gd - gd_ref) <= 16 * U * sd + 1e-37).all()
    assert (np.abs(gx - gx_ref) <= (40 + math.ceil(k / 256)) * U * sx).all()
    # without gradients: the same pairs in the same order
    assert ctx.energy(delta, x)[0] == e


def test_infinite_distance_and_refusals(ctx):
    """An infinite target distance stays accepted (u = 0: the pair's e is 1); zero, negative and NaN stay refused."""
    import paper_2112_14944_gb300 as P
    rng = np.random.default_rng(7)
    delta = rng.uniform(2.0, 9.0, (9, 9)).astype(np.float32)
    x = rng.uniform(-3.0, 3.0, (9, 2)).astype(np.float32)
    delta[4, 5] = np.inf
    e, _, gd = ctx.energy(delta, x, grad_pdist=True)
    e_ref, _, gd_ref, _, sd = reference(delta, x)
    assert abs(e - e_ref) <= 1e-5 * e_ref and gd[4, 5] == 0.0
    for bad in (0.0, -1.0, np.nan):
        worse = delta.copy()
        worse[8, 0] = bad
        with pytest.raises(P.PPRVizError):
            ctx.energy(worse, x)
