"""Certificates at the floor of the compensated FP32 residual. A hub of several
thousand edges holds about half of every walk, so what its row sum loses is what
the certificate cannot go below: kept to ~2^-48 of the row, the hub's own DPPR
(d / alpha times as large) is certified to 1e-9, the smallest eps of that path."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import paper_2112_14944_gb300 as P
    c = P.Context(0)
    yield c
    c.close()


def hub(leaves, chords, seed=0):
    """Node 0 joined to all others, and random edges among those."""
    rng = np.random.default_rng(seed)
    e = rng.integers(1, leaves + 1, (chords, 2))
    e = e[e[:, 0] != e[:, 1]]
    u = np.concatenate([np.zeros(leaves, np.int64), e.min(1)])
    v = np.concatenate([np.arange(1, leaves + 1), e.max(1)])
    key = np.unique(u * (leaves + 1) + v)
    u, v = key // (leaves + 1), key % (leaves + 1)
    s, d = np.concatenate([u, v]), np.concatenate([v, u])
    order = np.lexsort((d, s))
    rp = np.zeros(leaves + 2, dtype=np.int64)
    np.cumsum(np.bincount(s, minlength=leaves + 1), out=rp[1:])
    return synth.Graph(leaves + 1, rp, d[order].astype(np.int32))


@pytest.mark.parametrize("k", [20, 50, 200])  # 32-, 64- and 128-wide groups
@pytest.mark.parametrize("leaves,chords,bits", [(3000, 3000, 48), (9000, 2000, None)])
def test_a_hubs_row_is_certified_to_the_smallest_eps(ctx, leaves, chords, bits, k):
    import paper_2112_14944_gb300 as P
    G = ctx.upload_graph(hub(leaves, chords))
    view = np.arange(k, dtype=np.int32)
    _, _, cert, st = ctx.dppr(G, view, 0.15, 1e-9, P.FP32_CSR, out64=True)
    assert st == 0 and cert.max() <= 1e-9
    if bits is not None:  # d / alpha times 2^-bits of the walk's mass
        assert cert[0] <= leaves / 0.15 * 2.0 ** -bits
