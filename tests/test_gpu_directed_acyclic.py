"""FP32 propagation of 2,048 source columns and more on directed graphs, where
the solves may start from the walk's dominant mode: graphs without cycles (no
mode: what 40 power steps leave is no eigenvector), chains of classes, periodic
walks, weighted graphs. Every entry lies within the two certificates of the
plain FP64 power iteration, and where there is no mode to use a call takes the
sweeps of one without the analysis (fewer than 2,048 columns)."""
import numpy as np
import pytest

import synth
from test_gpu_directed_modes import from_edges

pytestmark = pytest.mark.gpu
K = 2100      # columns of a call that may use the mode
FEW = 2047    # columns of a call that never does


@pytest.fixture(scope="module")
def ctx():
    import paper_2112_14944_gb300 as P
    c = P.Context(0)
    yield c
    c.close()


def descending(g, seed, weights=None):
    """The edges of an undirected graph, from the later to the earlier node of a random order."""
    order = np.random.default_rng(seed).permutation(g.n)
    src = np.repeat(np.arange(g.n), np.diff(g.row_ptr))
    keep = order[src] > order[g.col]
    rp = np.zeros(g.n + 1, dtype=np.int64)
    np.cumsum(np.bincount(src[keep], minlength=g.n), out=rp[1:])
    w = None
    if weights is not None:
        w = np.exp(np.random.default_rng(weights).normal(size=int(keep.sum()))).astype(np.float32)
    return synth.Graph(g.n, rp, g.col[keep].astype(np.int32), w, directed=True)


def random_dag(n, out, seed):
    rng = np.random.default_rng(seed)
    return from_edges(n, {(i, int(t)) for i in range(n - 1) for t in rng.integers(i + 1, n, out)})


def layered(layers=34, width=120, sinks=20, inside=1, ahead=20, seed=0):
    """Layers of a few edges inside and many to the next one; the last feeds nodes without out-edges."""
    rng = np.random.default_rng(seed)
    edges = set()
    for a in range(layers):
        nxt = width if a + 1 < layers else sinks
        for i in range(width):
            edges |= {(a * width + i, a * width + int(t)) for t in rng.choice(width, inside, replace=False) if t != i}
            edges |= {(a * width + i, (a + 1) * width + int(t)) for t in rng.choice(nxt, min(ahead, nxt), replace=False)}
    return from_edges(layers * width + sinks, edges)


def pairs(seed=4):
    """400 closed 2-cycles (eigenvalues 1 and -1) and nodes that lead into them."""
    rng = np.random.default_rng(seed)
    edges = {(2 * i, 2 * i + 1) for i in range(400)} | {(2 * i + 1, 2 * i) for i in range(400)}
    edges |= {(800 + i, int(t)) for i in range(1400) for t in rng.integers(0, 2200, 4) if t != 800 + i}
    return from_edges(2200, edges)


def weighted():
    g = synth.directed_from(synth.chung_lu(3000, 20, 2.5, seed=1), p_both=0.5, seed=2)
    w = np.exp(np.random.default_rng(4).normal(size=g.nnz)).astype(np.float32)
    return synth.Graph(g.n, g.row_ptr, g.col, w, directed=True)


ACYCLIC = {
    "power_law_10000": lambda: descending(synth.chung_lu(10000, 20, 2.5, seed=0), 0),
    "power_law_10000b": lambda: descending(synth.chung_lu(10000, 20, 2.5, seed=4), 4),
    "power_law_3000": lambda: descending(synth.chung_lu(3000, 20, 2.5, seed=4), 4),
    "power_law_weighted": lambda: descending(synth.chung_lu(10000, 20, 2.5, seed=2), 2, weights=3),
    "random_3000": lambda: random_dag(3000, 8, 1),
    "random_5000": lambda: random_dag(5000, 10, 2),
    "layered": layered,  # (a few edges inside a layer: cycles of one layer only)
}
OTHERS = {
    "cycle": lambda: from_edges(2150, {(i, (i + 1) % 2150) for i in range(2150)}),
    "pairs": pairs,
    "weighted": weighted,
    "power_law": lambda: synth.directed_from(synth.chung_lu(4000, 20, 2.5, seed=1), p_both=0.3, seed=3),
}


def within_certificates(ctx, G, view, alpha, eps, D, cert):
    import paper_2112_14944_gb300 as P
    R, _, c64, st = ctx.dppr(G, view, alpha, 1e-9, P.FP64, out64=True)
    assert st == 0 and np.isfinite(D).all() and cert.max() <= eps
    assert (np.abs(D - R) <= (cert + c64)[:, None] + 2.0 ** -40 * np.abs(R)).all()


def per_group(ctx):
    s = ctx.stats()
    return s["sweeps_main"] / s["groups"], s["refine_passes"] / s["groups"]


@pytest.mark.parametrize("alpha", [0.15, 0.5, 0.03])
@pytest.mark.parametrize("kind", [*ACYCLIC, *OTHERS])
def test_many_columns_within_certificates_of_fp64(ctx, kind, alpha):
    import paper_2112_14944_gb300 as P
    G = ctx.upload_graph({**ACYCLIC, **OTHERS}[kind]())
    view = synth.sample_view(G.n, K, seed=5).astype(np.int32)
    D, _, cert, st = ctx.dppr(G, view, alpha, 1e-6, P.FP32_CSR, out64=True)
    assert st == 0
    within_certificates(ctx, G, view, alpha, 1e-6, D, cert)


@pytest.mark.parametrize("kind,eps", [("random_5000", 1e-8), ("random_3000", 1e-10)])
def test_acyclic_graphs_converge_at_small_eps(ctx, kind, eps):
    import paper_2112_14944_gb300 as P
    G = ctx.upload_graph(ACYCLIC[kind]())
    view = synth.sample_view(G.n, K, seed=6).astype(np.int32)
    D, _, cert, st = ctx.dppr(G, view, 0.15, eps, P.FP32_CSR, out64=True)
    assert st == 0
    within_certificates(ctx, G, view, 0.15, eps, D, cert)


@pytest.mark.parametrize("kind", list(ACYCLIC))
def test_acyclic_graphs_take_the_sweeps_of_the_plain_path(ctx, kind):
    """One refinement pass at most, and the main sweeps of a call without the analysis."""
    import paper_2112_14944_gb300 as P
    G = ctx.upload_graph(ACYCLIC[kind]())
    view = synth.sample_view(G.n, K, seed=7).astype(np.int32)
    ctx.dppr(G, view[:FEW], 0.15, 1e-6, P.FP32_CSR)
    few = per_group(ctx)
    ctx.dppr(G, view, 0.15, 1e-6, P.FP32_CSR)
    many = per_group(ctx)
    assert many[0] == few[0] and many[1] <= max(1.0, few[1])


@pytest.mark.parametrize("kind", ["power_law", "weighted"])
def test_a_true_mode_is_used(ctx, kind):
    """Where the walk mixes well apart from one mode, its solves take less than half the sweeps."""
    import paper_2112_14944_gb300 as P
    G = ctx.upload_graph(OTHERS[kind]())
    view = synth.sample_view(G.n, K, seed=8).astype(np.int32)
    ctx.dppr(G, view[:FEW], 0.15, 1e-6, P.FP32_CSR)
    few = per_group(ctx)
    ctx.dppr(G, view, 0.15, 1e-6, P.FP32_CSR)
    assert per_group(ctx)[0] < 0.5 * few[0]
