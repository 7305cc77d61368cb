"""Source groups of 32 and 64 columns (few sources, or a state beyond L2)
against the 128-wide groups of an all-nodes call: every DPPR entry of the two
lies within the sum of its certificates, on hub rows split into segments,
isolated nodes, weights and directed graphs."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

ALPHA = 0.15


@pytest.fixture(scope="module")
def ctx():
    import paper_2112_14944_gb300 as P
    c = P.Context(0)
    yield c
    c.close()


def graph(kind):
    if kind == "hubs":
        return synth.chung_lu(901, 12, 2.2, seed=3)  # rows of more than 64 edges, some isolated nodes
    if kind == "weighted":
        return synth.dense_clustered(300, blocks=4, density=0.04, seed=2)
    return synth.directed_from(synth.chung_lu(901, 12, 2.2, seed=3), seed=5)


_wide = {}


def wide(ctx, kind, eps):
    """(uploaded graph, DPPR of all nodes, certificates) with 128-wide groups."""
    import paper_2112_14944_gb300 as P
    if (kind, eps) not in _wide:
        G = ctx.upload_graph(graph(kind))
        view = np.arange(G.n, dtype=np.int32)
        D, _, cert, st = ctx.dppr(G, view, ALPHA, eps, P.FP32_CSR, out64=True)
        assert st == 0 and ctx.stats()["source_group"] >= 128
        _wide[kind, eps] = G, D, cert
    return _wide[kind, eps]


@pytest.mark.parametrize("eps", [1e-6, 1e-10])
@pytest.mark.parametrize("k", [1, 31, 32, 33, 64, 65])
@pytest.mark.parametrize("kind", ["hubs", "weighted", "directed"])
def test_narrow_groups_match_wide(ctx, kind, k, eps):
    import paper_2112_14944_gb300 as P
    G, D, cert = wide(ctx, kind, eps)
    view = synth.sample_view(G.n, k, seed=k)
    Dn, _, cn, st = ctx.dppr(G, view, ALPHA, eps, P.FP32_CSR, out64=True)
    assert st == 0 and cn.max() <= eps
    assert ctx.stats()["source_group"] == (32 if k <= 32 else 64 if k <= 64 else 128)
    ref = D[np.ix_(view, view)]
    # the outputs are float-float products rounded below 2^-40 of an entry
    assert (np.abs(Dn - ref) <= (cn + cert[view])[:, None] + 2.0 ** -40 * np.abs(ref)).all()


@pytest.mark.parametrize("children", [1, 32, 40, 64, 70])
@pytest.mark.parametrize("kind", ["hubs", "directed"])
def test_narrow_level_groups(ctx, kind, children):
    """Level-l DPPR of leaf sets of uneven size: averages of the node rows (Eq. (2))."""
    G, D, cert = wide(ctx, kind, 1e-10)
    sizes = 1 + np.arange(children) % 5
    ptr, idx = synth.random_leaf_sets(G.n, sizes, seed=children)
    sets = [idx[ptr[i]:ptr[i + 1]] for i in range(children)]
    L, _, cl, st = ctx.level_dppr(G, sets, ALPHA, 1e-6, out64=True)
    assert st == 0
    ref = np.array([[D[np.ix_(a, b)].sum() / (len(a) * len(b)) for b in sets] for a in sets])
    miss = np.array([cert[a].mean() for a in sets])
    assert (np.abs(L - ref) <= (cl + miss)[:, None] + 1e-12 * np.abs(ref)).all()


def test_tau_push_checks_its_inputs_on_the_device(ctx):
    """Bad DPR entries at either end are refused for host and device arrays, -0.0 is
    accepted, and repeated leaves are refused for few leaves and for many."""
    import paper_2112_14944_gb300 as P
    import torch
    g = synth.chung_lu(901, 12, 2.2, seed=3)
    G = ctx.upload_graph(g)
    dpr, _ = ctx.dpr(G)
    ptr, idx = synth.random_leaf_sets(g.n, [3, 2, 4], seed=1)
    ok, _, _ = ctx.tau_push(G, ptr, idx, dpr)
    zero = dpr.copy()
    zero[-1] = -0.0 if zero[-1] == 0.0 else zero[-1]
    assert np.allclose(ctx.tau_push(G, ptr, idx, zero)[0], ok, rtol=1e-12, atol=0)
    for at, value in ((0, -1e-300), (g.n - 1, np.nan), (450, np.inf), (7, -np.inf)):
        bad = dpr.copy()
        bad[at] = value
        with pytest.raises(P.PPRVizError):
            ctx.tau_push(G, ptr, idx, bad)
        out = torch.empty(3, 3, dtype=torch.float64, device="cuda")
        dev = [torch.from_numpy(a).cuda() for a in (ptr, idx, bad)]
        with pytest.raises(P.PPRVizError):
            ctx.tau_push(G, *dev, ldppr_out=out, want_pdist=False)
    for many in (False, True):
        ptr, idx = synth.random_leaf_sets(g.n, [40, 40] if many else [2, 2], seed=2)
        idx[-1] = idx[0]
        with pytest.raises(P.PPRVizError):
            ctx.tau_push(G, ptr, idx, dpr)


def resident_graph(kind, n):
    if kind == "hubs":  # rows split into segments
        return synth.chung_lu(n, 10, 2.2, seed=1)
    if kind == "weighted":
        return synth.dense_clustered(n, blocks=4, density=12.0 / n, seed=2)
    i = np.arange(n, dtype=np.int64)  # a cycle: no split
    col = np.sort(np.stack([(i - 1) % n, (i + 1) % n], 1), axis=1).astype(np.int32)
    return synth.Graph(n, 2 * np.arange(n + 1, dtype=np.int64), col.ravel())


@pytest.mark.parametrize("n", [40, 129, 4863, 4864, 4865, 5003])
@pytest.mark.parametrize("kind", ["hubs", "flat", "weighted"])
def test_sweeps_around_one_resident_grid(ctx, kind, n):
    """Sweeps whose blocks are all resident at once (152 x 1,024 threads: 4,864 rows of
    one 128-wide group) are launched as dependents of the one before, larger ones plainly:
    the FP32 and FP64 solves agree within their certificates on both sides."""
    import paper_2112_14944_gb300 as P
    G = ctx.upload_graph(resident_graph(kind, n))
    view = synth.sample_view(n, min(n, 128), seed=n)
    D, _, c32, s32 = ctx.dppr(G, view, ALPHA, 1e-8, P.FP32_CSR, out64=True)
    R, _, c64, s64 = ctx.dppr(G, view, ALPHA, 1e-11, P.FP64, out64=True)
    assert s32 == 0 and s64 == 0
    assert (np.abs(D - R) <= (c32 + c64)[:, None] + 2.0 ** -40 * np.abs(R)).all()


@pytest.mark.parametrize("n", [8, 102, 103, 512, 513])
def test_analysis_of_small_graphs_in_one_launch(ctx, n):
    """Complete graphs on either side of 16 n + edges = 12,000 and cycles around 512
    nodes: the deflated sweeps converge from either analysis."""
    import paper_2112_14944_gb300 as P
    if n < 512:
        col = np.array([[j for j in range(n) if j != i] for i in range(n)], dtype=np.int32).ravel()
        g = synth.Graph(n, (n - 1) * np.arange(n + 1, dtype=np.int64), col)
    else:
        g = resident_graph("flat", n)
    G = ctx.upload_graph(g)
    view = np.arange(n, dtype=np.int32)
    D, _, c32, s32 = ctx.dppr(G, view, ALPHA, 1e-8, P.FP32_CSR, out64=True)
    R, _, c64, s64 = ctx.dppr(G, view, ALPHA, 1e-11, P.FP64, out64=True)
    assert s32 == 0 and s64 == 0
    assert (np.abs(D - R) <= (c32 + c64)[:, None] + 2.0 ** -40 * np.abs(R)).all()
