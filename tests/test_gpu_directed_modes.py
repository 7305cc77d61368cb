"""FP32 propagation on directed graphs whose walks stress the deflated power
sweeps (no dominant mode, several, modes of modulus 1, dangling nodes
everywhere) against the plain FP64 power iteration: every DPPR entry lies
within the sum of the two certificates."""
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


def from_edges(n, edges, weights=None):
    e = np.array(sorted(edges), dtype=np.int64).reshape(-1, 2)
    rp = np.zeros(n + 1, dtype=np.int64)
    np.cumsum(np.bincount(e[:, 0], minlength=n), out=rp[1:])
    w = None if weights is None else np.asarray(weights, dtype=np.float32)[: len(e)]
    return synth.Graph(n, rp, e[:, 1].astype(np.int32), w, directed=True)


def graph(kind):
    rng = np.random.default_rng(4)
    if kind == "dag":          # nilpotent: no dominant mode
        return from_edges(200, {(i, j) for i in range(200) for j in rng.integers(i + 1, 201, 4) if j < 200})
    if kind == "cycle":        # every eigenvalue on the unit circle
        return from_edges(150, {(i, (i + 1) % 150) for i in range(150)})
    if kind == "two_classes":  # two closed classes and a transient part feeding both
        e = {(i, (i * 7 + d) % 60) for i in range(60) for d in (1, 3)}
        e |= {(60 + i, 60 + (i * 5 + d) % 50) for i in range(50) for d in (1, 2, 4)}
        e |= {(110 + i, int(t)) for i in range(90) for t in rng.integers(0, 200, 3)}
        return from_edges(200, {(a, b) for a, b in e if a != b})
    if kind == "pairs":        # closed 2-cycles: eigenvalues 1 and -1
        e = {(2 * i, 2 * i + 1) for i in range(40)} | {(2 * i + 1, 2 * i) for i in range(40)}
        e |= {(80 + i, int(t)) for i in range(100) for t in rng.integers(0, 180, 4)}
        return from_edges(180, {(a, b) for a, b in e if a != b})
    if kind == "star_in":      # all mass into one dangling node
        return from_edges(140, {(i, 0) for i in range(1, 140)})
    if kind == "no_edges":
        return from_edges(33, set())
    if kind == "weighted":
        g = synth.directed_from(synth.chung_lu(500, 9, 2.5, seed=1), seed=2)
        w = np.exp(rng.normal(size=g.nnz)).astype(np.float32)
        return synth.Graph(g.n, g.row_ptr, g.col, w, directed=True)
    return synth.directed_from(synth.chung_lu(700, 6, 2.3, seed=9), p_both=0.5, dangling=0.08, seed=3)


@pytest.mark.parametrize("alpha", [0.15, 0.5, 0.03])
@pytest.mark.parametrize("kind", ["dag", "cycle", "two_classes", "pairs", "star_in", "no_edges", "weighted", "sparse"])
def test_directed_fp32_within_certificates_of_fp64(ctx, kind, alpha):
    import paper_2112_14944_gb300 as P
    g = graph(kind)
    G = ctx.upload_graph(g)
    view = np.arange(g.n, dtype=np.int32)
    eps = 1e-6
    D, _, cert, st = ctx.dppr(G, view, alpha, eps, P.FP32, out64=True)
    D64, _, c64, st64 = ctx.dppr(G, view, alpha, eps, P.FP64, out64=True)
    assert st == 0 and st64 == 0 and cert.max() <= eps
    assert (np.abs(D - D64) <= (cert + c64)[:, None] + 2.0 ** -40 * np.abs(D64)).all()
    # the same graph twice: the first call computed the modes, the second reuses them
    D2, _, c2, _ = ctx.dppr(G, view, alpha, eps, P.FP32, out64=True)
    assert np.array_equal(D, D2) and np.array_equal(cert, c2)


@pytest.mark.parametrize("kind", ["dag", "two_classes", "star_in", "no_edges", "sparse"])
def test_directed_solves_before_and_after_the_mode_analysis(ctx, kind):
    """The walk's dominant mode is computed once a graph's solves have come to 2,048
    source columns; the solves before and after agree with the FP64 path."""
    import paper_2112_14944_gb300 as P
    G = ctx.upload_graph(graph(kind))
    view = np.arange(G.n, dtype=np.int32)
    R, _, c64, s64 = ctx.dppr(G, view, 0.15, 1e-11, P.FP64, out64=True)
    assert s64 == 0
    for _ in range(2048 // G.n + 2):
        D, _, cert, st = ctx.dppr(G, view, 0.15, 1e-8, P.FP32_CSR, out64=True)
        assert st == 0
        assert (np.abs(D - R) <= (cert + c64)[:, None] + 2.0 ** -40 * np.abs(R)).all()
