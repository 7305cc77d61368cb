"""Source-group widths of the level-l DPPR beyond 64 supernodes: narrow groups
only on graphs large enough for them, and the same values at every width
(supernodes of one leaf reduce to pprviz_dppr's DPPR)."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,nsup,kind,group", [
    (43000, 70, "unweighted", 128), (45000, 96, "unweighted", 128), (70001, 70, "unweighted", 64),
    (130001, 70, "unweighted", 32), (200001, 100, "unweighted", 64), (45000, 96, "weighted", 128),
    (200001, 100, "weighted", 128), (300001, 130, "weighted", 32), (43000, 70, "directed", 128),
    (50001, 96, "directed", 64), (150001, 100, "directed", 32),
])
def test_level_group_width(n, nsup, kind, group):
    import paper_2112_14944_gb300 as P
    g = synth.chung_lu(n, 4, 2.5, seed=3)
    if kind == "weighted":  # symmetric weights from the pair
        u, v = np.repeat(np.arange(n), np.diff(g.row_ptr)), g.col.astype(np.int64)
        w = (0.5 + ((np.minimum(u, v) * 7919 + np.maximum(u, v) * 104729) % 997) / 997.0).astype(np.float32)
        g = synth.Graph(n, g.row_ptr, g.col, w)
    if kind == "directed":
        g = synth.directed_from(g, seed=4)
    c = P.Context(0)
    try:
        G = c.upload_graph(g)
        view = synth.sample_view(n, nsup, seed=1).astype(np.int32)
        L, _, cl, st = c.level_dppr(G, [view[i:i + 1] for i in range(nsup)], 0.15, 1e-6, out64=True)
        assert st == 0 and cl.max() <= 1e-6
        assert c.stats()["source_group"] == group
        D, _, cd, st = c.dppr(G, view, 0.15, 1e-6, P.FP32_CSR, out64=True)
        assert st == 0
        assert (np.abs(L - D) <= (cl + cd)[:, None] + 2.0 ** -40 * np.abs(D)).all()
    finally:
        c.close()
