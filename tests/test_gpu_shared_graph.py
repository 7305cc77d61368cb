"""A graph used by several contexts at once, each with a host thread of its own:
what a graph keeps is made on first use, once, whichever thread comes first."""
import threading

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu
THREADS = 4


def graphs():
    yield "directed", synth.directed_from(synth.chung_lu(2300, 12, 2.5, seed=1), p_both=0.3, seed=3)
    yield "undirected", synth.chung_lu(2300, 12, 2.5, seed=2)            # split rows, spectral bound
    yield "small", synth.sbm([60, 70], 0.2, 0.05, seed=3)                # analysis in one launch
    yield "dense", synth.dense_clustered(700, blocks=4, density=0.2, seed=4)  # dense weights


@pytest.mark.parametrize("kind", [k for k, _ in graphs()])
def test_first_solves_of_one_graph_from_several_threads(kind):
    import paper_2112_14944_gb300 as P
    g = dict(graphs())[kind]
    view = np.arange(g.n, dtype=np.int32)
    ctxs = [P.Context(0) for _ in range(THREADS)]
    try:
        R, _, c64, st = ctxs[0].dppr(ctxs[0].upload_graph(g), view, 0.15, 1e-9, P.FP64, out64=True)
        assert st == 0
        for _ in range(3):  # a new graph each time: the first solves run side by side
            G = ctxs[0].upload_graph(g)
            out, start = [None] * THREADS, threading.Barrier(THREADS)

            def solve(t):
                start.wait()
                out[t] = ctxs[t].dppr(G, view, 0.15, 1e-6, P.FP32, out64=True)

            threads = [threading.Thread(target=solve, args=(t,)) for t in range(THREADS)]
            for t in threads:
                t.start()
            for t in threads:
                t.join()
            for o in out:
                assert o is not None and o[3] == 0 and o[2].max() <= 1e-6
                assert (np.abs(o[0] - R) <= (o[2] + c64)[:, None] + 2.0 ** -40 * np.abs(R)).all()
    finally:
        for c in ctxs:
            c.close()
