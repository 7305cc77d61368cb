"""A certificate that is not a number is not a certificate: weights whose sums
leave FP32's range make the FP32 residual NaN or infinite, and every solver
reports that as not converged, never as success."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu
EPS = 1e-6


@pytest.fixture(scope="module")
def ctx():
    import paper_2112_14944_gb300 as P
    c = P.Context(0)
    yield c
    c.close()


def huge(directed=False):
    """Three nodes, all pairs, weights 3e38: every strength is 6e38, beyond FP32's largest number."""
    return synth.Graph(3, np.array([0, 2, 4, 6], np.int64), np.array([1, 2, 0, 2, 0, 1], np.int32),
                       np.full(6, 3e38, np.float32), directed=directed)


def tame():
    return synth.sbm([30, 30], 0.3, 0.05, seed=1)


@pytest.mark.parametrize("directed", [False, True])
def test_dppr_without_a_finite_certificate_is_not_converged(ctx, directed):
    import paper_2112_14944_gb300 as P
    from paper_2112_14944_gb300 import _binding as B
    G = ctx.upload_graph(huge(directed))
    view = np.arange(3, dtype=np.int32)
    _, _, cert, st = ctx.dppr(G, view, 0.15, EPS, P.FP32_CSR, out64=True)
    assert not (cert <= EPS).all()
    assert st == B.PPRVIZ_E_NOT_CONVERGED
    assert not ctx.stats()["max_cert"] <= EPS


def test_level_dppr_without_a_finite_certificate_is_not_converged(ctx):
    from paper_2112_14944_gb300 import _binding as B
    G = ctx.upload_graph(huge())
    _, _, cert, st = ctx.level_dppr(G, [np.array([0], np.int32), np.array([1, 2], np.int32)], 0.15, EPS)
    assert not (cert <= EPS).all()
    assert st == B.PPRVIZ_E_NOT_CONVERGED


def test_one_view_without_a_finite_certificate_is_not_converged(ctx):
    from paper_2112_14944_gb300 import _binding as B
    graphs = [ctx.upload_graph(tame()), ctx.upload_graph(huge()), ctx.upload_graph(tame())]
    off = np.concatenate([[0], np.cumsum([g.n for g in graphs])]).astype(np.int64)
    n = int(off[-1])
    x, stress, cert = np.empty((n, 2), np.float32), np.empty(3), np.empty(n)
    st = B.pprviz_views_batch(ctx.h, [g.h for g in graphs], off, 0.15, EPS, 1, synth.uniform_x0(n, seed=1), None, x,
                              stress, cert, 0)
    assert not (cert[off[1]:off[2]] <= EPS).all()
    assert (cert[:off[1]] <= EPS).all() and (cert[off[2]:] <= EPS).all()
    assert st == B.PPRVIZ_E_NOT_CONVERGED
    assert not ctx.stats()["max_cert"] <= EPS
