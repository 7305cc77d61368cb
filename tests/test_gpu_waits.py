"""Bounded waits that run out: the resident layout's grid barrier and the 3xTF32
sweep's completion waits end after their deadline, the call reports E_TIMEOUT,
and the next call on the context is right. (pprviz_test_expire_wait makes one
CTA leave out a signal; nothing faults.)"""
import time

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


def expires(ctx, launches, call):
    import paper_2112_14944_gb300 as P
    from paper_2112_14944_gb300 import _binding as B
    good = call()
    for _ in range(launches):
        B.pprviz_test_expire_wait(ctx.h)
    t0 = time.perf_counter()
    with pytest.raises(P.PPRVizError) as ei:
        call()
    assert ei.value.status == B.PPRVIZ_E_TIMEOUT and "wait expired" in B.pprviz_last_error(ctx.h)
    assert time.perf_counter() - t0 < 30.0
    again = call()
    assert np.array_equal(good[0], again[0])


@pytest.mark.parametrize("k", [300, 1500])
def test_resident_layout_barrier(ctx, k):
    import paper_2112_14944_gb300 as P
    rng = np.random.default_rng(k)
    r = rng.uniform(2.0, 12.0, (k, k)).astype(np.float32)
    delta = (r + r.T) / 2
    np.fill_diagonal(delta, 0)
    x0 = synth.uniform_x0(k, seed=1)
    # the first launch that can withhold is the inverse, the second the layout itself
    expires(ctx, 2, lambda: ctx.layout(delta, x0, 3, P.FP32))


def test_launches_without_a_wait_are_not_counted(ctx):
    """One pivot block and one CTA wait for nobody: the aid passes over them."""
    import paper_2112_14944_gb300 as P
    from paper_2112_14944_gb300 import _binding as B
    small, large = np.full((4, 4), 3.0, np.float32), np.full((300, 300), 3.0, np.float32)
    np.fill_diagonal(small, 0)
    np.fill_diagonal(large, 0)
    x4, x300 = synth.uniform_x0(4, seed=1), synth.uniform_x0(300, seed=1)
    good = ctx.layout(small, x4, 2, P.FP32)[0]
    B.pprviz_test_expire_wait(ctx.h)
    B.pprviz_test_expire_wait(ctx.h)
    assert np.array_equal(ctx.layout(small, x4, 2, P.FP32)[0], good)
    with pytest.raises(P.PPRVizError) as ei:
        ctx.layout(large, x300, 2, P.FP32)
    assert ei.value.status == B.PPRVIZ_E_TIMEOUT


@pytest.mark.parametrize("columns", [128, 300])  # 128- and 256-wide tiles
@pytest.mark.parametrize("sweep", [1, 3])
def test_tensor_core_sweep(ctx, columns, sweep):
    import paper_2112_14944_gb300 as P
    G = ctx.upload_graph(synth.dense_clustered(700, blocks=4, density=0.2, seed=2))
    view = np.arange(columns, dtype=np.int32)
    expires(ctx, sweep, lambda: ctx.dppr(G, view, 0.15, 1e-6, P.FP32_TC))
