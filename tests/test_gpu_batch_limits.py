"""A batch whose phases give up (level limit, barrier wait): IM_E_TIMEOUT after
every graph's remaining rounds ran over the counters such phases leave behind,
and the context gives the plain results afterwards."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

TIMEOUT = -5


@pytest.mark.parametrize("library", ["plain", "bounds"])
@pytest.mark.parametrize("buckets", [0, 1])
@pytest.mark.parametrize("limits", [{"max_levels": 2}, {"barrier_wait_ns": 0}], ids=["levels", "barrier"])
def test_a_batch_that_gives_up_leaves_the_context_usable(limits, buckets, library):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2410_14047_gb300 as im
    path = im.LIB_PATH
    if library == "bounds":
        from paper_2410_14047_gb300 import _build
        _build.build_bounds()
        path = im.BOUNDS_LIB_PATH
    graphs = [W.erdos_renyi(500 + 37 * i, 6 * (500 + 37 * i), seed=i) for i in range(8)]
    graphs += [W.from_edges(60, [(i, i + 1) for i in range(59)]), W.from_edges(1, []), W.from_edges(2, [(0, 1)])]
    p = [0.3] * 8 + [1.0] * 3
    J, K = [64, 1024] * 5 + [1024], [30] * 9 + [1, 2]
    ctx = im.im_ctx_create(0, lib_path=path)
    im.im_ctx_set_tuning(ctx, {"buckets": buckets})
    B = im.im_batch_load(ctx, graphs, p)
    want = im.im_batch_select_seeds(B, J, K, seed=3, rebuild_eps=0.0)
    for _ in range(2):
        im.im_ctx_set_limits(ctx, **limits)
        with pytest.raises(im.IMError) as ei:
            im.im_batch_select_seeds(B, J, K, seed=3, rebuild_eps=0.0)
        assert ei.value.status == TIMEOUT
        im.im_ctx_set_limits(ctx)
        got = im.im_batch_select_seeds(B, J, K, seed=3, rebuild_eps=0.0)
        for a, b in zip(got, want):
            assert a["seeds"].tolist() == b["seeds"].tolist()
            assert np.array_equal(a["score"], b["score"])
