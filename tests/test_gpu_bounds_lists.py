"""The bounds-checked variant over the stores of the bucketed lists, the listed
words of an incremental rebuild, a batch's seeds and the spread's queue: no bit
raised, and the oracle's results."""
import numpy as np
import pytest

import oracle as O
import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def im():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2410_14047_gb300 as lib
    from paper_2410_14047_gb300 import _build
    _build.build_bounds()
    lib.load_library(lib.BOUNDS_LIB_PATH)
    return lib


@pytest.mark.parametrize("J", [16, 64, 512, 1024])
@pytest.mark.parametrize("model", [{"kind": "uniform", "p": 0.02}, {"kind": "wc"}], ids=["p002", "wc"])
def test_bounds_checked_lists_and_rebuilds(im, model, J):
    g = W.chung_lu(6000, 12.0, 2.1, seed=6)
    ctx = im.im_ctx_create(0, lib_path=im.BOUNDS_LIB_PATH)
    im.im_ctx_set_tuning(ctx, {"buckets": 2, "incremental": 1})
    G = im.im_graph_load(ctx, g.rowptr, g.col, model)
    r = im.im_select_seeds(G, 5, J, seed=13, rebuild_eps=0.0, return_sketch=True)
    ref = O.select_seeds(g, O.thresholds(g, model), J, 5, 13, 0.0, "reverse")
    assert r["seeds"].tolist() == ref["seeds"].tolist()
    assert np.array_equal(r["score"], ref["score"])
    assert np.array_equal(r["sketch"].registers(), ref["M"])


@pytest.mark.parametrize("buckets", [0, 2])
def test_bounds_checked_batch(im, buckets):
    graphs = [W.erdos_renyi(400 + 90 * i, 3000, seed=i) for i in range(5)]
    ctx = im.im_ctx_create(0, lib_path=im.BOUNDS_LIB_PATH)
    im.im_ctx_set_tuning(ctx, {"buckets": buckets})
    B = im.im_batch_load(ctx, graphs, [0.1] * 5)
    for g, r in zip(graphs, im.im_batch_select_seeds(B, [64] * 5, [4] * 5, seed=3)):
        ref = O.select_seeds(g, O.thresholds(g, {"kind": "uniform", "p": 0.1}), 64, 4, 3, 0.01, "reverse")
        assert r["seeds"].tolist() == ref["seeds"].tolist()
        assert np.array_equal(r["score"], ref["score"])


@pytest.mark.parametrize("R", [33, 1025])
def test_bounds_checked_spread(im, R):
    g = W.rmat(10, 8, seed=4)
    model = {"kind": "uniform", "p": 0.2}
    G = im.im_graph_load(im.im_ctx_create(0, lib_path=im.BOUNDS_LIB_PATH), g.rowptr, g.col, model)
    r = im.im_spread_mc(G, [0, 5, 9], R, seed=8)
    assert (r["sum"], r["sumsq"]) == O.spread_ic(g, O.thresholds(g, model), [0, 5, 9], R, seed=8)
