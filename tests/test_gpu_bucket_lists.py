"""Bucketed live lists and the queues of a phase at the sizes where their
kernels change course: rows across the 32- and 512-edge borders of a warp's
share, runs of empty rows, every chunk count, levels with more entries than a
block's buffer holds; all against the oracle."""
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
    lib.load_library()
    return lib


def _graph():
    """A source of 1500 edges, a target of 700, rows of one edge, and long
    runs of vertices without edges."""
    edges = [(0, v) for v in range(1, 1501)] + [(v, 5000) for v in range(1, 701)]
    edges += [(5000, v) for v in range(6000, 6033)] + [(v, v + 1) for v in range(6000, 6600)]
    return W.from_edges(9000, edges)


MODELS = [{"kind": "uniform", "p": 1.0}, {"kind": "uniform", "p": 0.3}, {"kind": "uniform", "p": 0.004},
          {"kind": "wc"}, {"kind": "trivalency", "seed": 5}]


@pytest.mark.parametrize("J", [16, 32, 512, 1024])
@pytest.mark.parametrize("model", MODELS, ids=["p1", "p03", "p0004", "wc", "tri"])
def test_selection_over_bucketed_lists(im, model, J):
    g = _graph()
    ctx = im.im_ctx_create(0)
    im.im_ctx_set_tuning(ctx, {"buckets": 1, "chain": 8})
    r = im.im_select_seeds(im.im_graph_load(ctx, g.rowptr, g.col, model), 4, J, seed=9, rebuild_eps=-1.0,
                           return_sketch=True)
    ref = O.select_seeds(g, O.thresholds(g, model), J, 4, 9, -1.0, "reverse")
    assert r["seeds"].tolist() == ref["seeds"].tolist()
    assert np.array_equal(r["score"], ref["score"])
    assert np.array_equal(r["sketch"].registers(), ref["M"])


@pytest.mark.parametrize("buckets", [0, 1])
def test_levels_larger_than_the_blocks_buffers(im, buckets):
    # every vertex changes at every level: 304 blocks of 1024 entries hold less
    # than a level's 400,000 vertices (or their chunks' buckets)
    g = W.erdos_renyi(400_000, 1_600_000, seed=8)
    model = {"kind": "uniform", "p": 0.4}
    ctx = im.im_ctx_create(0)
    im.im_ctx_set_tuning(ctx, {"buckets": buckets, "dense_div": 0})
    sk = im.im_sketch_build(im.im_graph_load(ctx, g.rowptr, g.col, model), 32, 3)
    X, salt = O.draw_sims(3, 32)
    assert np.array_equal(sk.registers(), O.build_reverse(g, O.thresholds(g, model), 32, X, salt))
