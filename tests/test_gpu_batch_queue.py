"""A batch of so many tiny graphs that one round's seeds have more live chunks than
the bucket queue holds: the cover walks every bucket instead, with the solo
runs' results."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def test_seeds_of_many_tiny_graphs_past_the_queue():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2410_14047_gb300 as im
    # 20,000 seeds of 64 live chunks (J = 1024, p = 1); the queue holds 2^20
    # entries.  A dense graph whose edges never fire keeps the lists below
    # their bound of 4 entries an edge.
    pair = W.from_edges(2, [(0, 1)])
    dense = W.erdos_renyi(1500, 330_000, seed=2)
    G = 20_000
    ctx = im.im_ctx_create(0)
    im.im_ctx_set_tuning(ctx, {"buckets": 1})
    B = im.im_batch_load(ctx, [pair] * G + [dense], [1.0] * G + [0.0])
    res = im.im_batch_select_seeds(B, [1024] * (G + 1), [2] * (G + 1), seed=4)
    for g, p, rs in ((pair, 1.0, res[:G]), (dense, 0.0, res[G:])):
        H = im.im_graph_load(ctx, g.rowptr, g.col, {"kind": "uniform", "p": p})
        want = im.im_select_seeds(H, 2, 1024, seed=4)
        for r in rs:
            assert r["seeds"].tolist() == want["seeds"].tolist()
            assert np.array_equal(r["score"], want["score"])
