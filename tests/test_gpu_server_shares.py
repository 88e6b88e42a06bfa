"""Served queries on shares of the GPU's blocks: any number of slots (from one
query holding every block to more slots than an even share of eight blocks), and a
caller's own selections at the same time, give the plain path's results."""
import threading

import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("slots", [1, 3, 8, 40])
def test_shares_give_plain_results_beside_a_callers_selections(slots):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2410_14047_gb300 as im
    g = W.rmat(11, 8, seed=3)
    ctx = im.im_ctx_create(0)
    G = im.im_graph_load(ctx, g.rowptr, g.col, {"kind": "wc"})
    queries = [{"graph": 0, "K": 3 + i % 4, "J": (32, 128, 1024)[i % 3], "seed": i, "rebuild_eps": -1.0,
                "model": {"kind": "wc"} if i % 2 else {"kind": "uniform", "p": 0.05}} for i in range(3 * slots)]
    plain = [im.im_select_seeds(G, q["K"], q["J"], model=q["model"], seed=q["seed"], rebuild_eps=-1.0)
             for q in queries[:12]]
    srv = im.Server(0, slots=slots)
    srv.add_graph(G)
    own = []

    def select():
        c = im.im_ctx_create(0)
        H = im.im_graph_load(c, g.rowptr, g.col, {"kind": "wc"})
        own.extend(im.im_select_seeds(H, 4, 128, seed=7)["seeds"].tolist() for _ in range(10))

    t = threading.Thread(target=select)
    t.start()
    results = [srv.wait(k) for k in [srv.submit(**q) for q in queries]]
    t.join()
    assert not any(r["status"] for r in results), [r["error"] for r in results if r["status"]]
    for q, r, p in zip(queries, results, plain):
        assert r["seeds"].tolist() == p["seeds"].tolist()
        assert np.array_equal(r["score"], p["score"])
    assert len(own) == 10 and all(s == own[0] for s in own)
