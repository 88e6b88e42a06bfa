"""Two servers, a caller's selections, step-level calls and a batch on one GPU at
the same time: their phases divide the device's blocks, and each gives what it
gives alone."""
import threading

import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("slots", [(3, 5), (40, 2)], ids=["few", "many"])
def test_callers_at_the_same_time_give_what_each_gives_alone(slots):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2410_14047_gb300 as im
    g = W.rmat(11, 8, seed=3)
    wc = {"kind": "wc"}
    graphs = [W.erdos_renyi(300 + 50 * i, 2000, seed=i) for i in range(6)]

    def context():
        c = im.im_ctx_create(0)
        return c, im.im_graph_load(c, g.rowptr, g.col, wc)

    def select(G):
        r = im.im_select_seeds(G, 5, 128, seed=7, rebuild_eps=-1.0)
        return r["seeds"].tolist(), r["score"].tolist()

    def steps(G):
        sk = im.im_sketch_build(G, 64, 11)
        out = []
        for _ in range(3):
            s = sk.pick()[0]
            out.append((s, sk.cover(s)))
            sk.rebuild()
        return out, sk.sums().tolist()

    def batch(B):
        return [(r["seeds"].tolist(), r["score"].tolist())
                for r in im.im_batch_select_seeds(B, [64, 128] * 3, [4] * 6, seed=5)]

    kinds = [{"graph": 0, "K": 3 + i % 4, "J": (32, 128, 1024)[i % 3], "seed": i, "rebuild_eps": -1.0,
              "model": wc if i % 2 else {"kind": "uniform", "p": 0.05}} for i in range(12)]
    ctx, G = context()
    plain = [im.im_select_seeds(G, q["K"], q["J"], model=q["model"], seed=q["seed"], rebuild_eps=-1.0) for q in kinds]
    B = im.im_batch_load(ctx, graphs, [0.1] * 6)
    alone = {"select": select(G), "steps": steps(G), "batch": batch(B)}

    servers = [im.Server(0, slots=k) for k in slots]
    for s in servers:
        s.add_graph(G)
    own = {"select": [], "steps": [], "batch": []}

    def caller(name):
        c, H = context()
        if name == "batch":
            H = im.im_batch_load(c, graphs, [0.1] * 6)
        for _ in range(6):
            own[name].append({"select": select, "steps": steps, "batch": batch}[name](H))

    threads = [threading.Thread(target=caller, args=(k,)) for k in own]
    for t in threads:
        t.start()
    tickets = [[s.submit(**q) for q in kinds * 10] for s in servers]
    results = [[s.wait(k) for k in ts] for s, ts in zip(servers, tickets)]
    for t in threads:
        t.join()
    for rs in results:
        assert len(rs) == 10 * len(plain)
        for r, p in zip(rs, plain * 10):
            assert r["status"] == 0, r["error"]
            assert r["seeds"].tolist() == p["seeds"].tolist()
            assert np.array_equal(r["score"], p["score"])
    for name, rs in own.items():
        assert len(rs) == 6 and all(r == alone[name] for r in rs), name
