"""Monte-Carlo spread where its level kernel changes course: one edge a vertex,
rows across a batch, one and two batches of simulations, edges that always
fire (every lane of a step has a hit) and never do; against the oracle's
coins."""
import pytest

import oracle as O
import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("R", [31, 33, 1024, 1025])
@pytest.mark.parametrize("p", [1.0, 0.25, 0.0])
def test_spread_steps(R, p):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2410_14047_gb300 as im
    edges = [(0, v) for v in range(1, 70)] + [(v, v + 1) for v in range(69, 130)]
    edges += [(v, 200 + (3 * v + k) % 37) for v in range(1, 33) for k in range(v % 5)]
    g = W.from_edges(240, sorted(set(edges)))
    model = {"kind": "uniform", "p": p}
    G = im.im_graph_load(im.im_ctx_create(0), g.rowptr, g.col, model)
    seeds = [0, 3, 130, 239]
    r = im.im_spread_mc(G, seeds, R, seed=21)
    assert (r["sum"], r["sumsq"]) == O.spread_ic(g, O.thresholds(g, model), seeds, R, seed=21)
