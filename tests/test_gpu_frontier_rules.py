"""Rules that choose a frontier path by sizes, at the sizes where they switch:
registers and seeds equal the oracle's on both sides of each line."""
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


def _hub_graph(deg, n=60_000, m=700_000):
    """Random edges among vertices 1.. and a hub 0 with in-edges from 1..deg
    (more edges than a small level's limit, so hubs are not scanned there anyway)."""
    g = W.erdos_renyi(n, m, seed=4)
    u = np.repeat(np.arange(n), np.diff(g.rowptr))
    keep = (u != 0) & (g.col != 0)
    edges = np.unique(np.concatenate([np.stack([u[keep], g.col[keep]], 1),
                                      np.stack([np.arange(1, deg + 1), np.zeros(deg, np.int64)], 1)]), axis=0)
    rowptr = np.zeros(n + 1, np.int32)
    np.add.at(rowptr, edges[:, 0] + 1, 1)
    return W.Graph(n, np.cumsum(rowptr).astype(np.int32), edges[:, 1].astype(np.int32))


@pytest.mark.parametrize("J", [32, 256])
@pytest.mark.parametrize("deg,searched", [(1535, True), (1536, False), (256, False), (257, True)])
def test_hub_search_up_to_two_candidates_a_simulation(im, deg, searched, J):
    # p = 1/1024: 2^31 / 512 hashes agree above the threshold's top bit, so a
    # hub of 1536 in-edges has 3 candidates a simulation; 256 is heavy_indeg
    g = _hub_graph(deg)
    model = {"kind": "uniform", "p": 1.0 / 1024}
    ctx = im.im_ctx_create(0)
    im.im_ctx_set_tuning(ctx, {"buckets": 0})
    sk = im.im_sketch_build(im.im_graph_load(ctx, g.rowptr, g.col, model), J, 3)
    assert (im.im_last_stats(ctx)["sweep_heavy"] > 0) == searched
    X, salt = O.draw_sims(3, J)
    assert np.array_equal(sk.registers(), O.build_reverse(g, O.thresholds(g, model), J, X, salt))
