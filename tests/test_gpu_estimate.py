"""Exact estimate sums at every register width and pieces-a-lane knob: rows of one rank
on both sides of the ranks where the sum's form changes (13 | 14, 29 | 30), visited
rows, single large ranks, random mixes; against 64-bit arithmetic."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def _rows(J, rng):
    rows = [np.full(J, r) for r in (0, 1, 13, 14, 28, 29, 30, 31, 32, 255)]
    for r in (29, 30, 32):  # one large rank among small ones, at the ends and inside
        for j in (0, J // 2 + 1, J - 1):
            row = np.minimum(rng.geometric(0.5, J) - 1, 20)
            row[j] = r
            rows.append(row)
    rows += [np.minimum(rng.geometric(0.5, J) - 1, 32) for _ in range(200)]
    rows += [rng.integers(0, 30, J) for _ in range(200)]
    rows += [rng.integers(0, 33, J) for _ in range(20)]
    rows += [np.where(rng.random(J) < 0.5, 255, rng.integers(12, 24, J)) for _ in range(200)]
    return np.stack(rows).astype(np.uint8)


@pytest.mark.parametrize("tile", [1, 2, 4])
@pytest.mark.parametrize("J", [16, 32, 64, 128, 256, 512, 1024])
def test_sums_and_pick_are_exact(J, tile):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2410_14047_gb300 as im
    M = _rows(J, np.random.default_rng(J))
    n = M.shape[0]
    g = W.from_edges(n, [(0, 1)])
    ctx = im.im_ctx_create(0)
    im.im_ctx_set_tuning(ctx, {"pick_tile": tile})
    sk = im.im_sketch_build(im.im_graph_load(ctx, g.rowptr, g.col, {"kind": "uniform", "p": 0.5}), J, 1)
    sk.set_registers(M)
    r = M.astype(np.int64)
    S = np.where(r == 255, 1 << 32, 1 << (32 - np.minimum(r, 32))).sum(1).astype(np.uint64)
    assert np.array_equal(sk.sums(), S)
    u, least, est = sk.pick()
    assert (u, least) == (int(np.argmin(S)), int(S.min()))
    assert est == J * 4294967296.0 / (0.77351 * float(S.min()))
