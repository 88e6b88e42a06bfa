"""Estimate sums whose partial sums need every bit the matrix product has to keep:
a quad of lanes full of the largest lower terms (rank 14) with the smallest ones
(ranks 28, 29) among them, and full of the largest upper terms (ranks 0, visited)
with the smallest (rank 13); at every register width and pieces-a-lane knob.  The
widest is J = 1024 with 4 pieces a lane: 256 terms, 510 + 2^-14, 24 bits."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def _rows(J):
    spots = sorted({s for s in (0, 1, 15, 16, J // 2, J - 16, J - 2, J - 1) if s < J})
    rows = []
    for big, smalls in ((14, (28, 29)), (0, (13,)), (255, (13, 29))):
        rows.append(np.full(J, big))
        for small in smalls:
            for k in range(len(spots)):
                for m in (1, 2, 3):
                    row = np.full(J, big)
                    row[spots[k:k + m]] = small
                    rows.append(row)
            row = np.full(J, small)  # and the other way round
            row[J // 2] = big
            rows.append(row)
            for a, b in ((big, small), (small, big)):
                rows.append(np.where(np.arange(J) % 2 == 0, a, b))
    return np.stack(rows).astype(np.uint8)


@pytest.mark.parametrize("tile", [1, 2, 4])
@pytest.mark.parametrize("J", [16, 64, 128, 256, 512, 1024])
def test_extreme_sums_are_exact(J, tile):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2410_14047_gb300 as im
    M = _rows(J)
    n = M.shape[0]
    g = W.from_edges(n, [(0, 1)])
    ctx = im.im_ctx_create(0)
    im.im_ctx_set_tuning(ctx, {"pick_tile": tile})
    sk = im.im_sketch_build(im.im_graph_load(ctx, g.rowptr, g.col, {"kind": "uniform", "p": 0.5}), J, 1)
    sk.set_registers(M)
    r = M.astype(np.int64)
    S = np.where(r == 255, 1 << 32, 1 << (32 - np.minimum(r, 32))).sum(1).astype(np.uint64)
    assert np.array_equal(sk.sums(), S)
    # every row's sum through the pick, the least first
    order = np.lexsort((np.arange(n), S))
    for u in order[: min(n, 40)]:
        assert sk.pick()[:2] == (int(u), int(S[u]))
