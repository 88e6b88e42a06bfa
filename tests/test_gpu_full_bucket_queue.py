"""A level of a huge graph (63 million edges and more, where the packed queue counter
needs it) that changes more buckets than the queue holds: further entries are
refused, the next level walks every bucket, and the registers are those of the
edge scans, which have no such queue."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_a_full_bucket_queue_of_a_huge_graph():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2410_14047_gb300 as im
    # 70,000 vertices, 64 chunks each (J = 1024): up to 4.5 million buckets, a
    # queue of 2^20.  A tenth of the vertices has no out-edge and never
    # changes, so that the second level's work is below m and it queues buckets.
    n, src = 70_000, 63_000
    gen = torch.Generator(device="cuda")
    gen.manual_seed(12)
    key = torch.randint(0, src, (66_000_000,), generator=gen, device="cuda") * n + torch.randint(
        0, n, (66_000_000,), generator=gen, device="cuda")
    key = torch.unique(key)
    u, v = torch.div(key, n, rounding_mode="floor"), key % n
    v, u = v[u != v], u[u != v]
    m = int(u.numel())
    assert m >= (1 << 26) - (1 << 22)
    rowptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    rowptr[1:] = torch.cumsum(torch.bincount(u, minlength=n), 0)
    rowptr, col = rowptr.to(torch.int32).cpu().numpy(), v.to(torch.int32).cpu().numpy()
    del key, u, v
    torch.cuda.empty_cache()
    ctx = im.im_ctx_create(0)
    G = im.im_graph_load(ctx, rowptr, col, {"kind": "uniform", "p": 0.002})
    registers = {}
    for buckets in (0, 1):
        im.im_ctx_set_tuning(ctx, {"buckets": buckets})
        im.im_ctx_set_trace(ctx, True)
        sk = im.im_sketch_build(G, 1024, 5)
        most = max(t["count"] for t in im.im_last_trace(ctx))
        im.im_ctx_set_trace(ctx, False)
        registers[buckets] = sk.registers()
        assert (most >= 1 << 20) == (buckets == 1)  # more than the queue holds
    assert np.array_equal(registers[0], registers[1])
