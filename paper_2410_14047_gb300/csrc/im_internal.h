// Library-internal entry points shared by the translation units of the shared
// library (hidden symbols: not part of the C ABI).
#pragma once
#include <cuda_runtime.h>
#include <condition_variable>
#include <cstdint>
#include <mutex>

#include "../../include/difuser_im.h"

namespace imi {

// The resident blocks that the running queries of a server divide among them.
// A phase runs all its levels in one cooperative launch whose blocks wait for
// one another, so the grids in flight never add up to more than the GPU holds
// at once: a query takes blocks before its first launch, gives back or takes
// more only while none of its launches is in flight, and returns them at its
// end.  The even share is total / running: a query that joins waits until the
// others, at their next seed, have come down to it.
class BlockShares {
public:
    explicit BlockShares(int total) : total_(total), free_(total) {}
    // A query starts; leave ends it and returns what it holds.
    void enter();
    void leave(int held);
    // Its first phase comes: waits for its share, returns it.
    int take();
    // No phase of it is in flight: its new share in place of `held`.
    int adjust(int held);

private:
    int even() const { return total_ / running_ > 0 ? total_ / running_ : 1; }
    std::mutex mu_;
    std::condition_variable cv_;
    const int total_;
    int free_;
    int running_ = 0;
};

// Blocks that fit the current device at once in every phase launch (0: no
// cooperative launch).
int resident_blocks();

// A context that runs on `stream`, allocates from `pool` (stream-ordered) and
// takes the grids of its phase launches from `shares` (NULL: a launch a level).
im_status ctx_create_worker(int device, cudaStream_t stream, cudaMemPool_t pool, BlockShares* shares, im_ctx** out);
void ctx_set_budget(im_ctx* c, uint64_t bytes);
const char* ctx_error(const im_ctx* c);

// Alg. 4 of one query on context c, reading the resident graph g; the graph
// may belong to another context (same device) and is not modified.
im_status select_seeds_on(im_ctx* c, im_graph* g, int32_t K, int32_t J, const im_model* model,
                          uint64_t seed, double rebuild_eps, int32_t* seeds_out, double* score_out,
                          double* estimate_out);

// Device bytes one such query allocates (upper bound, allocator rounding included).
uint64_t query_bytes(const im_graph* g, int32_t J, int32_t K);
// Device bytes the graph holds; its vertex count; the device of its context.
uint64_t graph_bytes(const im_graph* g);
int32_t graph_n(const im_graph* g);
int graph_device(const im_graph* g);
// Validates a per-query model against the graph (uniform, WC, trivalency only
// when the graph was loaded with one of those).
im_status check_query_model(const im_graph* g, const im_model* model, char* msg, size_t cap);

}  // namespace imi
