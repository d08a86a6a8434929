// Batched solve internals shared by dsg_batch_solve and the server: the
// per-graph tables of one block-per-graph launch.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace dsg {

struct BatchArgs {
    uint32_t G;
    const uint64_t* const* goff;  // per graph: its n+1 row offsets (positions in its gadj)
    const uint32_t* const* gadj;  // per graph: adjacency base
    const uint64_t* slot;         // per graph: first scratch / output slot
    const uint32_t* gn;           // per graph: vertex count
    const uint32_t* p;
    const uint32_t* q;
    const uint8_t* want_core;
    const uint32_t* order;  // graph ids, largest first
    uint32_t* core;         // core numbers per vertex slot (nullable)
    uint8_t* out_set;       // membership in the densest set found (nullable)
    uint64_t* res;          // 4 per graph: E, V, rounds, best_round
    unsigned long long* next;   // low half: graphs taken, high half: teams that have taken one
    uint32_t hot_deg;
    unsigned long long* stats;  // nullable, 3 counters summed over the batch: sum over graphs and rounds of
                                // |S_r|, alive-neighbour decrements of the peels, adjacency entries scanned
};

// The graphs of a launch in its order (host): vertices and row entries.
struct BatchSizes {
    const uint32_t* n;
    const uint64_t* e;
};

// Launch the block-per-graph kernel over a.order[0, a.G) on stream s
// (asynchronous) with `block` threads per block (256, 512 or 1024; 0: 512),
// at most max_grid blocks (0: as many as fit).  a.next must be zeroed and
// every table filled.  The kernel works on slabs of scratch, one per block:
// the k-th block to start gets one for the largest of the graphs from the
// k-th on, which are all it can meet.  At most scratch_max bytes of them, and
// half as many while there is no memory for them, but at least one.  *slabs
// gets them, to be freed by the caller in stream order; the first word is an
// error word to read when the launch is done.
cudaError_t batch_launch(const BatchArgs& a, const BatchSizes& sizes, size_t scratch_max, cudaStream_t s, void** slabs,
                         uint32_t block = 0, uint32_t max_grid = 0);

// The same with a thread-block cluster per graph (on at most max_sms SMs; 0:
// all), for the graphs too large for a block of their own to keep the launch
// short.
cudaError_t batch_cluster_launch(const BatchArgs& a, const BatchSizes& sizes, size_t scratch_max, cudaStream_t s,
                                 void** slabs, uint32_t max_sms = 0);

// Whether a graph of a batch of `total` work (2m + n, summed) is solved by the
// whole GPU, before the others.
bool batch_takes_grid(uint64_t work, uint32_t n, uint64_t total);
// How many of the others, given largest first, get a cluster each; the rest
// get a block each.
uint32_t batch_clusters(const uint64_t* work, uint32_t G, uint64_t total);

// Blocks of `block` threads the block-per-graph kernel can keep resident on the GPU.
uint32_t batch_slots_for(uint32_t block);

}  // namespace dsg
