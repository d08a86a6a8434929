// Shared pieces of the peel and core kernels: the frontier representation
// (short rows listed by vertex, long rows cut into fixed-size chunk items),
// the row scanner that walks a frontier's adjacency, and entry points shared
// between translation units.
#pragma once

#include <algorithm>
#include <condition_variable>
#include <mutex>

#include "dsg_common.cuh"

namespace dsg {

// Adjacency entries are read once per solve: load them with the streaming
// (evict-first) policy so they do not push the per-vertex state (degrees,
// marks), which every entry looks up at random, out of L2.
__device__ __forceinline__ uint32_t ld_stream(const uint32_t* p) { return __ldcs(p); }

// Tuning knobs of the round kernels (see tune.cu for the defaults and the
// autotuner that picks them).
struct Tuning {
    uint32_t block = 512;       // threads per block of the persistent kernels
    uint32_t blocks_per_sm = 0; // 0: as many as fit
    uint32_t short_max = 32;    // kept for saved tables and callers; no kernel tells short rows apart any more
    uint32_t chunk_len = 256;   // rows are cut into pieces of at most this many entries
    uint32_t hot_deg = 0;       // decrements of vertices at or above this degree are combined in shared memory
                                // (0: by the number of blocks, hot_threshold)
    uint32_t local_max = 1024;  // k-core: rows up to this length reached while draining stay in the block
    uint32_t local_work = 16384; // k-core: ... while that block's local share of the sub-round stays within this
    uint32_t inline_max = 256;   // k-core: rows up to this length claimed by a block's level scan are drained by
                                 // that block; longer ones by every warp in the next sub-round
    uint32_t tail_max = 65536;   // k-core: scale of the graphs and remaining graphs whose core numbers are searched
                                 // bit by bit instead of level by level (kTailHandOver, kTailWhole; 0: never)
    uint32_t batch_split = 0;    // batches: a graph whose work (2m + n) exceeds this is solved by the
                                 // grid-wide kernels, the others by a block each (0: batch_takes_grid)
    uint32_t batch_block = 512;  // batches: threads per block of the block-per-graph kernel
    uint32_t peel_lazy = 1;      // peel: thin-tail rounds test only the candidate list (0: every round
                                 // tests the whole alive list); read from the global tuning only
    uint32_t peel_vec = 0;       // kept for callers; the 128-bit row loads it chose were slower and are gone
};

// Tuning of a batch of G graphs with `work` = sum of (2m + n): the autotuned
// entry of its class if there is one, else current_tuning().
Tuning tuning_for_batch(uint32_t G, uint64_t work);

Tuning current_tuning();

// Tuning for a solve of kernel 0 (peel) or 1 (core numbers) on graph g: the
// autotuned entry of g's size class if there is one, else current_tuning().
Tuning tuning_for(const dsg_graph* g, int kernel);

// Autotuned solve times (ms) of g's size class for the peel (at the tuning
// eps) and the core numbers; false unless both were tuned.
bool tuned_times(const dsg_graph* g, double* peel_ms, double* core_ms);

// Counts one kernel launch and, when profiling is on, brackets it with CUDA
// events on its stream.  Construct right before the launch, destroy right
// after it:  { LaunchScope ls("name", s); kernel<<<...>>>(...); }
class LaunchScope {
  public:
    LaunchScope(const char* name, cudaStream_t s);
    ~LaunchScope();
  private:
    const char* name_;
    cudaStream_t s_;
    void* a_ = nullptr;
    void* b_ = nullptr;
    bool timed_ = false;
};

// Ingest raw pairs held in a CSR (each entry (v, adj[j]) is one pair).
dsg_status ingest_from_csr_entries(uint32_t n, const uint64_t* off, const uint32_t* adj, uint64_t total,
                                   uint32_t flags, cudaStream_t s, dsg_graph** out);

// Room on the GPU, in blocks of an SM each, for the grids of several host
// threads whose blocks wait for one another: as long as all that run at once
// fit side by side, none depends on another's leaving.
class GridRoom {
  public:
    // least: what a thread that wants that much waits for
    void set(uint32_t blocks, uint32_t least) {
        free_ = blocks;
        least_ = least;
    }
    // Up to `want` blocks, as many as are free once there are min(want, least).
    uint32_t take(uint32_t want) {
        std::unique_lock<std::mutex> lk(mu_);
        cv_.wait(lk, [&] { return free_ >= std::min(want, least_); });
        const uint32_t got = std::min(want, free_);
        free_ -= got;
        return got;
    }
    void give(uint32_t blocks) {
        {
            std::lock_guard<std::mutex> lk(mu_);
            free_ += blocks;
        }
        cv_.notify_all();
    }

  private:
    std::mutex mu_;
    std::condition_variable cv_;
    uint32_t free_ = 1, least_ = 1;
};

// dsg_graph_from_edges; room (nullable): other work is on the GPU, take few
// blocks, and those that wait for one another from there.
dsg_status graph_from_edges(uint32_t n, uint64_t m_raw, const uint32_t* src, const uint32_t* dst, uint32_t flags,
                            GridRoom* room, void* stream, dsg_graph** out);

// One peel on a graph (any dsg_graph, including a view into a packed batch):
// set_dev (device, nullable) gets the densest-set mask; out4 = E, V, rounds,
// best_round.
// extra2 (nullable): sum over the rounds of |S_r| and the alive-neighbour decrements.
dsg_status peel_into(const dsg_graph* g, uint32_t p, uint32_t q, uint8_t* set_dev, uint64_t out4[4],
                     uint64_t* extra2 = nullptr);

// Core numbers of a graph into core_out (host or device); stats nullable.
dsg_status run_kcore(const dsg_graph* g, uint32_t* core_out, uint64_t* stats, uint32_t nstats,
                     uint64_t* trace_dev = nullptr, uint64_t trace_cap = 0, uint64_t* stamps = nullptr);

// The core numbers of the vertices whose claim bit is clear (at most cap of
// them, none with a core number below lo; deg holds their degrees), on the
// compacted remaining graph; writes them into deg and adds what a level run
// would count (levels, remaining entries) and the atomics into stats5[0],
// [2], [4]; with a trace buffer, block 0 stamps each wave there.
constexpr uint32_t kTailMaxVertices = 131072;  // largest Tuning::tail_max
// The search takes over from the levels once at most kTailHandOver * tail_max
// vertices remain, and takes graphs of up to kTailWhole * tail_max vertices
// whole (core numbers, ms, at hand-overs of 65,536 / 131,072 / 262,144 /
// 524,288 vertices: Chung-Lu 2^24 20.5 / 18.7 / 17.7 / 18.0, 3 10^6 4.93 /
// 4.43 / 4.31 / 4.45, 2 10^6 4.13 / 3.74 / 3.55 / 3.78; whole against the best
// hand-over: Chung-Lu 7 10^5 1.29 / 1.52, 3 10^5 0.98 / 1.16, 10^5 0.65 / 0.91,
// R-MAT 2^20 2.37 / 2.36, 2^18 0.84 / 1.04, Erdos-Renyi 10^6 0.86 / 1.41;
// at 2 10^6 vertices of mean degree 30 it no longer wins: 3.71 / 3.55).
constexpr uint64_t kTailHandOver = 4;
constexpr uint64_t kTailWhole = 16;
constexpr uint64_t kTailMaxEntries = 1ull << 36;  // beyond: levels only
dsg_status kcore_tail(const dsg_graph* g, uint32_t* deg, const uint32_t* claim, uint32_t cap, uint32_t lo,
                      uint64_t* stats5, uint64_t* trace = nullptr, uint64_t trace_cap = 0, uint64_t* stamps = nullptr);

// The same on a whole graph of r vertices (rows off, adj;
// rid nullable: original ids); limits of the grid from g.
dsg_status core_split(uint32_t r, uint32_t lo, const uint64_t* off, const uint32_t* adj, uint64_t entries,
                      const uint32_t* rid, uint32_t* core, const dsg_graph* g, Scratch& sc, uint64_t* stats5,
                      uint64_t* trace, uint64_t trace_cap, uint64_t* stamps);

// floor(2(p+q)E / (qS)) clamped to 32 bits; S > 0 (Algorithm 1's threshold).
// A division of two 64-bit numbers unless one of them needs 128 bits.
__device__ __forceinline__ uint32_t peel_threshold(uint64_t p, uint64_t q, uint64_t E, uint64_t S) {
    const uint64_t a = 2 * (p + q);
    uint64_t t;
    if (__umul64hi(a, E) == 0 && __umul64hi(q, S) == 0) {
        t = a * E / (q * S);
    } else {
        const unsigned __int128 w = (unsigned __int128)a * E / ((unsigned __int128)q * S);
        t = w > 0xffffffffu ? 0xffffffffu : (uint64_t)w;
    }
    return t > 0xffffffffu ? 0xffffffffu : (uint32_t)t;
}

// Device check that a graph is canonical (sorted rows, no loops, no repeats,
// symmetric, ids < n).  DSG_EINVAL with a message if not.
dsg_status validate_csr(const dsg_graph* g);

// Grid size for a cooperative launch of `kernel` with `block` threads and
// `smem` dynamic shared memory, capped so small problems use few blocks (and
// at max_grid when that is non-zero).
template <class K>
cudaError_t coop_grid(K kernel, uint32_t block, size_t smem, uint64_t work_items, uint32_t blocks_per_sm,
                      uint32_t* grid, uint32_t max_grid = 0) {
    int per_sm = 0;
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, (int)block, smem);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    if (blocks_per_sm && (int)blocks_per_sm < per_sm) per_sm = (int)blocks_per_sm;
    uint64_t g = (uint64_t)per_sm * (uint64_t)dev_info().sms;
    uint64_t need = (work_items + block - 1) / block;
    if (need < 1) need = 1;
    if (g > need) g = need;
    if (max_grid && g > max_grid) g = max_grid;
    *grid = (uint32_t)g;
    return cudaSuccess;
}

// A launch of thread-block clusters of `blocks` blocks, `grid` blocks in all.
inline cudaLaunchConfig_t cluster_config(uint32_t grid, uint32_t blocks, uint32_t threads, size_t smem, cudaStream_t s,
                                         cudaLaunchAttribute* attr) {
    attr->id = cudaLaunchAttributeClusterDimension;
    attr->val.clusterDim.x = blocks;
    attr->val.clusterDim.y = 1;
    attr->val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cfg;
}

// How many such clusters of a kernel the current context can hold at once, the
// kernel's attributes for them set: 0 where a cluster of that size has no
// place (a partitioned or capped GPU) or DSG_CLUSTERS is 0; the grid or the
// blocks beside it do the work then.  Asked once per thread, context and
// kernel (always the same blocks, threads and shared memory).
uint32_t clusters_fit(const void* kernel, uint32_t blocks, uint32_t threads, size_t smem);
template <class... P>
uint32_t clusters_fit(void (*kernel)(P...), uint32_t blocks, uint32_t threads, size_t smem) {
    return clusters_fit(reinterpret_cast<const void*>(kernel), blocks, threads, smem);
}

// One cluster.
template <class... P, class... A>
cudaError_t launch_cluster(void (*kernel)(P...), uint32_t blocks, uint32_t threads, size_t smem, cudaStream_t s,
                           A... args) {
    cudaLaunchAttribute attr;
    const cudaLaunchConfig_t cfg = cluster_config(blocks, blocks, threads, smem, s, &attr);
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}

// Graphs that one cluster of 16 blocks handles sooner than a grid does: the
// meetings are the cluster's barrier instead of a word in L2.
constexpr uint32_t kSmallBlocks = 16;

__device__ __forceinline__ uint64_t ld_relaxed_u64(const unsigned long long* p) {
    uint64_t v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ uint32_t ld_relaxed_u32(const uint32_t* p) {
    uint32_t v;
    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}

// p, as the address of the same object in block 0 of the cluster.
template <class T>
__device__ __forceinline__ T* at_block0(T* p) {
    uint64_t q;
    asm("mapa.u64 %0, %1, 0;" : "=l"(q) : "l"(reinterpret_cast<uint64_t>(p)));
    return reinterpret_cast<T*>(q);
}

// Several blocks meet, on a word that also sums a count:
// low half arrivals, high half the blocks' `mine`.  The grid's sum comes back
// with the wait, so nothing is read for it afterwards.  Two words take turns:
// a block that is already on its way to the next meeting must not add to the
// sum that a slower block is still to read (to come back to the same word it
// has to pass the other, which needs the slower block).  The words start at
// zero.  Every thread of the block calls it; thread 0's `mine` counts.  A wait
// above limit_ns records ERR_TIMEOUT and clears sm.ok, as does seeing the
// error of another block.  With one block (size == 1) it is a block barrier.
// The low half is never reset and carries into the high one every 2^32
// arrivals (a path of 2^24 vertices at eps = 0 has 2^23 rounds, each an
// arrival of every block on each word): a block that counts them modulo 2^32
// knows at which meeting that is, and takes it off.

// The counts handed in at the meeting after which a word of `blocks` blocks has
// had `arrivals` arrivals (modulo 2^32); high: the word's high half after the
// meeting before it.
__host__ __device__ __forceinline__ uint32_t meet_count(uint64_t word, uint32_t high, uint32_t arrivals,
                                                        uint32_t blocks) {
    return (uint32_t)(word >> 32) - (high + (arrivals < blocks ? 1u : 0u));
}
// A block's view of the meetings, kept by its thread 0 (the others read got and ok).
struct MeetSmem {
    uint32_t arrivals[2], high[2];  // by word, after its last meeting
    uint32_t par;                   // the next meeting's word
    uint32_t got, ok;
};
__device__ __forceinline__ void meet_init(MeetSmem& sm, uint32_t arrivals = 0) {
    sm.arrivals[0] = sm.arrivals[1] = arrivals;
    sm.high[0] = sm.high[1] = sm.par = 0;
    sm.ok = 1;
}

// The blocks that work on one graph: a co-resident grid (CL = false), or one
// thread-block cluster (CL = true: the words are in a block's shared memory,
// the wait is the cluster's barrier).
template <bool CL>
struct Team {
    uint32_t rank, size;  // this block among them, and how many (1: meet is a block barrier)
    unsigned long long (*bar)[16];
    uint32_t* err;
    uint64_t limit_ns;

    __device__ __forceinline__ uint32_t meet(uint32_t mine, MeetSmem& sm) {
        // read before the wait, written after the others may go on: the chain from the word's arrival
        // to the block's release is a subtraction and one store
        uint32_t par = 0, high = 0, arrivals = 0;
        if (threadIdx.x == 0) {
            par = sm.par;
            high = sm.high[par];
            arrivals = sm.arrivals[par] + size;
        }
        if constexpr (CL) {
            unsigned long long* word = &bar[par][0];
            if (threadIdx.x == 0 && mine) atomicAdd(word, (unsigned long long)mine);
            cluster_sync();
            if (threadIdx.x == 0) {
                const uint32_t sum = (uint32_t)ld_volatile_u64((const uint64_t*)word);
                sm.got = sum - high;
                high = sum;
            }
        } else {
            __syncthreads();
            if (threadIdx.x == 0) {
                if (size == 1) {
                    sm.got = mine;
                } else {
                    unsigned long long* word = &bar[par][0];
                    red_add_release_u64(word, (uint64_t)mine << 32 | 1ull);
                    uint64_t w;
                    uint32_t polls = 0;
                    const uint64_t t0 = global_ns();
                    while ((int32_t)((uint32_t)(w = ld_acquire_u64(word)) - arrivals) < 0) {
                        if ((++polls & 63u) == 0) {
                            if (global_ns() - t0 > limit_ns) atomicOr(err, ERR_TIMEOUT);
                            if (ld_volatile_u32(err) & ERR_TIMEOUT) {
                                sm.ok = 0;
                                break;
                            }
                        }
                    }
                    sm.got = meet_count(w, high, arrivals, size);
                    high = (uint32_t)(w >> 32);
                }
            }
        }
        __syncthreads();
        const uint32_t got = sm.got;
        if (threadIdx.x == 0) {
            sm.par = par ^ 1u;
            sm.high[par] = high;
            sm.arrivals[par] = arrivals;
        }
        return got;
    }
};

// Per-block table that combines degree decrements aimed at the same
// high-degree vertex, so a hub adjacent to thousands of failing vertices
// takes one global atomic per block and phase instead of one per edge.
// Open addressing over kAggSlots (key, count) pairs; a full probe sequence
// falls back to a direct global atomic.
constexpr uint32_t kAggBits = 11;
constexpr uint32_t kAggSlots = 1u << kAggBits;
constexpr uint32_t kAggEmpty = 0xffffffffu;

// The degree at which combining pays: a vertex takes about deg / blocks
// decrements per block, so combining helps once that is well above one, and
// while the vertices above it still fit the table (one block or a cluster per
// graph, 1,500 graphs of up to 100,000 vertices: 2.94 ms with the blocks' rule
// alone, 2.52 from degree 1,024, 2.46 from 4,096).
__device__ __forceinline__ uint32_t hot_threshold(uint32_t hot_deg, uint32_t blocks) {
    return hot_deg ? hot_deg : blocks <= 16 ? 4096u : max(4u * blocks, 1024u);
}

struct AggTable {
    uint32_t key[kAggSlots];
    uint32_t cnt[kAggSlots];
};

__device__ __forceinline__ void agg_clear(AggTable& t) {
    for (uint32_t i = threadIdx.x; i < kAggSlots; i += blockDim.x) {
        t.key[i] = kAggEmpty;
        t.cnt[i] = 0;
    }
}

// Adds one to u's slot; false if no slot could be claimed.
__device__ __forceinline__ bool agg_add(AggTable& t, uint32_t u) {
    uint32_t h = (u * 0x9E3779B1u) >> (32 - kAggBits);
#pragma unroll
    for (uint32_t i = 0; i < 4; ++i) {
        uint32_t s = (h + i) & (kAggSlots - 1);
        uint32_t prev = atomicCAS(&t.key[s], kAggEmpty, u);
        if (prev == kAggEmpty || prev == u) {
            atomicAdd(&t.cnt[s], 1u);
            return true;
        }
    }
    return false;
}

constexpr uint32_t kBatch = 4;  // entries handed to a visitor per thread and call

// Shared memory of the block-wide walker below.
template <int TB>
struct BlockTile {
    uint32_t start[TB];  // exclusive prefix of row lengths
    uint64_t beg[TB];    // row start in adj
    uint32_t v[TB];      // row owner
    uint32_t scan_tmp[33];
};

// Walk the rows of a block-private list F[lo, hi) with the whole block:
// TB rows at a time, their lengths prefix-summed, the concatenated entries
// spread evenly over all threads (a few long rows are shared by every warp).
// Same visitor contract as scan_frontier; every thread of the block calls it.
template <int TB, class Fn>
__device__ __forceinline__ void scan_block_list(const uint64_t* __restrict__ off, const uint32_t* __restrict__ adj,
                                                const uint32_t* F, uint64_t lo, uint64_t hi, BlockTile<TB>& sm,
                                                Fn& fn) {
    const uint32_t tid = threadIdx.x;
    for (uint64_t t = lo; t < hi; t += TB) {
        uint32_t cnt = (uint32_t)min((uint64_t)TB, hi - t);
        uint32_t v = 0, len = 0;
        uint64_t b = 0;
        if (tid < cnt) {
            v = F[t + tid];
            b = off[v];
            len = (uint32_t)(off[v + 1] - b);
        }
        uint32_t total;
        uint32_t st = block_excl_scan<uint32_t>(len, sm.scan_tmp, &total);
        sm.start[tid] = st;
        sm.beg[tid] = b;
        sm.v[tid] = v;
        __syncthreads();
        for (uint32_t e0 = tid; e0 < total; e0 += kBatch * TB) {
            uint32_t bu[kBatch], bv[kBatch], valid = 0;
#pragma unroll
            for (uint32_t j = 0; j < kBatch; ++j) {
                uint32_t e = e0 + j * TB;
                bu[j] = 0;
                bv[j] = 0;
                if (e < total) {
                    uint32_t a = 0, z = cnt;  // owner = last row whose start is <= e
                    while (z - a > 1) {
                        uint32_t mid = (a + z) >> 1;
                        if (sm.start[mid] <= e) a = mid; else z = mid;
                    }
                    bu[j] = ld_stream(adj + sm.beg[a] + (e - sm.start[a]));
                    bv[j] = sm.v[a];
                    valid |= 1u << j;
                }
            }
            fn(bu, bv, valid);
        }
        __syncthreads();
    }
}

// scan_block_list over rows whose starts and lengths are already known:
// row(i, v, beg, len) gives row i of cnt_all (its thread's, once; a row left
// out has length 0).
template <int TB, class Row, class Fn>
__device__ __forceinline__ void scan_block_rows(const uint32_t* __restrict__ adj, uint32_t cnt_all, Row row,
                                                BlockTile<TB>& sm, Fn& fn) {
    const uint32_t tid = threadIdx.x;
    for (uint32_t t = 0; t < cnt_all; t += TB) {
        const uint32_t cnt = min((uint32_t)TB, cnt_all - t);
        uint32_t v = 0, len = 0;
        uint64_t b = 0;
        if (tid < cnt) row(t + tid, v, b, len);
        uint32_t total;
        const uint32_t st = block_excl_scan<uint32_t>(len, sm.scan_tmp, &total);
        sm.start[tid] = st;
        sm.beg[tid] = b;
        sm.v[tid] = v;
        __syncthreads();
        auto fetch = [&](uint32_t e0, uint32_t (&bu)[kBatch], uint32_t (&bv)[kBatch]) {
            uint32_t valid = 0;
#pragma unroll
            for (uint32_t j = 0; j < kBatch; ++j) {
                const uint32_t e = e0 + j * TB;
                bu[j] = 0;
                bv[j] = 0;
                if (e < total) {
                    uint32_t a = 0, z = cnt;  // owner = last row whose start is <= e
                    while (z - a > 1) {
                        const uint32_t mid = (a + z) >> 1;
                        if (sm.start[mid] <= e) a = mid; else z = mid;
                    }
                    bu[j] = ld_stream(adj + sm.beg[a] + (e - sm.start[a]));
                    bv[j] = sm.v[a];
                    valid |= 1u << j;
                }
            }
            return valid;
        };
        for (uint32_t e0 = tid; e0 < total; e0 += kBatch * TB) {
            uint32_t bu[kBatch], bv[kBatch];
            const uint32_t valid = fetch(e0, bu, bv);
            fn(bu, bv, valid);
        }
        __syncthreads();
    }
}

// ------------------------------------------------------------- edge walker
// Visit every adjacency position j in [0, off[n]) with its row owner.
// Each warp takes one contiguous span of positions, finds the row of its first
// position by binary search over off, and then moves through the span
// kWalkU * 32 consecutive positions at a time (lane l takes l, l + 32, ...):
// pre(j) is issued for every position of a step before the owners are
// searched (so its loads overlap the search), and a lane finds each
// position's row among the next 32 row starts (one coalesced read by the
// warp): where no row is empty, as the number of starts up to the position in
// a bit map of the step (density of a web graph of 2^20 vertices 0.18 -> 0.16
// ms, row copy of a 268M-pair graph 1.76 -> 1.40 ms), else with a 5-step
// shuffle search; positions past those 32 rows (runs of
// short or empty rows) find their 32-row block from a coarse sample of the
// row starts (one coalesced read over 1,024 rows) and their row by a 5-step
// binary search inside it.
// fn(owner[], j[], pre[], valid) is called by all lanes together, bit t of
// valid set when slot t holds a position.
constexpr uint32_t kWalkU = 4;

template <class Pre, class Fn>
__device__ __forceinline__ void walk_all_entries(const uint64_t* off, uint32_t n, Pre& pre, Fn& fn) {
    const uint64_t total = off[n];
    const uint32_t lane = threadIdx.x & 31u;
    const uint64_t gw = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const uint64_t nw = ((uint64_t)gridDim.x * blockDim.x) >> 5;
    constexpr uint32_t kStep = 32 * kWalkU;
    uint64_t span = (total + nw - 1) / nw;
    span = span < 2 * kStep ? 2 * kStep : ((span + kStep - 1) / kStep * kStep);
    const uint64_t j0 = gw * span;
    if (j0 >= total) return;
    const uint64_t j1 = min(total, j0 + span);
    // row r with off[r] <= j0 < off[r + 1]
    uint32_t lo = 0, hi = n;
    while (hi - lo > 1) {
        const uint32_t mid = lo + ((hi - lo) >> 1);
        if (off[mid] <= j0) lo = mid; else hi = mid;
    }
    uint32_t r = lo;
    for (uint64_t jb = j0; jb < j1; jb += kStep) {
        uint64_t j[kWalkU];
        uint32_t pv[kWalkU], owner[kWalkU], valid = 0, done = 0;
#pragma unroll
        for (uint32_t t = 0; t < kWalkU; ++t) {
            j[t] = jb + lane + 32 * t;
            owner[t] = r;
            pv[t] = 0;
            if (j[t] < j1) {
                valid |= 1u << t;
                pv[t] = pre(j[t]);
            }
        }
        done = ~valid & ((1u << kWalkU) - 1);
        {
            const uint32_t base = r;
            const uint32_t idx = base + 1 + lane;
            // row starts relative to the step (none lies before it: row r holds the position before
            // jb or jb itself), clamped to what a position of the step can be compared with
            const uint32_t w = idx < n ? (uint32_t)min(off[idx] - jb, (uint64_t)kStep) : kStep;
            const uint32_t before = __shfl_up_sync(kFullMask, w, 1);
            // a position's row is base + the starts at or below it
            uint32_t c[kWalkU];
            if (!__any_sync(kFullMask, lane > 0 && w == before && w < kStep)) {
                // no empty row among them: the starts are distinct, one bit each in a map of the
                // step's positions, and the count is that of the bits up to the position (4
                // reductions and a few population counts instead of 20 shuffles)
                uint32_t below = 0;
#pragma unroll
                for (uint32_t t = 0; t < kWalkU; ++t) {
                    const uint32_t m = __reduce_or_sync(kFullMask, (w >> 5) == t ? 1u << (w & 31u) : 0u);
                    c[t] = below + __popc(m & (0xffffffffu >> (31u - lane)));
                    below += __popc(m);
                }
            } else {
                const uint32_t w31 = __shfl_sync(kFullMask, w, 31);
#pragma unroll
                for (uint32_t t = 0; t < kWalkU; ++t) {
                    const uint32_t e = lane + 32 * t;
                    c[t] = 0;
#pragma unroll
                    for (uint32_t step = 16; step > 0; step >>= 1) {
                        const uint32_t wv = __shfl_sync(kFullMask, w, c[t] + step - 1);
                        if (wv <= e) c[t] += step;
                    }
                    if (c[t] == 31 && w31 <= e) c[t] = 32;
                }
            }
#pragma unroll
            for (uint32_t t = 0; t < kWalkU; ++t) {
                if (!(done >> t & 1u) && c[t] < 32) {
                    owner[t] = base + c[t];
                    done |= 1u << t;
                }
            }
            // positions past the window (runs of short or empty rows): every
            // pending position lies at or above off[b].  Lane l reads
            // off[b + S l] (one coalesced read; S rows apart), a position's
            // count of those <= it names the S-row block holding its row, and
            // a binary search over that block's row starts (log2 S steps, all
            // lanes and slots at once) places it.  Positions beyond the 32
            // blocks move b up by 31 S; a pass that places nothing widens S;
            // after 64 passes a plain binary search places what is left.
            uint64_t b = (uint64_t)base + 32, S = 32;
            for (uint32_t pass = 0; __any_sync(kFullMask, done != (1u << kWalkU) - 1); ++pass) {
                if (pass == 64) {
                    // rows spread very far apart: a binary search over [b, n) places the rest
#pragma unroll
                    for (uint32_t t = 0; t < kWalkU; ++t) {
                        if (done >> t & 1u) continue;
                        uint64_t lo = b, hi = n;  // off[b] <= j < off[n]
                        while (hi - lo > 1) {
                            const uint64_t mid = lo + ((hi - lo) >> 1);
                            if (off[mid] <= j[t]) lo = mid; else hi = mid;
                        }
                        owner[t] = (uint32_t)lo;
                        done |= 1u << t;
                    }
                    break;
                }
                const uint64_t cidx = b + S * lane;
                const uint64_t cw = off[cidx < n ? cidx : n];  // off[n] = total: above every position
                const uint64_t cw31 = __shfl_sync(kFullMask, cw, 31);
                uint32_t placed = 0;
#pragma unroll
                for (uint32_t t = 0; t < kWalkU; ++t) {
                    uint32_t c = 0;
#pragma unroll
                    for (uint32_t step = 16; step > 0; step >>= 1) {
                        const uint64_t wv = __shfl_sync(kFullMask, cw, c + step - 1);
                        if (wv <= j[t]) c += step;
                    }
                    if (c == 31 && cw31 <= j[t]) c = 32;
                    if (!(done >> t & 1u) && c < 32) {
                        // off[b + S (c-1)] <= j < off[min(b + S c, n)]; c >= 1 since off[b] <= j
                        uint64_t lo = b + S * (c - 1), hi = b + S * c;
                        if (hi > n) hi = n;
                        while (hi - lo > 1) {
                            const uint64_t mid = lo + ((hi - lo) >> 1);
                            if (off[mid] <= j[t]) lo = mid; else hi = mid;
                        }
                        owner[t] = (uint32_t)lo;
                        done |= 1u << t;
                        ++placed;
                    }
                }
                // what is still pending lies at or above off[b + 31 S]
                b += 31 * S;
                if (!__any_sync(kFullMask, placed != 0)) S *= 32;
            }
        }
        fn(owner, j, pv, valid);
        // next step starts at or after the row of this step's last position
        const uint32_t last = valid >> (kWalkU - 1) & 1u ? owner[kWalkU - 1] : r;
        r = __shfl_sync(kFullMask, last, 31);
        if (!__shfl_sync(kFullMask, valid >> (kWalkU - 1) & 1u, 31)) break;  // span's final step
    }
}

}  // namespace dsg
