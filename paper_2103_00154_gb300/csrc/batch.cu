// Batched solve: many independent graphs in one persistent launch.
//
// The graphs are packed as one concatenated CSR: graph g owns global vertex
// slots [vtx_base[g], vtx_base[g+1]); its row for local vertex v is
// adj[off[vtx_base[g] + v] .. off[vtx_base[g] + v + 1]) and holds LOCAL ids.
// Each block pulls the next graph from a device counter (graphs are queued
// largest first, so the long ones start early) and solves it alone: the
// Bahmani peel of Algorithm 1 and, when asked, the core numbers of
// Algorithm 2's first phase.  A round's (or level's) barrier is the block's
// __syncthreads, so a graph costs no grid-wide synchronisation.
// Graphs that would keep one block busy long after the others are done get a
// thread-block cluster each instead, from a queue of their own.  Both run the
// body of the grid-wide peel, the clusters that of the bitwise core-number
// search too, with the block's or the cluster's barrier between rounds and
// waves, on a slab of scratch per team.
#include <string.h>

#include <algorithm>
#include <mutex>
#include <vector>

#include "core_split.cuh"
#include "dsg_batch.cuh"
#include "dsg_common.cuh"
#include "dsg_kernels.cuh"
#include "peel_body.cuh"

namespace dsg {

// Algorithm 2, first phase, on one graph by one block: level k collects the
// remaining vertices of degree k, then drains them (atomicSub on every
// neighbour; a == k+1 joins the level; a <= k is undone, so a vertex already
// at or below k never reads k+1 again); the level's frontier is one FIFO in
// global memory with a shared-memory cursor.  One block alone reads every row
// once here; the bitwise search reads it about seven times, which pays only
// where its waves are spread over several blocks (600 graphs of 1,000 to
// 100,000 vertices with core numbers: 7.2 ms against 14.1 ms).
template <int TB>
struct LevelSmem {
    BlockTile<TB> tile;
    uint32_t scan_tmp[33];
    uint32_t cursor;
};

template <int TB>
__device__ void kcore_block(uint32_t n, const uint64_t* off, const uint32_t* adj, uint32_t* deg, uint32_t* rem_a,
                            uint32_t* rem_b, uint32_t* Q, LevelSmem<TB>& sm) {
    const uint32_t tid = threadIdx.x;
    uint32_t mn = 0xffffffffu;
    for (uint32_t v = tid; v < n; v += TB) {
        uint32_t d = (uint32_t)(off[v + 1] - off[v]);
        deg[v] = d;
        mn = min(mn, d);
    }
    uint32_t k = block_min_u32(mn, sm.scan_tmp);
    const uint32_t* rem = nullptr;
    uint32_t* rem_next = rem_a;
    uint32_t rem_n = n, visited = 0;
    if (tid == 0) sm.cursor = 0;  // FIFO cursor
    __syncthreads();
    for (;;) {
        uint32_t kept = 0, mnext = 0xffffffffu;
        for (uint32_t t = 0; t < rem_n; t += TB) {
            uint32_t i = t + tid;
            bool keep = false;
            uint32_t v = 0;
            if (i < rem_n) {
                v = rem ? rem[i] : i;
                uint32_t d = deg[v];
                if (d == k) Q[atomicAdd(&sm.cursor, 1u)] = v;
                else if (d > k) {
                    keep = true;
                    mnext = min(mnext, d);
                }
            }
            uint32_t tot;
            uint32_t pre = block_excl_scan<uint32_t>(keep ? 1u : 0u, sm.scan_tmp, &tot);
            if (keep) rem_next[kept + pre] = v;
            kept += tot;
        }
        __syncthreads();
        uint32_t q_lo = visited, q_hi = sm.cursor;
        __syncthreads();
        while (q_lo < q_hi) {
            // every neighbour loses one degree at once (no read first); one
            // already at or below k gets it back
            auto visit = [&](const uint32_t* u, const uint32_t* v, uint32_t valid) {
                uint32_t need = 0, old[kBatch];
#pragma unroll
                for (uint32_t j = 0; j < kBatch; ++j) {
                    if (!(valid >> j & 1u) || u[j] == v[j]) continue;
                    old[j] = atomicSub(&deg[u[j]], 1u);
                    need |= 1u << j;
                }
#pragma unroll
                for (uint32_t j = 0; j < kBatch; ++j) {
                    if (!(need >> j & 1u)) continue;
                    if (old[j] == k + 1) Q[atomicAdd(&sm.cursor, 1u)] = u[j];
                    else if (old[j] <= k) atomicAdd(&deg[u[j]], 1u);
                    else mnext = min(mnext, old[j] - 1);
                }
            };
            scan_block_list<TB>(off, adj, Q, q_lo, q_hi, sm.tile, visit);
            q_lo = q_hi;
            q_hi = sm.cursor;
            __syncthreads();
        }
        visited = q_hi;
        if (visited >= n) break;
        k = block_min_u32(mnext, sm.scan_tmp);
        if (k == 0xffffffffu) break;
        rem_n = kept;
        rem = rem_next;
        rem_next = (rem_next == rem_a) ? rem_b : rem_a;
    }
    __syncthreads();
}

// Blocks of a cluster: 16 while there are at most kFewGraphs graphs (8 graphs of
// 100,000 to 300,000 vertices with core numbers 2.9 against 4.5 ms), else 8,
// of which 15 clusters fit the GPU against 7 (60 graphs to 300,000 vertices
// 5.0 against 5.6 ms).
constexpr uint32_t kClusterBlocks = 8, kClusterBlocksFew = 16, kFewGraphs = 14;
constexpr uint32_t kClusterTB = 1024;

// A team's scratch for a graph of n vertices and e row entries: offsets and
// size.  The peel's arrays, a block's level lists (the peel's first three) and
// the search's share the space.  Larger graphs need no less of anything.
constexpr uint32_t kBatchChunk = 256;  // entries of a row piece of the peel
struct SlabLayout {
    uint64_t listA, listB, items, map, peel_end;
    uint64_t ds, key, pieces, queue, search_end;
    uint64_t cap;  // row pieces of the search
};
__host__ __device__ inline SlabLayout slab_layout(uint64_t n, uint64_t e) {
    auto up = [](uint64_t bytes) { return (bytes + 255) & ~uint64_t(255); };
    SlabLayout l = {};
    l.listA = up(4 * n);  // after the states
    l.listB = 2 * l.listA;
    l.items = 3 * l.listA;
    l.map = l.items + up(8 * (n + e / kBatchChunk + 1));
    l.peel_end = l.map + up((n + 15) / 16 * 4);
    l.cap = n + e / kPiece + 1;
    l.ds = l.listA;  // after the degrees
    l.key = l.listB;
    l.pieces = l.key + up(4 * ((n + 63) & ~uint64_t(63)) * split_key_buffers(e));
    l.queue = l.pieces + up(16 * l.cap);
    l.search_end = l.queue + up(16 * l.cap);
    return l;
}

struct Slab {
    uint64_t at;    // its place in the scratch
    uint64_t n, e;  // the graphs it is for
};

struct BatchKernelArgs {
    BatchArgs b;
    unsigned char* scratch;  // the error word, the table of the slabs, the slabs
    const Slab* slabs;       // by the order in which the teams start
};

template <int TB>
struct BatchSmem {
    union {
        PeelSmem<TB> peel;
        SplitSmem<TB> split;
        LevelSmem<TB> level;
    };
    union {  // the running graph's arguments: read from here, not held in registers
        PeelArgs pargs;
        SplitArgs sargs;
    };
    PeelCtl pctl;
    SplitCtl sctl;
    uint32_t item, slot;
    unsigned char* slab;  // the team's, once it has taken a graph ...
    SlabLayout lay;       // ... and its layout
};

// The two bodies as functions of their own: inlined into one kernel they spill
// each other's registers.
template <int TB, uint32_t size>
__device__ __noinline__ PeelOut team_peel(const PeelArgs& a, PeelSmem<TB>& sm, uint32_t rank) {
    return peel_body<TB, (size > 1)>(a, Team<(size > 1)>{rank, size, a.ctl->bar, &a.ctl->err, 0}, sm);
}
template <int TB, uint32_t size>
__device__ __noinline__ void team_split(const SplitArgs& a, SplitSmem<TB>& sm, uint32_t rank) {
    split_body<TB, (size > 1)>(a, Team<(size > 1)>{rank, size, a.ctl->bar, &a.ctl->err, 0}, sm);
}

// A team -- one block, or (CL) a cluster -- takes graphs from
// the queue until none is left: Algorithm 1, then the core numbers if asked.
// What bounds it: as the grid-wide kernels, L2 gathers in the wide waves and
// dependent round trips in the thin ones, but a meeting is the block's barrier
// or the cluster's and two accesses to a neighbour's shared memory.
template <int TB, uint32_t size>  // size: blocks of the team
__global__ void __launch_bounds__(TB, 1024 / TB) batch_kernel(BatchKernelArgs c) {
    constexpr bool CL = size > 1;
    __shared__ BatchSmem<TB> sm;
    const BatchArgs& b = c.b;
    const uint32_t tid = threadIdx.x, rank = CL ? cluster_rank() : 0;
    PeelCtl* const pctl = CL ? at_block0(&sm.pctl) : &sm.pctl;
    SplitCtl* const sctl = CL ? at_block0(&sm.sctl) : &sm.sctl;
    uint32_t* const item0 = CL ? at_block0(&sm.item) : &sm.item;
    uint32_t* const slot0 = CL ? at_block0(&sm.slot) : &sm.slot;
    if (tid == 0) sm.slab = nullptr;
    uint32_t* const err = reinterpret_cast<uint32_t*>(c.scratch);
    auto sync = [] {
        if constexpr (CL) cluster_sync();
        else __syncthreads();
    };
    for (;;) {
        if (rank == 0) {
            static_assert(sizeof(PeelCtl) % 4 == 0 && sizeof(SplitCtl) % 4 == 0, "cleared word by word");
            for (uint32_t i = tid; i < sizeof(PeelCtl) / 4; i += TB) reinterpret_cast<uint32_t*>(&sm.pctl)[i] = 0;
            for (uint32_t i = tid; i < sizeof(SplitCtl) / 4; i += TB) reinterpret_cast<uint32_t*>(&sm.sctl)[i] = 0;
            if (tid == 0) {
                // a team's first graph comes with its place among the teams that have started: no more
                // have than graphs are taken, so this graph and all it takes later are no earlier in the
                // order than that place, which the slab is sized for
                const unsigned long long t = atomicAdd(b.next, sm.slab ? 1ull : 1ull << 32 | 1ull);
                sm.item = min((uint32_t)t, b.G);
                sm.slot = (uint32_t)(t >> 32);
            }
        }
        sync();
        const uint32_t item = ld_volatile_u32(item0);
        if (item >= b.G) break;
        const uint32_t g = b.order[item];
        const uint64_t vb = b.slot[g];
        const uint32_t n = b.gn[g];
        const uint64_t* off = b.goff[g];
        if (tid == 0) {
            PeelArgs& a = sm.pargs;
            if (!sm.slab) {
                const Slab z = c.slabs[ld_volatile_u32(slot0)];
                sm.slab = c.scratch + z.at;
                sm.lay = slab_layout(z.n, z.e);
            }
            const SlabLayout& l = sm.lay;
            unsigned char* const slab = sm.slab;
            a.n = n;
            a.m = n ? (off[n] - off[0]) / 2 : 0;
            a.p = b.p[g];
            a.q = b.q[g];
            a.off = off;
            a.adj = b.gadj[g];
            a.st = reinterpret_cast<uint32_t*>(slab);
            a.listA = reinterpret_cast<uint32_t*>(slab + l.listA);
            a.listB = reinterpret_cast<uint32_t*>(slab + l.listB);
            a.items = reinterpret_cast<uint64_t*>(slab + l.items);
            a.map = reinterpret_cast<uint32_t*>(slab + l.map);
            a.candA = a.candB = nullptr;
            a.hist_S = a.hist_E = nullptr;
            a.hist_cap = ~0ull;
            a.ctl = pctl;
            a.limit_ns = 0;
            a.chunk_len = kBatchChunk;
            a.hot_deg = b.hot_deg;
            a.trace = nullptr;
            a.trace_cap = 0;
            a.r0 = a.S0 = a.E0 = a.best_round0 = a.best_E0 = a.best_V0 = a.max_rounds = a.arrivals0 = 0;
        }
        __syncthreads();
        {
            const PeelOut o = team_peel<TB, size>(sm.pargs, sm.peel, rank);
            if (rank == 0 && tid == 0) {
                b.res[4 * (uint64_t)g + 0] = n ? o.best_E : 0;
                b.res[4 * (uint64_t)g + 1] = n ? o.best_V : 0;
                b.res[4 * (uint64_t)g + 2] = o.rounds;
                b.res[4 * (uint64_t)g + 3] = o.best_round;
                if (b.stats) {
                    atomicAdd(&b.stats[0], pctl->tested);
                    atomicAdd(&b.stats[1], pctl->dec);
                    atomicAdd(&b.stats[2], (unsigned long long)(2 * sm.pargs.m));
                }
                if (pctl->err) atomicOr(err, pctl->err);
            }
            if (b.out_set) {
                const uint32_t* st = sm.pargs.st;
                for (uint32_t v = rank * TB + tid; v < n; v += size * TB)
                    b.out_set[vb + v] = (__ldcg(st + v) & ~kDead) > o.best_round ? 1 : 0;
            }
        }
        sync();  // the peel's arrays and arguments are read before the search takes their place
        if (b.core && (!b.want_core || b.want_core[g]) && n) {
            if constexpr (CL) {
                if (tid == 0) {
                    SplitArgs& a = sm.sargs;
                    const SlabLayout& l = sm.lay;
                    unsigned char* const slab = sm.slab;
                    a.r = n;
                    a.lo = 0;
                    a.off = off;
                    a.adj = b.gadj[g];
                    a.rid = nullptr;
                    a.d = reinterpret_cast<uint32_t*>(slab);
                    a.ds = reinterpret_cast<uint32_t*>(slab + l.ds);
                    a.key = reinterpret_cast<uint32_t*>(slab + l.key);
                    a.kstride = ((uint64_t)n + 63) & ~uint64_t(63);
                    a.pieces = reinterpret_cast<uint4*>(slab + l.pieces);
                    a.queue = reinterpret_cast<uint4*>(slab + l.queue);
                    a.cap = l.cap;
                    a.core = b.core + vb;
                    a.ctl = sctl;
                    a.limit_ns = 0;
                    a.trace = nullptr;
                    a.trace_cap = 0;
                }
                __syncthreads();
                team_split<TB, size>(sm.sargs, sm.split, rank);
                sync();  // its keys are read, its counters written
                if (rank == 0 && tid == 0 && sctl->err) atomicOr(err, sctl->err);
                __syncthreads();
            } else {
                const SlabLayout& l = sm.lay;
                unsigned char* const slab = sm.slab;
                kcore_block<TB>(n, off, b.gadj[g], b.core + vb, reinterpret_cast<uint32_t*>(slab),
                                reinterpret_cast<uint32_t*>(slab + l.listA),
                                reinterpret_cast<uint32_t*>(slab + l.listB), sm.level);
            }
        }
    }
    sync();  // no block leaves while another reads block 0's shared memory
}

// Scratch for `teams` teams over the graphs of the launch (fewer if theirs
// would take more than scratch_max bytes or cannot be had), cleared error word.
static cudaError_t batch_slabs(BatchKernelArgs& c, const BatchSizes& sizes, bool search, uint64_t* teams,
                               size_t scratch_max, cudaStream_t s, void** slabs) {
    const uint32_t G = c.b.G;
    std::vector<Slab> all(*teams);  // by place: for the most vertices and the most entries from there on
    std::vector<uint64_t> bytes(*teams);
    uint32_t n = 0;
    uint64_t e = 0;
    for (uint32_t k = G; k-- > 0;) {
        n = std::max(n, sizes.n[k]);
        e = std::max(e, sizes.e[k]);
        if (k < *teams) {
            all[k] = {0, n, e};
            const SlabLayout l = slab_layout(n, e);
            bytes[k] = c.b.core && search ? std::max(l.peel_end, l.search_end) : l.peel_end;
            // (the kernel's time depends on the addresses by a few percent; over seven places of the
            // allocation each, 1,500 graphs of up to 100,000 vertices took 2.11 ms with slabs packed
            // tightly, 2.07 in steps of 64 KB and 2.11 in steps of 2 MB)
            if (bytes[k] >= 1u << 16) bytes[k] = (bytes[k] + 0xffff) & ~uint64_t(0xffff);
        }
    }
    uint64_t t = 1, total = bytes[0];
    while (t < *teams && total + bytes[t] <= scratch_max) total += bytes[t++];
    constexpr uint64_t kHead = 256;  // the error word's share
    void* p = nullptr;
    for (;;) {
        uint64_t at = (kHead + t * sizeof(Slab) + 255) & ~uint64_t(255);
        for (uint64_t k = 0; k < t; at += bytes[k++]) all[k].at = at;
        const cudaError_t err = dev_alloc(&p, at, s);
        if (err == cudaSuccess) break;
        if (err != cudaErrorMemoryAllocation || t == 1) return err;
        cudaGetLastError();  // handled here
        t = (t + 1) / 2;
    }
    *slabs = p;
    *teams = t;
    c.scratch = static_cast<unsigned char*>(p);
    c.slabs = reinterpret_cast<const Slab*>(c.scratch + kHead);
    std::vector<unsigned char> head(kHead + t * sizeof(Slab), 0);
    memcpy(head.data() + kHead, all.data(), t * sizeof(Slab));
    return cudaMemcpyAsync(p, head.data(), head.size(), cudaMemcpyHostToDevice, s);
}

template <int TB>
static uint32_t slots_tb() {
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, batch_kernel<TB, 1>, TB, 0) != cudaSuccess ||
        per_sm < 1)
        per_sm = 1;
    return (uint32_t)per_sm * (uint32_t)dev_info().sms;
}

// Block slots of the block-per-graph kernel at `block` threads.
static uint32_t batch_slots(uint32_t block) {
    switch (block) {
        case 256: return slots_tb<256>();
        case 1024: return slots_tb<1024>();
        default: return slots_tb<512>();
    }
}

uint32_t batch_slots_for(uint32_t block) { return batch_slots(block); }

cudaError_t batch_launch(const BatchArgs& a, const BatchSizes& sizes, size_t scratch_max, cudaStream_t s, void** slabs,
                         uint32_t block, uint32_t max_grid) {
    BatchKernelArgs c = {};
    c.b = a;
    uint64_t teams = std::min<uint64_t>(batch_slots(block), a.G);
    if (max_grid) teams = std::min<uint64_t>(teams, max_grid);
    cudaError_t e = batch_slabs(c, sizes, false, &teams, scratch_max, s, slabs);
    if (e != cudaSuccess) return e;
    const uint32_t grid = (uint32_t)teams;
    LaunchScope ls("batch_solve", s);
    switch (block) {
        case 256: batch_kernel<256, 1><<<grid, 256, 0, s>>>(c); break;
        case 1024: batch_kernel<1024, 1><<<grid, 1024, 0, s>>>(c); break;
        default: batch_kernel<512, 1><<<grid, 512, 0, s>>>(c); break;
    }
    return cudaGetLastError();
}

cudaError_t batch_cluster_launch(const BatchArgs& a, const BatchSizes& sizes, size_t scratch_max, cudaStream_t s,
                                 void** slabs, uint32_t max_sms) {
    BatchKernelArgs c = {};
    c.b = a;
    const uint32_t fit_few =
        a.G <= kFewGraphs ? clusters_fit(batch_kernel<kClusterTB, kClusterBlocksFew>, kClusterBlocksFew, kClusterTB, 0) : 0;
    const uint32_t size = fit_few ? kClusterBlocksFew : kClusterBlocks;
    auto* const kernel = fit_few ? batch_kernel<kClusterTB, kClusterBlocksFew> : batch_kernel<kClusterTB, kClusterBlocks>;
    uint64_t teams = fit_few ? fit_few : clusters_fit(batch_kernel<kClusterTB, kClusterBlocks>, kClusterBlocks, kClusterTB, 0);
    if (teams == 0) return cudaErrorInvalidConfiguration;  // (batch_clusters gives no graph to clusters then)
    teams = std::min<uint64_t>(teams, a.G);
    if (max_sms) teams = std::min<uint64_t>(teams, std::max<uint32_t>(1, max_sms / size));
    const cudaError_t e = batch_slabs(c, sizes, true, &teams, scratch_max, s, slabs);
    if (e != cudaSuccess) return e;
    cudaLaunchAttribute attr;
    const cudaLaunchConfig_t cfg = cluster_config((uint32_t)teams * size, size, kClusterTB, 0, s, &attr);
    LaunchScope ls("batch_clusters", s);
    return cudaLaunchKernelEx(&cfg, kernel, c);
}

// More than a quarter of the batch (8 graphs of 100,000 to 300,000 vertices: all
// in clusters 4.4 ms, three of them on the whole GPU first 5.7), or too large
// for the search to take it whole.
bool batch_takes_grid(uint64_t work, uint32_t n, uint64_t total) {
    return (work > (1u << 20) && work > total / 4) || n > kTailWhole * 65536;
}

// More than twice a block's share of the batch (it would be the last to end; at
// one share the clusters hold SMs that the blocks use better: 600 graphs with
// core numbers 7.2 against 9.2 ms) and more than 2^17 units of work (40 graphs
// of 3,000 to 35,000 vertices: 0.44 ms against 0.53 from 2^15 and 0.69 from
// 2^18).
uint32_t batch_clusters(const uint64_t* work, uint32_t G, uint64_t total) {
    const uint64_t share = total / batch_slots(512);
    uint32_t k = 0;
    if (G == 0 || !clusters_fit(batch_kernel<kClusterTB, kClusterBlocks>, kClusterBlocks, kClusterTB, 0)) return 0;
    while (k < G && work[k] > (1u << 17) && work[k] > 2 * share) ++k;
    return k;
}

// want_core[g] read from host or device memory.
static bool host_want_core(const uint8_t* want_core, uint32_t g, cudaStream_t s) {
    uint8_t w = 1;
    if (copy_any(&w, want_core + g, 1, s) != cudaSuccess) return true;
    cudaStreamSynchronize(s);
    return w != 0;
}

template <class T>
static cudaError_t to_device(Scratch& sc, const T* src, size_t count, cudaStream_t s, const T** out) {
    if (!src || count == 0) {
        *out = src;
        return cudaSuccess;
    }
    if (is_device_ptr(src)) {
        *out = src;
        return cudaSuccess;
    }
    T* d;
    cudaError_t e = sc.get(&d, count);
    if (e != cudaSuccess) return e;
    e = copy_any(d, src, count * sizeof(T), s);
    *out = d;
    return e;
}

// ends[g] = off[vb[g]] for g = 0..G: every graph's first adjacency offset
// (and the batch's end), gathered for one copy to the host.
__global__ void gather_ends_kernel(const uint64_t* __restrict__ off, const uint64_t* __restrict__ vb, uint32_t G1,
                                   uint64_t* __restrict__ ends) {
    const uint32_t g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g < G1) ends[g] = off[vb[g]];
}

// A second stream and two events for a call, taken from those that calls of the
// same context have given back: as many exist as calls ran at once, however
// many threads made them.
struct BatchSide {
    unsigned long long ctx = 0;
    cudaStream_t s = nullptr;
    cudaEvent_t fork = nullptr, join = nullptr;
};
static std::mutex g_side_mu;
static std::vector<BatchSide> g_sides;  // not in use

class SideGuard {
  public:
    ~SideGuard() {
        if (!b_.s) return;
        std::lock_guard<std::mutex> lk(g_side_mu);
        g_sides.push_back(b_);
    }
    cudaError_t take() {
        unsigned long long ctx = current_ctx_id();
        int dev = 0;
        if (!ctx && cudaGetDevice(&dev) == cudaSuccess) ctx = ~(unsigned long long)dev;  // no ids: one context a device
        {
            std::lock_guard<std::mutex> lk(g_side_mu);
            for (size_t i = 0; i < g_sides.size(); ++i) {
                if (g_sides[i].ctx != ctx) continue;
                b_ = g_sides[i];
                g_sides.erase(g_sides.begin() + i);
                return cudaSuccess;
            }
        }
        BatchSide b;
        b.ctx = ctx;
        cudaError_t e = cudaStreamCreateWithFlags(&b.s, cudaStreamNonBlocking);
        if (e == cudaSuccess) e = cudaEventCreateWithFlags(&b.fork, cudaEventDisableTiming);
        if (e == cudaSuccess) e = cudaEventCreateWithFlags(&b.join, cudaEventDisableTiming);
        if (e == cudaSuccess) {
            b_ = b;
            return e;
        }
        if (b.fork) cudaEventDestroy(b.fork);
        if (b.s) cudaStreamDestroy(b.s);
        return e;
    }
    explicit operator bool() const { return b_.s != nullptr; }
    const BatchSide* operator->() const { return &b_; }

  private:
    BatchSide b_;
};

}  // namespace dsg

using namespace dsg;

extern "C" dsg_status dsg_batch_solve(const dsg_batch* b, dsg_batch_result* r, void* stream) {
    clear_error();
    DSG_CHECK_ARG(b && r, "batch / result is NULL");
    DSG_CHECK_ARG(b->vtx_base && b->off && b->eps_num && b->eps_den, "batch arrays are NULL");
    const uint32_t G = b->num_graphs;
    cudaStream_t s = (cudaStream_t)stream;
    if (G == 0) return DSG_OK;
    // host copies of the small per-graph arrays (ordering, checks)
    std::vector<uint64_t> vb(G + 1);
    std::vector<uint32_t> hp(G), hq(G);
    DSG_TRY_CUDA(copy_any(vb.data(), b->vtx_base, (G + 1) * sizeof(uint64_t), s));
    DSG_TRY_CUDA(copy_any(hp.data(), b->eps_num, G * sizeof(uint32_t), s));
    DSG_TRY_CUDA(copy_any(hq.data(), b->eps_den, G * sizeof(uint32_t), s));
    DSG_TRY_CUDA(cudaStreamSynchronize(s));
    DSG_CHECK_ARG(vb[0] == 0, "vtx_base[0] must be 0");
    for (uint32_t g = 0; g < G; ++g) {
        DSG_CHECK_ARG(vb[g + 1] >= vb[g], "vtx_base must not decrease");
        DSG_CHECK_ARG(vb[g + 1] - vb[g] < 0x80000000ull, "a graph has 2^31 vertices or more");
        DSG_CHECK_ARG(hq[g] != 0, "eps_den must be positive");
    }
    const uint64_t N = vb[G];
    uint64_t total = 0;
    DSG_TRY_CUDA(copy_any(&total, b->off + N, sizeof(uint64_t), s));
    DSG_TRY_CUDA(cudaStreamSynchronize(s));
    DSG_CHECK_ARG(total == 0 || b->adj, "adj is NULL");
    Scratch sc(s);
    const uint64_t* d_off;
    DSG_TRY_CUDA(to_device(sc, b->off, N + 1, s, &d_off));
    // largest first (by adjacency length, then vertices): every graph's first offset, gathered
    // on the device and copied in one piece
    std::vector<uint64_t> hoff_ends(G + 1);
    {
        const uint64_t* d_vb;
        DSG_TRY_CUDA(to_device(sc, vb.data(), G + 1, s, &d_vb));
        uint64_t* d_ends;
        DSG_TRY_CUDA(sc.get(&d_ends, G + 1));
        {
            LaunchScope ls("batch_ends", s);
            gather_ends_kernel<<<(G + 1 + 255) / 256, 256, 0, s>>>(d_off, d_vb, G + 1, d_ends);
        }
        DSG_TRY_CUDA(cudaGetLastError());
        DSG_TRY_CUDA(cudaMemcpyAsync(hoff_ends.data(), d_ends, (G + 1) * sizeof(uint64_t), cudaMemcpyDeviceToHost, s));
        DSG_TRY_CUDA(cudaStreamSynchronize(s));
    }
    std::vector<uint32_t> order(G);
    for (uint32_t g = 0; g < G; ++g) order[g] = g;
    auto work = [&](uint32_t x) { return (hoff_ends[x + 1] - hoff_ends[x]) + (vb[x + 1] - vb[x]); };
    std::stable_sort(order.begin(), order.end(), [&](uint32_t x, uint32_t y) { return work(x) > work(y); });
    BatchArgs a;
    a.G = G;
    const uint32_t* d_adj;
    DSG_TRY_CUDA(to_device(sc, b->adj, total, s, &d_adj));
    DSG_TRY_CUDA(to_device(sc, b->eps_num, G, s, &a.p));
    DSG_TRY_CUDA(to_device(sc, b->eps_den, G, s, &a.q));
    DSG_TRY_CUDA(to_device(sc, b->want_core, b->want_core ? G : 0, s, &a.want_core));
    {
        std::vector<const uint64_t*> hoffp(G);
        std::vector<const uint32_t*> hadjp(G);
        std::vector<uint32_t> hn(G);
        for (uint32_t g = 0; g < G; ++g) {
            hoffp[g] = d_off + vb[g];
            hadjp[g] = d_adj;
            hn[g] = (uint32_t)(vb[g + 1] - vb[g]);
        }
        const uint64_t** t_off;
        const uint32_t** t_adj;
        uint64_t* t_slot;
        uint32_t* t_n;
        DSG_TRY_CUDA(sc.get(&t_off, G));
        DSG_TRY_CUDA(sc.get(&t_adj, G));
        DSG_TRY_CUDA(sc.get(&t_slot, G));
        DSG_TRY_CUDA(sc.get(&t_n, G));
        DSG_TRY_CUDA(copy_any(t_off, hoffp.data(), G * sizeof(void*), s));
        DSG_TRY_CUDA(copy_any(t_adj, hadjp.data(), G * sizeof(void*), s));
        DSG_TRY_CUDA(copy_any(t_slot, vb.data(), G * sizeof(uint64_t), s));
        DSG_TRY_CUDA(copy_any(t_n, hn.data(), G * sizeof(uint32_t), s));
        a.goff = t_off;
        a.gadj = t_adj;
        a.slot = t_slot;
        a.gn = t_n;
        // the tables live in stream-ordered scratch: keep the host vectors alive until the copies ran
        DSG_TRY_CUDA(cudaStreamSynchronize(s));
    }
    bool core_direct = r->core && is_device_ptr(r->core);
    bool set_direct = r->out_set && is_device_ptr(r->out_set);
    a.core = nullptr;
    if (r->core) {
        if (core_direct) {
            a.core = r->core;
        } else {
            // start from the caller's values so graphs without core numbers stay untouched
            DSG_TRY_CUDA(sc.get(&a.core, N ? N : 1));
            DSG_TRY_CUDA(copy_any(a.core, r->core, N * sizeof(uint32_t), s));
        }
    }
    a.out_set = nullptr;
    if (r->out_set) {
        if (set_direct) a.out_set = r->out_set;
        else DSG_TRY_CUDA(sc.get(&a.out_set, N ? N : 1));
    }
    DSG_TRY_CUDA(sc.get(&a.res, 4 * (size_t)G));
    DSG_TRY_CUDA(sc.get(&a.next, 1));
    DSG_TRY_CUDA(cudaMemsetAsync(a.next, 0, sizeof(unsigned long long), s));
    uint64_t total_work = 0;
    for (uint32_t g = 0; g < G; ++g) total_work += work(g);
    const Tuning tu = tuning_for_batch(G, total_work);
    a.hot_deg = tu.hot_deg;
    const uint32_t block = tu.batch_block ? tu.batch_block : 512;
    unsigned long long* d_stats = nullptr;
    if (r->stats) {
        DSG_TRY_CUDA(sc.get(&d_stats, 3));
        DSG_TRY_CUDA(cudaMemsetAsync(d_stats, 0, 3 * sizeof(unsigned long long), s));
    }
    a.stats = d_stats;
    uint64_t big_sum_S = 0, big_dec = 0, big_entries = 0;
    // which graphs run on the whole GPU one after the other, which get a cluster, which a block
    uint32_t nbig = 0, ncl = 0;
    if (tu.batch_split) {
        while (nbig < G && work(order[nbig]) > tu.batch_split) ++nbig;
    } else {
        // (one of many vertices may stand anywhere in the order)
        nbig = (uint32_t)(std::stable_partition(order.begin(), order.end(),
                                                [&](uint32_t x) {
                                                    return batch_takes_grid(work(x), (uint32_t)(vb[x + 1] - vb[x]),
                                                                            total_work);
                                                }) -
                          order.begin());
    }
    std::vector<uint32_t> on(G);  // vertices and row entries, in the order of the launches
    std::vector<uint64_t> oe(G), ow(G);
    for (uint32_t i = 0; i < G; ++i) {
        on[i] = (uint32_t)(vb[order[i] + 1] - vb[order[i]]);
        oe[i] = hoff_ends[order[i] + 1] - hoff_ends[order[i]];
        ow[i] = on[i] + oe[i];
    }
    ncl = nbig + (tu.batch_split ? 0 : batch_clusters(ow.data() + nbig, G - nbig, total_work));
    uint32_t* d_order;
    DSG_TRY_CUDA(sc.get(&d_order, G));
    DSG_TRY_CUDA(copy_any(d_order, order.data(), G * sizeof(uint32_t), s));
    std::vector<uint64_t> res(4 * (size_t)G, 0);
    for (uint32_t i = 0; i < nbig; ++i) {
        const uint32_t g = order[i];
        dsg_graph view;
        view.n = (uint32_t)(vb[g + 1] - vb[g]);
        view.m = (hoff_ends[g + 1] - hoff_ends[g]) / 2;
        view.off = const_cast<uint64_t*>(d_off) + vb[g];
        view.adj = const_cast<uint32_t*>(d_adj);
        view.owns = false;
        DSG_TRY_CUDA(cudaGetDevice(&view.device));
        view.stream = s;
        uint64_t extra[2] = {0, 0};
        dsg_status st = peel_into(&view, hp[g], hq[g], a.out_set ? a.out_set + vb[g] : nullptr, &res[4 * (size_t)g],
                                  r->stats ? extra : nullptr);
        if (st != DSG_OK) return st;
        big_sum_S += extra[0];
        big_dec += extra[1];
        big_entries += 2 * view.m;
        bool want = a.core && (!b->want_core || host_want_core(b->want_core, g, s));
        if (want) {
            st = run_kcore(&view, a.core + vb[g], nullptr, 0);
            if (st != DSG_OK) return st;
        }
    }
    // clusters and blocks run side by side: the blocks fill the SMs the clusters leave
    uint32_t h_err[2] = {0, 0};
    // what a launch may take for its slabs: a few times the graphs' own size, so that small graphs
    // among large ones do not hold memory in proportion to the large ones
    auto scratch_max = [&](uint32_t lo, uint32_t hi) {
        uint64_t bytes = 0;
        for (uint32_t i = lo; i < hi; ++i) bytes += 80 * (uint64_t)on[i] + 8 * oe[i] + 4096;
        return (size_t)bytes;
    };
    SideGuard side;
    void *slabs_cl = nullptr, *slabs_bl = nullptr;
    if (ncl > nbig) {
        BatchArgs ca = a;
        ca.order = d_order + nbig;
        ca.G = ncl - nbig;
        DSG_TRY_CUDA(sc.get(&ca.next, 1));
        DSG_TRY_CUDA(cudaMemsetAsync(ca.next, 0, sizeof(unsigned long long), s));
        if (ncl < G) {
            DSG_TRY_CUDA(side.take());
            DSG_TRY_CUDA(cudaEventRecord(side->fork, s));
            DSG_TRY_CUDA(cudaStreamWaitEvent(side->s, side->fork, 0));
        }
        const cudaError_t e = batch_cluster_launch(ca, {on.data() + nbig, oe.data() + nbig},
                                                   scratch_max(nbig, ncl), s, &slabs_cl);
        if (slabs_cl) sc.adopt(slabs_cl);
        if (e == cudaErrorMemoryAllocation && !slabs_cl) {
            cudaGetLastError();
            ncl = nbig;  // not even one cluster's scratch: a block each, which takes a quarter of it
        } else {
            DSG_TRY_CUDA(e);
        }
    }
    a.order = d_order + ncl;
    a.G = G - ncl;
    if (a.G) {
        cudaStream_t sb = side ? side->s : s;
        cudaError_t e = batch_launch(a, {on.data() + ncl, oe.data() + ncl}, scratch_max(ncl, G), sb, &slabs_bl, block);
        if (slabs_bl && e == cudaSuccess)
            e = cudaMemcpyAsync(&h_err[1], slabs_bl, sizeof(uint32_t), cudaMemcpyDeviceToHost, sb);
        if (slabs_bl) dev_free(slabs_bl, sb);
        if (side) {
            // the caller's stream waits for the blocks whatever became of the launch
            cudaEventRecord(side->join, sb);
            cudaStreamWaitEvent(s, side->join, 0);
        }
        DSG_TRY_CUDA(e);
    }
    if (slabs_cl) DSG_TRY_CUDA(cudaMemcpyAsync(&h_err[0], slabs_cl, sizeof(uint32_t), cudaMemcpyDeviceToHost, s));
    std::vector<uint64_t> res_dev(4 * (size_t)G);
    DSG_TRY_CUDA(cudaMemcpyAsync(res_dev.data(), a.res, res_dev.size() * sizeof(uint64_t), cudaMemcpyDeviceToHost, s));
    if (r->core && !core_direct) DSG_TRY_CUDA(copy_any(r->core, a.core, N * sizeof(uint32_t), s));
    if (r->out_set && !set_direct) DSG_TRY_CUDA(copy_any(r->out_set, a.out_set, N, s));
    DSG_TRY_CUDA(cudaStreamSynchronize(s));
    if (h_err[0] | h_err[1]) return status_from_err(h_err[0] | h_err[1], "batch");
    for (uint32_t i = nbig; i < G; ++i) {
        const uint32_t g = order[i];
        for (int k = 0; k < 4; ++k) res[4 * (size_t)g + k] = res_dev[4 * (size_t)g + k];
    }
    for (uint32_t g = 0; g < G; ++g) {
        if (r->E) r->E[g] = res[4 * (size_t)g + 0];
        if (r->V) r->V[g] = res[4 * (size_t)g + 1];
        if (r->rounds) r->rounds[g] = res[4 * (size_t)g + 2];
        if (r->best_round) r->best_round[g] = res[4 * (size_t)g + 3];
    }
    if (r->stats) {
        unsigned long long h[3] = {0, 0, 0};
        DSG_TRY_CUDA(cudaMemcpy(h, d_stats, sizeof(h), cudaMemcpyDeviceToHost));
        r->stats[0] = h[0] + big_sum_S;
        r->stats[1] = h[1] + big_dec;
        r->stats[2] = h[2] + big_entries;
        r->stats[3] = nbig;
    }
    return DSG_OK;
}
