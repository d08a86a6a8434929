// The last levels of the core numbers: the remaining graph compacted, and the
// bitwise search (core_split.cuh) on it or on a whole graph.
#include <algorithm>

#include "core_split.cuh"
#include "dsg_common.cuh"
#include "dsg_kernels.cuh"

namespace dsg {

__global__ void __launch_bounds__(kSplitTB, 1) core_split_kernel(SplitArgs a) {
    __shared__ SplitSmem<kSplitTB> sm;
    Team<false> team{blockIdx.x, gridDim.x, a.ctl->bar, &a.ctl->err, a.limit_ns};
    split_body<kSplitTB, false>(a, team, sm);
}

// The same by one cluster, its control block in shared memory (copied to
// a.ctl at the end).
__global__ void __launch_bounds__(kSplitTB, 1) core_split_cluster_kernel(SplitArgs a) {
    __shared__ SplitSmem<kSplitTB> sm;
    __shared__ SplitCtl ctl;
    SplitCtl* const global = a.ctl;
    a.ctl = at_block0(&ctl);
    const uint32_t rank = cluster_rank();
    uint32_t* const words = reinterpret_cast<uint32_t*>(&ctl);
    if (rank == 0)
        for (uint32_t i = threadIdx.x; i < sizeof(SplitCtl) / 4; i += kSplitTB) words[i] = 0;
    cluster_sync();
    split_body<kSplitTB, true>(a, Team<true>{rank, kSmallBlocks, a.ctl->bar, &a.ctl->err, 0}, sm);
    cluster_sync();  // every block's counts are in; no block leaves while another reads block 0's shared memory
    if (rank == 0)
        for (uint32_t i = threadIdx.x; i < sizeof(SplitCtl) / 4; i += kSplitTB)
            reinterpret_cast<uint32_t*>(global)[i] = words[i];
}

// ---------------------------------------------------------------- compaction

// The vertices not yet taken (claim bit clear), numbered in the order warps
// reach them: rid[i] = original id, newid[v] = i, cdeg[i] = current degree,
// flen[i] = full row length.  *r = their number.
__global__ void tail_collect_kernel(uint32_t n, const uint32_t* __restrict__ claim, const uint32_t* __restrict__ deg,
                                    const uint64_t* __restrict__ off, uint32_t* __restrict__ rid,
                                    uint32_t* __restrict__ newid, uint32_t* __restrict__ cdeg,
                                    uint32_t* __restrict__ flen, uint32_t* __restrict__ r, uint32_t cap) {
    const uint32_t words = (n + 31) >> 5;
    const uint32_t lane = threadIdx.x & 31u;
    for (uint32_t w0 = (blockIdx.x * blockDim.x + threadIdx.x) & ~31u; w0 < words;
         w0 += (gridDim.x * blockDim.x) & ~31u) {
        const uint32_t w = w0 + lane;
        uint32_t free_bits = 0;
        if (w < words) {
            free_bits = ~claim[w];
            const uint32_t hi = n - w * 32;  // vertices in this word
            if (hi < 32) free_bits &= (1u << hi) - 1u;
        }
        const uint32_t c = __popc(free_bits);
        const uint32_t inc = warp_incl_scan(c);
        uint32_t base = 0;
        if (lane == 31 && inc) base = atomicAdd(r, inc);
        base = __shfl_sync(kFullMask, base, 31) + inc - c;
        while (free_bits) {
            const uint32_t b = __ffs(free_bits) - 1;
            free_bits &= free_bits - 1;
            const uint32_t v = w * 32 + b;
            if (base < cap) {
                rid[base] = v;
                newid[v] = base;
                cdeg[base] = deg[v];
                flen[base] = (uint32_t)(off[v + 1] - off[v]);
            }
            ++base;
        }
    }
}

// Compacted rows: every entry of the remaining vertices' full rows whose
// neighbour remains, renumbered, at the row's next free slot (the order in a
// row does not matter to the core numbers).  Edge-balanced over the full rows.
// Bound by its chains of dependent reads (row, neighbour, claim bit, slot): one
// after the other for each entry they took 1.46 ms for 2^24 vertices and 2^28
// pairs, with a lane's four entries in flight together 1.16.
__global__ void __launch_bounds__(256) tail_fill_kernel(uint32_t r, const uint64_t* __restrict__ roff,
                                                        const uint32_t* __restrict__ rid,
                                                        const uint64_t* __restrict__ off,
                                                        const uint32_t* __restrict__ adj,
                                                        const uint32_t* __restrict__ claim,
                                                        const uint32_t* __restrict__ newid,
                                                        const uint64_t* __restrict__ coff,
                                                        uint32_t* __restrict__ fill, uint32_t* __restrict__ cadj,
                                                        uint32_t* __restrict__ err) {
    auto pre = [&](uint64_t) { return 0u; };
    auto put = [&](const uint32_t* i, const uint64_t* j, const uint32_t*, uint32_t valid) {
        uint32_t u[kWalkU], keep = 0;
#pragma unroll
        for (uint32_t t = 0; t < kWalkU; ++t) {
            u[t] = 0;
            if (valid >> t & 1u) u[t] = ld_stream(adj + off[rid[i[t]]] + (j[t] - roff[i[t]]));
        }
#pragma unroll
        for (uint32_t t = 0; t < kWalkU; ++t)
            if ((valid >> t & 1u) && !(claim[u[t] >> 5] >> (u[t] & 31u) & 1u)) keep |= 1u << t;
        // the slots of all kWalkU entries are asked for before the first is used
        uint32_t base[kWalkU], peers[kWalkU], to[kWalkU];
        uint64_t row[kWalkU], end[kWalkU];
#pragma unroll
        for (uint32_t t = 0; t < kWalkU; ++t) {
            const bool kept = keep >> t & 1u;
            peers[t] = __match_any_sync(kFullMask, kept ? i[t] : 0xffffffffu);
            base[t] = 0;
            if (kept && (threadIdx.x & 31u) == (uint32_t)(__ffs(peers[t]) - 1))
                base[t] = atomicAdd(&fill[i[t]], (uint32_t)__popc(peers[t]));
            to[t] = kept ? newid[u[t]] : 0u;
            row[t] = kept ? coff[i[t]] : 0u;
            end[t] = kept ? coff[i[t] + 1] : 0u;
        }
#pragma unroll
        for (uint32_t t = 0; t < kWalkU; ++t) {
            base[t] = __shfl_sync(kFullMask, base[t], __ffs(peers[t]) - 1);
            if (!(keep >> t & 1u)) continue;
            // a remaining vertex keeps exactly its degree's worth of neighbours; anything
            // past its row end means the state was not a finished level: flag, do not write
            const uint64_t at = row[t] + base[t] + __popc(peers[t] & lanemask_lt());
            if (at < end[t]) cadj[at] = to[t];
            else atomicOr(err, ERR_RANGE);
        }
    };
    walk_all_entries(roff, r, pre, put);
}

// What a level-by-level run would count on these vertices: levels[0] = distinct
// core numbers, levels[1] = sum over them of the vertices at or above.  One
// block; hist (kmax + 1 bins, zero beforehand) is filled first.
__global__ void __launch_bounds__(1024) tail_levels_kernel(uint32_t r, const uint32_t* __restrict__ rid,
                                                           const uint32_t* __restrict__ core, uint32_t bins,
                                                           uint32_t* hist, unsigned long long* levels) {
    __shared__ uint64_t tmp[33];
    for (uint32_t i = threadIdx.x; i < r; i += 1024) {
        const uint32_t c = core[rid ? rid[i] : i];
        if (c < bins) atomicAdd(&hist[c], 1u);
    }
    __syncthreads();
    uint64_t above = 0, nl = 0, ns = 0;
    for (int64_t top = (int64_t)bins - 1; top >= 0; top -= 1024) {
        const int64_t k = top - (int64_t)threadIdx.x;
        const uint64_t x = k >= 0 ? __ldcg(hist + k) : 0;
        uint64_t tot;
        const uint64_t pre = block_excl_scan<uint64_t>(x, tmp, &tot);
        if (x) {
            ++nl;
            ns += above + pre + x;
        }
        above += tot;
    }
    nl = block_sum<uint64_t>(nl, tmp);
    ns = block_sum<uint64_t>(ns, tmp);
    if (threadIdx.x == 0) {
        levels[0] = nl;
        levels[1] = ns;
    }
}

// Vertices plus row entries up to which one cluster searches (us, cluster /
// grid: work of 28,000 140 / 165, 113,000 164 / 179, 168,000 323 / 353,
// 244,000 363 / 378, 337,000 449 / 442, 372,000 300 / 251).
constexpr uint64_t kSmallCore = 250000;

// The bitwise search on a graph of r vertices (rows off, adj), none with a core number below lo; core numbers to core (by original
// id through rid, nullable: the vertices' own numbers).
dsg_status core_split(uint32_t r, uint32_t lo, const uint64_t* off, const uint32_t* adj, uint64_t entries,
                      const uint32_t* rid, uint32_t* core, const dsg_graph* g, Scratch& sc, uint64_t* stats5,
                      uint64_t* trace, uint64_t trace_cap, uint64_t* stamps) {
    cudaStream_t s = g->stream;
    SplitArgs a;
    a.r = r;
    a.lo = lo;
    a.off = off;
    a.adj = adj;
    a.rid = rid;
    a.core = core;
    a.limit_ns = wait_limit_ns();
    a.trace = trace;
    a.trace_cap = trace ? trace_cap : 0;
    a.kstride = ((uint64_t)r + 63) & ~uint64_t(63);
    a.cap = (uint64_t)r + entries / kPiece;
    // one allocation for all of it
    const uint64_t nbuf = split_key_buffers(entries);
    const uint64_t words = 16 * 64 + a.kstride * (2 + nbuf);
    static_assert(sizeof(SplitCtl) <= 16 * 64 * 4, "the control block's share of the allocation");
    uint32_t* w;
    DSG_TRY_CUDA(sc.get(&w, words + 8 * a.cap));
    a.ctl = reinterpret_cast<SplitCtl*>(w);
    a.d = w + 16 * 64;
    a.ds = a.d + a.kstride;
    a.key = a.ds + a.kstride;
    a.pieces = reinterpret_cast<uint4*>(w + words);
    a.queue = a.pieces + a.cap;
    const bool small = r + entries <= kSmallCore && (g->max_blocks == 0 || g->max_blocks >= kSmallBlocks) &&
                       clusters_fit(core_split_cluster_kernel, kSmallBlocks, kSplitTB, 0) > 0;
    if (small) {
        LaunchScope ls("kcore_split", s);
        DSG_TRY_CUDA(launch_cluster(core_split_cluster_kernel, kSmallBlocks, kSplitTB, 0, s, a));
    } else {
        DSG_TRY_CUDA(cudaMemsetAsync(a.ctl, 0, sizeof(SplitCtl), s));
        uint32_t grid = 1;
        DSG_TRY_CUDA(coop_grid(core_split_kernel, kSplitTB, 0, (uint64_t)r + entries / 16, 1, &grid, g->max_blocks));
        void* params[] = {&a};
        LaunchScope ls("kcore_split", s);
        DSG_TRY_CUDA(cudaLaunchCooperativeKernel((const void*)core_split_kernel, dim3(grid), dim3(kSplitTB), params, 0,
                                                 s));
    }
    unsigned long long* lev = nullptr;
    if (stats5) {
        uint32_t* hist;
        const uint32_t bins = (uint32_t)std::min<uint64_t>((uint64_t)lo + (1ull << kSplitBits), 1ull << 31);
        DSG_TRY_CUDA(sc.get(&hist, bins));
        DSG_TRY_CUDA(sc.get(&lev, 2));
        DSG_TRY_CUDA(cudaMemsetAsync(hist, 0, (size_t)bins * 4, s));
        LaunchScope ls("kcore_tail_levels", s);
        tail_levels_kernel<<<1, 1024, 0, s>>>(r, rid, core, bins, hist, lev);
        DSG_TRY_CUDA(cudaGetLastError());
    }
    SplitCtl h;
    unsigned long long hl[2] = {0, 0};
    DSG_TRY_CUDA(cudaMemcpyAsync(&h, a.ctl, sizeof(h), cudaMemcpyDeviceToHost, s));
    if (lev) DSG_TRY_CUDA(cudaMemcpyAsync(hl, lev, sizeof(hl), cudaMemcpyDeviceToHost, s));
    DSG_TRY_CUDA(cudaStreamSynchronize(s));
    dsg_status st = status_from_err(h.err, "kcore tail");
    if (st != DSG_OK) return st;
    if (stats5) {
        stats5[0] += hl[0];
        stats5[2] += hl[1];
        stats5[4] += h.atomics;
    }
    if (stamps) *stamps = h.stamps;
    return DSG_OK;
}

// Scan of n uint32 values into out[0..n] (exclusive, out[n] = total).
dsg_status scan_u32(const uint32_t* in, uint64_t n, uint64_t* out, Scratch& sc, cudaStream_t s);

dsg_status kcore_tail(const dsg_graph* g, uint32_t* deg, const uint32_t* claim, uint32_t cap, uint32_t lo,
                      uint64_t* stats5, uint64_t* trace, uint64_t trace_cap, uint64_t* stamps) {
    cudaStream_t s = g->stream;
    const uint32_t n = g->n;
    const uint64_t* off = g->off;
    const uint32_t* adj = g->adj;
    Scratch sc(s);
    uint32_t *rid, *newid, *cdeg, *flen, *cnt;
    DSG_TRY_CUDA(sc.get(&rid, cap));
    DSG_TRY_CUDA(sc.get(&newid, n));
    DSG_TRY_CUDA(sc.get(&cdeg, cap + 1));
    DSG_TRY_CUDA(sc.get(&flen, cap + 1));
    DSG_TRY_CUDA(sc.get(&cnt, 1));
    DSG_TRY_CUDA(cudaMemsetAsync(cnt, 0, sizeof(uint32_t), s));
    {
        const uint32_t words = (n + 31) >> 5;
        const uint32_t gb = (uint32_t)std::min<uint64_t>(((uint64_t)words + 255) / 256, (uint64_t)dev_info().sms * 8);
        LaunchScope ls("kcore_tail_collect", s);
        tail_collect_kernel<<<gb ? gb : 1, 256, 0, s>>>(n, claim, deg, off, rid, newid, cdeg, flen, cnt, cap);
    }
    DSG_TRY_CUDA(cudaGetLastError());
    uint32_t r = 0;
    DSG_TRY_CUDA(cudaMemcpyAsync(&r, cnt, sizeof(uint32_t), cudaMemcpyDeviceToHost, s));
    DSG_TRY_CUDA(cudaStreamSynchronize(s));
    if (r == 0) return DSG_OK;
    if (r > cap) {
        set_error("kcore tail: %u vertices remain, more than the %u it was sized for", r, cap);
        return DSG_ECUDA;
    }
    uint64_t *coff, *roff;
    DSG_TRY_CUDA(sc.get(&coff, (size_t)r + 1));
    DSG_TRY_CUDA(sc.get(&roff, (size_t)r + 1));
    dsg_status st = scan_u32(cdeg, r, coff, sc, s);
    if (st != DSG_OK) return st;
    st = scan_u32(flen, r, roff, sc, s);
    if (st != DSG_OK) return st;
    uint64_t ecount = 0;
    DSG_TRY_CUDA(cudaMemcpyAsync(&ecount, coff + r, sizeof(uint64_t), cudaMemcpyDeviceToHost, s));
    DSG_TRY_CUDA(cudaStreamSynchronize(s));
    uint32_t *cadj, *fill;
    DSG_TRY_CUDA(cudaMemsetAsync(cnt, 0, sizeof(uint32_t), s));  // now the fill's error word
    DSG_TRY_CUDA(sc.get(&cadj, ecount ? ecount : 1));
    DSG_TRY_CUDA(sc.get(&fill, r));
    DSG_TRY_CUDA(cudaMemsetAsync(fill, 0, (size_t)r * 4, s));
    {
        int per_sm = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, tail_fill_kernel, 256, 0) != cudaSuccess ||
            per_sm < 1)
            per_sm = 1;
        LaunchScope ls("kcore_tail_fill", s);
        tail_fill_kernel<<<(uint32_t)dev_info().sms * (uint32_t)per_sm, 256, 0, s>>>(r, roff, rid, off, adj, claim,
                                                                                    newid, coff, fill, cadj, cnt);
    }
    DSG_TRY_CUDA(cudaGetLastError());
    dsg_status st3 = core_split(r, lo, coff, cadj, ecount, rid, deg, g, sc, stats5, trace, trace_cap, stamps);
    if (st3 != DSG_OK) return st3;
    uint32_t fill_err = 0;
    DSG_TRY_CUDA(cudaMemcpyAsync(&fill_err, cnt, sizeof(uint32_t), cudaMemcpyDeviceToHost, s));
    DSG_TRY_CUDA(cudaStreamSynchronize(s));
    if (fill_err) {
        set_error("kcore tail: inconsistent remaining graph (err %u)", fill_err);
        return DSG_ECUDA;
    }
    return DSG_OK;
}

}  // namespace dsg
