// The last levels of Algorithm 2's first phase (core numbers), all at once: a
// bitwise search for every remaining vertex's core number.
//
// Once few vertices remain, a level of the grid-wide kernel costs mostly the
// latency of its cascade: there are hundreds of levels, each with a chain of
// a few dependent drains, and hardly any work in any of them.  Here the levels
// are not walked.  A remaining vertex's core number is lo + c, and c is found
// from its top bit down: for bit b, every group of vertices that agree on the
// bits above b is peeled at once to its (lo + c + 2^b)-core -- the vertices
// that stay have the bit set, those that leave do not -- so a remaining graph
// whose core numbers span K values takes log2 K peels instead of up to K
// levels, and a peel is a few waves, each of them spread over the whole grid
// (Chung-Lu, 700,001 vertices, 65,536 remaining: 9 peels and 103 waves
// instead of 97 levels of about 4.5 dependent drains each).
//
// A vertex's degree d counts its neighbours in its own group (not yet removed
// in this peel) and in every group above it; those have core numbers at least
// as large as the group's bound whatever this peel does.  So a removed vertex
// takes one from each neighbour of its own group only, and the one decrement
// that takes a neighbour from its bound to below it puts it in the next wave:
// no claim, no undo.  After the peel a vertex that stayed keeps its d (the
// groups above it are now its own survivors and those above), one that left
// gets back the d it had before the peel (ds): everyone it counted is still
// in its group or above.
//
// Bit b, for every vertex: key = c << 1 | first, first = d already below the
// bound.  The peel's first wave removes the `first` vertices either by
// pushing (their rows take one from each key == c << 1 neighbour) or by
// pulling (every other vertex counts its key == c << 1 | 1 neighbours),
// whichever reads fewer row pieces; the later waves push.  Rows are walked
// as pieces of at most kPiece entries, as many pieces per warp as spread the
// wave over all warps, the entries of a warp's pieces dealt out to its lanes
// (a hub's row is many warps' work, 32 short rows one warp's).
// key is written to a buffer of its own for every bit, so its look-ups may be
// cached in L1 although the kernel rewrites it while it runs.
//
// The blocks meet after every wave (grid_meet: the pieces that the wave queued
// come back with the wait).
// Every wait is bounded (ERR_TIMEOUT).
//
// What bounds it: the wide waves, L2 gathers (a bit's first wave on Chung-Lu
// 2^24, 65,287 vertices and about 45 M row entries read: 60 us); the thin ones,
// a chain of about eight dependent L2 round trips (the meeting, piece, row
// entry, key, decrement, queue slot, piece written and released): 4.5 us.
// Measured against one 16-block cluster walking the levels with the degrees
// in its shared memory, 65,536 vertices left to either: Chung-Lu 2^24 (870
// levels) 18.7 -> 3.6 ms, 700,001 vertices (97 levels) 2.04 -> 0.68 ms, R-MAT
// scale 18 (129 levels) 2.15 -> 0.76 ms.  Where it takes over:
// kTailHandOver and kTailWhole.
// Tried and dropped: a warp that goes on with the vertices it has removed
// instead of queueing them (1, 2 or 4 rows deep: 0.82, 0.84, 0.88 ms against
// 0.74 at 700,001 vertices -- the wave waits for the longest chain).
#include <algorithm>

#include "dsg_common.cuh"
#include "dsg_kernels.cuh"

namespace dsg {

constexpr uint32_t kSplitTB = 1024;
constexpr uint32_t kPiece = 128;  // entries per row piece: one step of a warp, 4 loads per lane in flight
constexpr uint32_t kSplitBits = 18;  // bits of c (a core number k takes k (k + 1) row entries: enough below 2^36)
// A vertex's key: pieces of its row above kKeyBits (kPiecesMax: that many or
// more, count them from the row), its c, and the `first` bit.
constexpr uint32_t kKeyBits = kSplitBits + 1;
constexpr uint32_t kKeyMask = (1u << kKeyBits) - 1u;
constexpr uint32_t kPiecesMax = (1u << (32 - kKeyBits)) - 1u;

__device__ __forceinline__ uint32_t pieces_of(uint64_t len) { return (uint32_t)((len + kPiece - 1) / kPiece); }

struct __align__(128) SplitCtl {
    unsigned long long bar[2][16];  // arrivals (low half) and pieces queued (high half), by parity
    unsigned long long tail[3][16];  // next queue slot, by bit modulo 3
    uint32_t above[32];  // vertices with degree >= lo + 2^b at the start
    unsigned long long npieces;
    unsigned long long atomics, waves, stamps;
    uint32_t err;
};

struct SplitArgs {
    uint32_t r;           // vertices, numbered 0..r-1
    uint32_t lo;          // no core number is below lo
    const uint64_t* off;  // rows, r + 1
    const uint32_t* adj;
    const uint32_t* rid;  // original ids (nullable: the numbers themselves)
    uint32_t* d;          // degrees in the running peel
    uint32_t* ds;         // degrees before it
    uint32_t* key;        // a buffer of kstride entries for every bit
    uint64_t kstride;
    uint4* pieces;        // every row's pieces: first entry (low word), vertex, entries | first entry >> 32 << 16
    uint4* queue;         // the waves' pieces, the vertex's c in the last word
    uint64_t cap;         // slots of each
    uint32_t* core;       // core numbers by original id
    SplitCtl* ctl;
    uint64_t limit_ns;
    uint64_t* trace;      // nullable: block 0 stamps (%globaltimer, kind << 32 | bit) per phase
    uint64_t trace_cap;
};

struct SplitSmem {
    uint32_t pushed;                  // pieces queued by this block in the running phase
    MeetSmem meet;
    uint32_t above[32];
    uint32_t cnt[kSplitTB / 32][32];  // pull: a warp's counts, per piece
};

// Write the pieces of the rows u[j] (bit j of hit; np[j] pieces each, c[j] to
// go with them) to list, at slots reserved at *tail: one atomic per warp, its
// round trip running beside the loads of the row bounds.  All lanes call it.
template <int K>
__device__ __forceinline__ void put_rows(const SplitArgs& a, uint4* list, unsigned long long* tail, uint32_t* pushed,
                                         uint32_t hit, const uint32_t (&u)[K], const uint32_t (&c)[K],
                                         uint32_t (&np)[K]) {
    const uint32_t lane = lane_id();
    uint32_t mine = 0;
#pragma unroll
    for (int j = 0; j < K; ++j)
        if ((hit >> j & 1u) && np[j] == kPiecesMax) np[j] = pieces_of(a.off[u[j] + 1] - a.off[u[j]]);
#pragma unroll
    for (int j = 0; j < K; ++j) mine += hit >> j & 1u ? np[j] : 0u;
    const uint32_t inc = warp_incl_scan(mine);
    const uint32_t total = __shfl_sync(kFullMask, inc, 31);
    unsigned long long base = 0;
    if (lane == 0 && total) {
        base = atomicAdd(tail, (unsigned long long)total);
        atomicAdd(pushed, total);
    }
    uint64_t beg[K], end[K];
#pragma unroll
    for (int j = 0; j < K; ++j) {
        beg[j] = hit >> j & 1u ? a.off[u[j]] : 0;
        end[j] = hit >> j & 1u ? a.off[u[j] + 1] : 0;
    }
    base = __shfl_sync(kFullMask, base, 0) + inc - mine;
    auto put = [&](unsigned long long at, uint64_t b, uint64_t e, uint32_t v, uint32_t vc, uint32_t k) {
        b += (uint64_t)k * kPiece;
        if (at + k < a.cap && b < e)
            list[at + k] = make_uint4((uint32_t)b, v, (uint32_t)min((uint64_t)kPiece, e - b) | (uint32_t)(b >> 32) << 16,
                                      vc);
    };
#pragma unroll
    for (int j = 0; j < K; ++j) {
        const uint32_t n_ = hit >> j & 1u ? np[j] : 0u;
        if (n_ <= 4)
            for (uint32_t k = 0; k < n_; ++k) put(base, beg[j], end[j], u[j], c[j], k);
        // a long row's pieces are written by the whole warp
        for (uint32_t pend = __ballot_sync(kFullMask, n_ > 4); pend; pend &= pend - 1) {
            const uint32_t o = __ffs(pend) - 1;
            const unsigned long long ob = __shfl_sync(kFullMask, base, o);
            const uint64_t bb = __shfl_sync(kFullMask, beg[j], o), be = __shfl_sync(kFullMask, end[j], o);
            const uint32_t ov = __shfl_sync(kFullMask, u[j], o), oc = __shfl_sync(kFullMask, c[j], o);
            const uint32_t on = __shfl_sync(kFullMask, n_, o);
            for (uint32_t k = lane; k < on; k += 32) put(ob, bb, be, ov, oc, k);
        }
        base += n_;
    }
}

// All blocks meet; returns the pieces queued by the grid since the last time.
__device__ __forceinline__ uint32_t split_meet(const SplitArgs& a, SplitSmem& sm, MeetState& st) {
    __syncthreads();
    uint32_t mine = 0;
    if (threadIdx.x == 0) {
        mine = sm.pushed;
        sm.pushed = 0;
    }
    return grid_meet(a.ctl->bar, &a.ctl->err, a.limit_ns, gridDim.x, mine, st, sm.meet);
}

__global__ void __launch_bounds__(kSplitTB, 1) core_split_kernel(SplitArgs a) {
    __shared__ SplitSmem sm;
    SplitCtl* const ctl = a.ctl;
    const uint32_t tid = threadIdx.x, lane = tid & 31u;
    const uint32_t r = a.r, lo = a.lo;
    const uint32_t gw = (blockIdx.x * kSplitTB + tid) >> 5, nw = gridDim.x * (kSplitTB / 32);
    const uint32_t nth = gridDim.x * kSplitTB;
    const uint32_t rpad = (r + 31u) & ~31u;  // whole warps in the per-vertex loops
    MeetState ms;
    uint64_t natom = 0, nwaves = 0, nstamp = 0;
    // trace pairs: kind 11 keys written, 12 first wave over, 13 a later wave over, 14 its pieces (value)
    auto stamp = [&](uint32_t kind, uint32_t b, uint64_t val) {
        if (!a.trace) return;
        if (blockIdx.x == 0 && tid == 0 && 2 * nstamp + 1 < a.trace_cap) {
            a.trace[2 * nstamp] = val;
            a.trace[2 * nstamp + 1] = (uint64_t)kind << 32 | b;
        }
        ++nstamp;
    };
    if (tid < 32) sm.above[tid] = 0;
    if (tid == 0) {
        sm.pushed = 0;
        sm.meet.ok = 1;
    }
    for (uint32_t i = tid; i < kSplitTB; i += kSplitTB) sm.cnt[i >> 5][i & 31u] = 0;
    __syncthreads();
    // ---- every row's pieces, and how many vertices reach lo + 2^b: in a simple graph a
    // (lo + 2^b)-core needs more vertices than that of at least that degree, which bounds the bits
    for (uint32_t i = blockIdx.x * kSplitTB + tid; i < rpad; i += nth) {
        uint32_t d = 0, top = 0;
        const uint32_t v1[1] = {i}, c1[1] = {0u};
        if (i < r) {
            d = (uint32_t)(a.off[i + 1] - a.off[i]);
            a.d[i] = d;
            a.ds[i] = d;
            top = d > lo ? 32u - (uint32_t)__clz(d - lo) : 0u;  // d >= lo + 2^b for b < top
        }
#pragma unroll 1
        for (uint32_t b = 0; b < kSplitBits; ++b) {
            const uint32_t m = __ballot_sync(kFullMask, top > b);
            if (m == 0) break;
            if (lane == 0) atomicAdd(&sm.above[b], (uint32_t)__popc(m));
        }
        uint32_t np1[1] = {pieces_of(d)};
        put_rows<1>(a, a.pieces, &ctl->npieces, &sm.pushed, d ? 1u : 0u, v1, c1, np1);
    }
    __syncthreads();
    if (tid < 32 && sm.above[tid]) atomicAdd(&ctl->above[tid], sm.above[tid]);
    const uint32_t npieces = split_meet(a, sm, ms);
    if (!sm.meet.ok) return;
    uint32_t bits = 0;
    {
        const uint32_t cnt = ld_relaxed_u32(&ctl->above[lane]);
        const uint32_t m = __ballot_sync(kFullMask, lane < kSplitBits && cnt > lo + (1u << lane));
        bits = m ? 32u - (uint32_t)__clz(m) : 0u;
    }
    // ---- one wave over list[from, to): push the rows' removal, or pull it
    // (first: list holds every row's pieces, only those of (push) the first or (pull) the
    // other vertices count)
    auto wave = [&](const uint4* list, uint32_t from, uint32_t to, const uint32_t* key, uint32_t bound, bool first,
                    bool pull, unsigned long long* tail) {
        const uint32_t n_ = to - from;
        uint32_t G = (n_ + nw - 1) / nw;
        if (G > 32) G = 32;
        uint32_t* const cnt = sm.cnt[tid >> 5];
        // lane l takes piece g0 + l nw + gw: neighbouring pieces (a hub's) go to different warps
        for (uint64_t g0 = 0; g0 < n_; g0 += (uint64_t)nw * G) {
            uint32_t len = 0, kv = 0, kc = 0, v = 0;
            uint64_t b0 = 0;
            const uint64_t at = g0 + (uint64_t)lane * nw + gw;
            if (lane < G && at < n_) {
                const uint4 it = __ldcg(list + from + at);
                v = it.y;
                len = it.z & 0xffffu;
                b0 = (uint64_t)(it.z >> 16) << 32 | it.x;
                if (first) {
                    kv = __ldca(key + v);
                    // push: neighbours of v's group that are not removed yet; pull: those removed first
                    kc = pull ? (kv | 1u) & kKeyMask : kv & (kKeyMask - 1u);
                    if ((kv & 1u) == (pull ? 1u : 0u)) len = 0;
                } else {
                    kc = it.w << 1;
                }
            }
            const uint32_t inc = warp_incl_scan(len);
            const uint32_t total = __shfl_sync(kFullMask, inc, 31);
            const uint32_t st = inc - len;
            b0 -= st;  // entry e of the warp's pieces is adj[b0 + e] for its owner's b0
            for (uint32_t e0 = lane; e0 < ((total + 31u) & ~31u); e0 += 32 * kBatch) {
                uint32_t u[kBatch], kk[kBatch], ow[kBatch], ku[kBatch], old[kBatch];
#pragma unroll
                for (uint32_t j = 0; j < kBatch; ++j) {
                    const uint32_t e = e0 + 32 * j;
                    uint32_t o = 0;
                    if (G > 1) {
#pragma unroll
                        for (uint32_t step = 16; step > 0; step >>= 1) {
                            const uint32_t s = __shfl_sync(kFullMask, st, o + step);
                            if (o + step < 32 && s <= e) o += step;
                        }
                    }
                    const uint64_t ob = __shfl_sync(kFullMask, b0, o);
                    kk[j] = __shfl_sync(kFullMask, kc, o);
                    ow[j] = o;
                    u[j] = e < total ? __ldg(a.adj + ob + e) : 0xffffffffu;
                }
#pragma unroll
                for (uint32_t j = 0; j < kBatch; ++j) ku[j] = u[j] < r ? __ldca(key + u[j]) : ~kk[j];
                if (pull) {
#pragma unroll
                    for (uint32_t j = 0; j < kBatch; ++j)
                        if ((ku[j] & kKeyMask) == kk[j]) atomicAdd(&cnt[ow[j]], 1u);
                } else {
                    uint32_t hit = 0;
#pragma unroll
                    for (uint32_t j = 0; j < kBatch; ++j) {
                        old[j] = 0;
                        if ((ku[j] & kKeyMask) == kk[j]) {
                            old[j] = atomicSub(&a.d[u[j]], 1u);
                            ++natom;
                        }
                    }
#pragma unroll
                    for (uint32_t j = 0; j < kBatch; ++j) {
                        if ((ku[j] & kKeyMask) == kk[j] && old[j] == bound + (kk[j] >> 1)) hit |= 1u << j;
                        ku[j] >>= kKeyBits;  // its pieces
                        kk[j] >>= 1;         // its c
                    }
                    if (__any_sync(kFullMask, hit != 0))
                        put_rows<kBatch>(a, a.queue, tail, &sm.pushed, hit, u, kk, ku);
                }
            }
            if (pull) {
                __syncwarp();
                const uint32_t take = cnt[lane];
                cnt[lane] = 0;
                const uint32_t v1[1] = {v}, c1[1] = {kc >> 1};
                uint32_t np1[1] = {kv >> kKeyBits};
                uint32_t hit = 0;
                if (take) {
                    const uint32_t old = atomicSub(&a.d[v], take);
                    ++natom;
                    const uint32_t mid = bound + c1[0];
                    hit = old >= mid && old - take < mid ? 1u : 0u;
                }
                if (__any_sync(kFullMask, hit != 0)) put_rows<1>(a, a.queue, tail, &sm.pushed, hit, v1, c1, np1);
                __syncwarp();
            }
        }
    };
    uint32_t* key = a.key;  // buffer of the running bit
    bool bad = false;
    for (uint32_t b = bits; b-- > 0;) {
        // ---- what the bit above decided, and this bit's keys
        const uint32_t bound = lo + (1u << b);
        const bool top = b + 1 == bits;
        unsigned long long* const tail = &ctl->tail[b % 3][0];
        if (blockIdx.x == 0 && tid == 0) ctl->tail[(b + 2) % 3][0] = 0;  // the next bit's, last used two bits ago
        uint32_t nfirst = 0;  // pieces of the first vertices
        for (uint32_t i = blockIdx.x * kSplitTB + tid; i < r; i += nth) {
            uint32_t c = 0, d = __ldcg(a.d + i);
            if (!top) {
                c = (__ldca(key - a.kstride + i) & kKeyMask) >> 1;
                if (d >= bound + (1u << b) + c) {
                    c += 2u << b;
                    a.ds[i] = d;
                } else {
                    d = a.ds[i];
                    a.d[i] = d;
                }
            }
            const bool first = d < bound + c;
            const uint32_t np = pieces_of(a.off[i + 1] - a.off[i]);
            key[i] = min(np, kPiecesMax) << kKeyBits | c << 1 | (first ? 1u : 0u);
            if (first) nfirst += np;
        }
        nfirst = warp_sum(nfirst);
        if (lane == 0 && nfirst) atomicAdd(&sm.pushed, nfirst);
        const uint32_t np = split_meet(a, sm, ms);
        if (!sm.meet.ok) return;
        stamp(11, b, global_ns());
        if (np != 0 && np != npieces) {
            const bool pull = npieces - np < np;
            wave(a.pieces, 0, npieces, key, bound, true, pull, tail);
            ++nwaves;
            uint32_t from = 0, to = split_meet(a, sm, ms);
            if (!sm.meet.ok) return;
            stamp(12, b, global_ns());
            stamp(14, b, to);
            while (from < to && to <= a.cap) {
                wave(a.queue, from, to, key, bound, false, false, tail);
                ++nwaves;
                from = to;
                to += split_meet(a, sm, ms);
                if (!sm.meet.ok) return;
                stamp(13, b, global_ns());
                stamp(14, b, to - from);
            }
            if (to > a.cap) {  // cannot happen: a row is queued once per bit
                bad = true;
                break;
            }
        }
        key += a.kstride;
    }
    // ---- the last bit's decision; core numbers out
    for (uint32_t i = blockIdx.x * kSplitTB + tid; i < r; i += nth) {
        uint32_t c = 0;
        if (bits) {
            c = (__ldca(key - a.kstride + i) & kKeyMask) >> 1;
            if (__ldcg(a.d + i) >= lo + 1u + c) c += 1u;
        }
        a.core[a.rid ? a.rid[i] : i] = lo + c;
    }
    natom = warp_sum(natom);
    if (lane == 0 && natom) atomicAdd(&ctl->atomics, (unsigned long long)natom);
    if (blockIdx.x == 0 && tid == 0) {
        ctl->waves = nwaves;
        ctl->stamps = nstamp;
        if (bad) atomicOr(&ctl->err, ERR_CAPACITY);
    }
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
#pragma unroll
        for (uint32_t t = 0; t < kWalkU; ++t) {
            const uint32_t key = (keep >> t & 1u) ? i[t] : 0xffffffffu;
            const uint32_t peers = __match_any_sync(kFullMask, key);
            const uint32_t leader = __ffs(peers) - 1;
            uint32_t base = 0;
            if (key != 0xffffffffu && (threadIdx.x & 31u) == leader) base = atomicAdd(&fill[key], __popc(peers));
            base = __shfl_sync(kFullMask, base, leader);
            if (key != 0xffffffffu) {
                // a remaining vertex keeps exactly its degree's worth of neighbours; anything
                // past its row end means the state was not a finished level: flag, do not write
                const uint64_t at = coff[key] + base + __popc(peers & lanemask_lt());
                if (at < coff[key + 1]) cadj[at] = newid[u[t]];
                else atomicOr(err, ERR_RANGE);
            }
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
    DSG_TRY_CUDA(sc.get(&a.d, r));
    DSG_TRY_CUDA(sc.get(&a.ds, r));
    // the bits searched: (lo + 2^b)^2 stays below the row entries
    uint64_t nbuf = 1;
    while (nbuf < kSplitBits && (1ull << (2 * nbuf)) <= entries) ++nbuf;
    DSG_TRY_CUDA(sc.get(&a.key, a.kstride * nbuf));
    DSG_TRY_CUDA(sc.get(&a.pieces, a.cap));
    DSG_TRY_CUDA(sc.get(&a.queue, a.cap));
    DSG_TRY_CUDA(sc.get(&a.ctl, 1));
    DSG_TRY_CUDA(cudaMemsetAsync(a.ctl, 0, sizeof(SplitCtl), s));
    uint32_t grid = 1;
    DSG_TRY_CUDA(coop_grid(core_split_kernel, kSplitTB, 0, (uint64_t)r + entries / 16, 1, &grid, g->max_blocks));
    {
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
