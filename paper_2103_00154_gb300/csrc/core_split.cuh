// The bitwise search for core numbers, by the blocks of one team (a grid or a
// cluster).
//
// The last levels of Algorithm 2's first phase, all at once.  Once few
// vertices remain, a level of the grid-wide kernel costs mostly the latency of
// its cascade: there are hundreds of levels, each with a chain of a few
// dependent drains, and hardly any work in any of them.  Here the levels
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
// (a hub's row is many warps' work, 32 short rows one warp's); the lanes find
// an entry's piece by counting piece starts in a bit map and look it up in
// shared memory (with a shuffle search and three shuffles per entry, a quarter
// of the wide waves' load-store work, 0.85 ms on R-MAT scale 18 and 2.73 on
// scale 20 beside its peels; 0.81 and 2.63 this way).
// key is written to a buffer of its own for every bit, so its look-ups may be
// cached in L1 although the kernel rewrites it while it runs.
//
// The blocks meet after every wave (Team::meet: the pieces that the wave queued
// come back with the wait).  A grid's wait is bounded (ERR_TIMEOUT); a cluster's
// is the hardware's barrier over blocks that were launched together.
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
// 0.74 at 700,001 vertices -- the wave waits for the longest chain); waves of
// at most 32, 64 or 160 pieces by block 0 alone while the others wait at one
// meeting (1.288, 1.295, 1.365 ms against 1.274 there, 5.43, 5.39, 5.51
// against 5.07 on Chung-Lu 2^24).
#pragma once

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

template <int TB>
struct SplitSmem {
    uint32_t pushed;                  // pieces queued by this block in the running phase
    MeetSmem meet;
    uint32_t above[32];
    uint32_t cnt[TB / 32][32];  // pull: a warp's counts, per piece
    uint4 own[TB / 32][32];     // a warp's pieces that have entries: row position to add an entry to, key looked for
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

// All blocks meet; returns the pieces queued by all since the last time.
template <int TB, bool CL>
__device__ __forceinline__ uint32_t split_meet(SplitSmem<TB>& sm, Team<CL>& team) {
    __syncthreads();
    uint32_t mine = 0;
    if (threadIdx.x == 0) {
        mine = sm.pushed;
        sm.pushed = 0;
    }
    return team.meet(mine, sm.meet);
}

// The search by a team of blocks; a.ctl (zero beforehand) is in global memory
// or, for a cluster, in the shared memory of one of its blocks.
template <int TB, bool CL>
__device__ __forceinline__ void split_body(const SplitArgs& a, Team<CL> team, SplitSmem<TB>& sm) {
    SplitCtl* const ctl = a.ctl;
    const uint32_t tid = threadIdx.x, lane = tid & 31u;
    const uint32_t r = a.r, lo = a.lo;
    const uint32_t gw = (team.rank * TB + tid) >> 5, nw = team.size * (TB / 32);
    const uint32_t nth = team.size * TB;
    const uint32_t rpad = (r + 31u) & ~31u;  // whole warps in the per-vertex loops
    uint32_t natom = 0, nwaves = 0, nstamp = 0;
    // trace pairs: kind 11 keys written, 12 first wave over, 13 a later wave over, 14 its pieces (value)
    auto stamp = [&](uint32_t kind, uint32_t b, uint64_t val) {
        if (!a.trace) return;
        if (team.rank == 0 && tid == 0 && 2 * nstamp + 1 < a.trace_cap) {
            a.trace[2 * nstamp] = val;
            a.trace[2 * nstamp + 1] = (uint64_t)kind << 32 | b;
        }
        ++nstamp;
    };
    if (tid < 32) sm.above[tid] = 0;
    if (tid == 0) {
        sm.pushed = 0;
        meet_init(sm.meet);
    }
    sm.cnt[tid >> 5][lane] = 0;
    __syncthreads();
    // ---- every row's pieces, and how many vertices reach lo + 2^b: in a simple graph a
    // (lo + 2^b)-core needs more vertices than that of at least that degree, which bounds the bits
    for (uint32_t i = team.rank * TB + tid; i < rpad; i += nth) {
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
    const uint32_t npieces = split_meet(sm, team);
    if (!sm.meet.ok) return;
    uint32_t bits = 0;
    {
        const uint32_t cnt = ld_volatile_u32(&ctl->above[lane]);
        const uint32_t m = __ballot_sync(kFullMask, lane < kSplitBits && cnt > lo + (1u << lane));
        bits = m ? 32u - (uint32_t)__clz(m) : 0u;
    }
    // ---- one wave over list[from, to): push the rows' removal, or pull it
    // (first: list holds every row's pieces, only those of (push) the first or (pull) the
    // other vertices count)
    auto wave = [&](const uint4* list, uint32_t from, uint32_t to, const uint32_t* key, uint32_t bound, bool first,
                    bool pull, unsigned long long* tail) {
        const uint32_t n_ = to - from;
        // pieces per warp and turn, the same for every turn
        const uint32_t turns = (uint32_t)(((uint64_t)n_ + 32ull * nw - 1) / (32ull * nw));
        const uint32_t G = turns ? (uint32_t)(((uint64_t)n_ + (uint64_t)nw * turns - 1) / ((uint64_t)nw * turns)) : 1u;
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
            // the pieces that have entries, in order, for the entries to look up
            const uint32_t nz = __ballot_sync(kFullMask, len != 0);
            const uint32_t mypos = __popc(nz & lanemask_lt());
            uint4* const own = sm.own[tid >> 5];
            __syncwarp();
            if (len) own[mypos] = make_uint4((uint32_t)b0, (uint32_t)(b0 >> 32), kc, 0u);
            __syncwarp();
            for (uint32_t e0 = lane; e0 < ((total + 31u) & ~31u); e0 += 32 * kBatch) {
                uint32_t u[kBatch], kk[kBatch], ow[kBatch], ku[kBatch], old[kBatch];
                // an entry's piece: the one whose start is the last at or before it, by counting the
                // starts in a map of the step's positions
                const uint32_t E = e0 - lane;
                uint32_t before = __popc(__ballot_sync(kFullMask, len != 0 && st < E));
                const uint32_t rel = len != 0 && st >= E ? st - E : 0xffffffffu;
#pragma unroll
                for (uint32_t j = 0; j < kBatch; ++j) {
                    const uint32_t e = e0 + 32 * j;
                    const uint32_t m = __reduce_or_sync(kFullMask, (rel >> 5) == j ? 1u << (rel & 31u) : 0u);
                    const uint32_t o = before + __popc(m & (0xffffffffu >> (31u - lane))) - 1u;
                    before += __popc(m);
                    const uint4 p = own[o];
                    kk[j] = p.z;
                    ow[j] = o;
                    u[j] = e < total ? __ldg(a.adj + ((uint64_t)p.y << 32 | p.x) + e) : 0xffffffffu;
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
                const uint32_t take = len ? cnt[mypos] : 0u;
                if (len) cnt[mypos] = 0;
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
        if (team.rank == 0 && tid == 0) ctl->tail[(b + 2) % 3][0] = 0;  // the next bit's, last used two bits ago
        uint32_t nfirst = 0;  // pieces of the first vertices
        for (uint32_t i = team.rank * TB + tid; i < r; i += nth) {
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
        const uint32_t np = split_meet(sm, team);
        if (!sm.meet.ok) return;
        stamp(11, b, global_ns());
        if (np != 0 && np != npieces) {
            const bool pull = npieces - np < np;
            wave(a.pieces, 0, npieces, key, bound, true, pull, tail);
            ++nwaves;
            uint32_t from = 0, to = split_meet(sm, team);
            if (!sm.meet.ok) return;
            stamp(12, b, global_ns());
            stamp(14, b, to);
            while (from < to && to <= a.cap) {
                wave(a.queue, from, to, key, bound, false, false, tail);
                ++nwaves;
                from = to;
                to += split_meet(sm, team);
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
    for (uint32_t i = team.rank * TB + tid; i < r; i += nth) {
        uint32_t c = 0;
        if (bits) {
            c = (__ldca(key - a.kstride + i) & kKeyMask) >> 1;
            if (__ldcg(a.d + i) >= lo + 1u + c) c += 1u;
        }
        a.core[a.rid ? a.rid[i] : i] = lo + c;
    }
    const uint64_t nall = warp_sum((uint64_t)natom);
    if (lane == 0 && nall) atomicAdd(&ctl->atomics, (unsigned long long)nall);
    if (team.rank == 0 && tid == 0) {
        ctl->waves = nwaves;
        ctl->stamps = nstamp;
        if (bad) atomicOr(&ctl->err, ERR_CAPACITY);
    }
}

// Key buffers for a graph of `entries` row entries: the bits searched, since
// (lo + 2^b)^2 stays below the entries.
__host__ __device__ inline uint64_t split_key_buffers(uint64_t entries) {
    uint64_t nbuf = 1;
    while (nbuf < kSplitBits && (1ull << (2 * nbuf)) <= entries) ++nbuf;
    return nbuf;
}

}  // namespace dsg
