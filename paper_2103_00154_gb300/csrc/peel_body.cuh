// Algorithm 1 (P-Bahmani): the round-synchronous (2+2eps) densest-subgraph
// peel as one persistent cooperative kernel.
//
// Per round r, with S_r and E_r = |E(S_r)| known to every block:
//   phase 1 (Algorithm 1's first part, over the active vertices): every alive vertex is
//     tested against T_r = floor(2(p+q)E_r / (q|S_r|)), i.e. deg <= 2(1+eps)rho
//     exactly; failures are marked (state word and status map) and their rows
//     queued as pieces of at most chunk_len entries, survivors are compacted
//     into the next alive list (warp ballots, one scan of the warps' totals
//     and one atomic per list and block tile); the degrees of the failures are
//     summed (X);
//   the blocks meet (Algorithm 1's synchronisation between its two parts),
//     on a word that also sums the pieces queued;
//   phase 2 (Alg. 1 part 2; not where every vertex left has failed and there
//     are at most kLastMax of them): every adjacency entry u of every failed v
//     is read once, the pieces dealt to the warps in groups as large as spread them
//     over all warps and a group's entries to the warp's lanes; u's bits in
//     the status map say whether it is still alive (and whether it is a hub);
//     an alive u loses one degree (atomicSub, combined per block for hubs) and
//     the decrement is counted (D);
//   the blocks meet again; every block derives S_{r+1} and E_{r+1} from the
//     monotone counters and keeps the densest set (strict ">": a later round
//     replaces the best only when strictly denser, as in Algorithm 1); block 0
//     records the history.
// Once the alive rows hold at most kSoloEntries entries and the alive list
// kSoloList vertices, block 0 of a grid runs the remaining rounds alone and the
// others leave: a round then costs block barriers and shared-memory cursors
// only.  (Lazy rounds leave the list as it is, so a lazy tail stays with the
// grid until a round tests everyone again.)
// The edges removed in round r (Algorithm 1's reduction) are (X + D) / 2: the
// failures' degrees count every edge between two failures twice and every
// edge from a failure to a survivor once, and D counts the latter once more.
// So phase 2 never needs to tell a neighbour that failed in this round from
// one that failed earlier, and reads only the status map (2 bits per vertex,
// L2-resident) rather than the state words.
//
// Vertex state is one 32-bit word: an alive vertex holds its degree inside
// S_r (< 2^31); a failed one holds 0x80000000 | (round it failed, 1-based).
// Status map: word u / 16, bit 2 (u % 16) = u has failed, bit 2 (u % 16) + 1
// = u is a hub (first-round degree at or above the hub threshold).
#pragma once

#include <type_traits>

#include "dsg_common.cuh"
#include "dsg_kernels.cuh"

namespace dsg {

constexpr uint32_t kDead = 0x80000000u;

struct __align__(128) PeelCtl {
    unsigned long long bar[2][16];  // the blocks' meetings (Team::meet)
    uint32_t err;
    uint32_t hubs[8];               // rows of 2^(kHubBit0 + b) entries and more, below 2^(kHubBit0 + b + 1) but for the last
    uint32_t pad1[23];
    unsigned long long items;   // cursor of the piece list (all rounds)
    unsigned long long pad3[15];
    unsigned long long surv;    // cursor of survivor writes (all rounds)
    unsigned long long pad5[15];
    unsigned long long cand;    // cursor of candidate-list writes (all rounds)
    unsigned long long pad8[15];
    // sums over the rounds, one addition per block and round each: failures, their degrees (X), the
    // entries of their rows, alive-neighbour decrements (D)
    unsigned long long failed, xsum, rows, dec;
    unsigned long long pad9[12];
    unsigned long long tested, lazy_rounds;  // statistics kept by block 0: vertex tests, lazy rounds
    unsigned long long rounds, best_round, best_E, best_V;
    unsigned long long stamps;
    unsigned long long cur_S, cur_E;  // |S_r| and |E(S_r)| where the launch stopped
    unsigned long long scanned;       // row entries read by the neighbour scans
};

struct PeelArgs {
    uint32_t n;
    uint64_t m;
    uint64_t p, q;
    const uint64_t* off;
    const uint32_t* adj;
    uint32_t* st;
    uint32_t* listA;
    uint32_t* listB;
    uint64_t* items;      // pieces of the failed rows: first entry << kLenBits | entries
    uint32_t* map;        // status map, (n + 15) / 16 words
    uint32_t* candA;      // nullable (then no lazy rounds): two candidate lists of n entries
    uint32_t* candB;
    uint64_t* hist_S;     // nullable: no history (hist_cap without bound)
    uint64_t* hist_E;
    uint64_t hist_cap;
    PeelCtl* ctl;
    uint64_t limit_ns;
    uint32_t chunk_len;
    uint32_t hot_deg;
    uint64_t* trace;      // nullable: block 0 stamps %globaltimer after every meeting
    uint64_t trace_cap;
    // resuming a paused peel (r0 > 0): the state words in st are the pause's,
    // S0/E0/best the pause's values, and the first round scans every vertex,
    // skipping those already failed; max_rounds > 0 pauses after that many rounds
    uint64_t r0, S0, E0, best_round0, best_E0, best_V0;
    uint64_t max_rounds;
    uint32_t arrivals0;   // that each word of ctl->bar already counts (0 but for the test of their wrap)
};

constexpr uint32_t kLenBits = 24;         // of a piece: entries (chunk_len is kept below 2^24)
constexpr uint32_t kSoloEntries = 16384;  // block 0 alone: row entries left (each is read once more at most) ...
constexpr uint32_t kSoloList = 4096;      // ... and entries of the alive list
// Vertices left below which a round first looks whether any survived it (a
// round trip) before it scans: the last round's rows, mostly hubs', are not
// read (Chung-Lu 2^24: 789 vertices, 104 us; 3 10^6 vertices: 215, 17 us).
constexpr uint32_t kLastMax = 1u << 16;
// Hubs (their decrements are combined per block before they go to L2): on
// large graphs as many of the largest rows as the table of kAggSlots entries
// can help, counted by powers of two before the first round.  More of them
// overflow the table (a few failed probes, then the atomic all the same),
// fewer leave contended words to L2 (ms at hubs from degree 608 / 1,024 /
// 4,096 / 16,384 / 65,536: Chung-Lu 2^24, 1,810 vertices of degree >= 16,384,
// 4.02 / 3.87 / 3.47 / 3.31 / 4.96; 3 10^6 vertices, 1,350 of degree >= 4,096,
// 0.756 / 0.733 / 0.770 / 1.13 / 1.72).  The count is a pass over the row
// offsets; smaller graphs take hot_threshold's rule, as good there.
constexpr uint32_t kHubCountMin = 1u << 20;  // vertices
constexpr uint32_t kHubsMax = 2 * kAggSlots;
constexpr uint32_t kHubBit0 = 10, kHubBits = 8;  // 1,024 .. 131,072

template <int TB>
struct PeelSmem {
    AggTable agg;
    uint32_t agg_used;
    uint32_t threshold, last;
    uint32_t wit[TB / 32];         // a tile's pieces per warp, then their exclusive prefix
    uint32_t surv_at[4][TB / 32];  // a tile's survivors per (slice, warp), then their exclusive prefix in id order
    unsigned long long base[2];    // the tile's first piece and first survivor
    unsigned long long cursor[2];  // block 0 alone: the two lists' cursors
    unsigned long long add[4];     // this block's part of failed, xsum, rows, dec in the running phase
    uint64_t own[TB / 32][32];     // phase 2, a warp's pieces: row position to add an entry to
    unsigned long long cum[5];     // failed, xsum, rows, dec and the candidate cursor after the round
    unsigned long long scanned;    // rows after the last round that was scanned
    MeetSmem meet;
};

// Bits 0..15 of x spread to the even positions 0, 2, ..., 30.
__device__ __forceinline__ uint32_t spread16(uint32_t x) {
    x &= 0xffffu;
    x = (x | (x << 8)) & 0x00ff00ffu;
    x = (x | (x << 4)) & 0x0f0f0f0fu;
    x = (x | (x << 2)) & 0x33333333u;
    x = (x | (x << 1)) & 0x55555555u;
    return x;
}

// What every block knows once the peel is over (or paused).
struct PeelOut {
    uint64_t rounds, best_round, best_E, best_V;
};

// The peel by a team of blocks; a.ctl is in global memory or, for a cluster,
// in the shared memory of one of its blocks.  A block that leaves early (a
// wait ran out, or block 0 goes on alone) returns without a result.
template <int TB, bool CL>
__device__ __forceinline__ PeelOut peel_body(const PeelArgs& a, Team<CL> team, PeelSmem<TB>& sm) {
    constexpr uint32_t kW = TB / 32;
    PeelCtl* ctl = a.ctl;
    const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
    const bool resume = a.r0 > 0;
    uint64_t S = resume ? a.S0 : a.n, E = resume ? a.E0 : a.m;
    uint64_t r = a.r0;
    uint64_t item_lo = 0, surv_base = 0;
    const uint32_t* alive = nullptr;  // first round: identity (a fresh peel) or every vertex (a resumed one)
    uint32_t* next = a.listA;
    uint64_t alive_len = 0;           // entries of `alive` (after lazy rounds some of them have failed)
    // lazy rounds (thin tail): the candidate list holds every alive vertex whose degree is at or below
    // the bound B; a round whose threshold is within B tests only that list
    const bool lazy_ok = a.candA != nullptr;
    uint32_t* cur_cand = a.candA;
    uint32_t* next_cand = a.candB;
    uint64_t cand_n = 0, cand_base = 0, S_prev = S;
    bool have_cands = false;
    uint64_t cand_from = 0, cand_rest = 2;  // no candidates are collected before round cand_from
    uint32_t B = 0;
    uint64_t best_E = resume ? a.best_E0 : E, best_V = resume ? a.best_V0 : S;
    uint64_t best_round = resume ? a.best_round0 : 0;
    uint64_t nstamp = 0, tested = 0, lazy_rounds = 0;
    auto stamp = [&]() {
        if (a.trace && team.rank == 0 && tid == 0 && nstamp < a.trace_cap) a.trace[nstamp] = global_ns();
        ++nstamp;
    };
    stamp();
    agg_clear(sm.agg);
    uint32_t hot = hot_threshold(a.hot_deg, team.size);
    bool solo = team.size == 1;
    uint32_t size = team.size;  // blocks at work
    if (tid < 2) sm.cursor[tid] = 0;
    if (tid < 4) {
        sm.add[tid] = 0;
        sm.cum[tid] = 0;
    }
    __syncwarp();  // cleared by four threads, then set by one of them
    if (tid == 0) {
        meet_init(sm.meet, a.arrivals0);
        sm.cum[0] = resume ? (uint64_t)a.n - a.S0 : 0;
        sm.cum[1] = resume ? 2 * (a.m - a.E0) : 0;
        sm.cum[4] = 0;
        sm.agg_used = 0;
        sm.scanned = 0;
    }
    if (team.rank == 0 && tid == 0 && !resume && a.hist_S) {
        a.hist_S[0] = S;
        a.hist_E[0] = E;
    }
    if (a.hot_deg == 0 && a.n >= kHubCountMin && team.size > 1) {
        // hubs: the vertices of the 2^b least above which at most kHubsMax lie, b >= kHubBit0
        if (tid < kHubBits) sm.wit[tid] = 0;
        __syncthreads();
        for (uint64_t v = (uint64_t)team.rank * TB + tid; v < a.n; v += (uint64_t)team.size * TB) {
            const uint32_t len = (uint32_t)(a.off[v + 1] - a.off[v]);
            if (len >> kHubBit0) atomicAdd(&sm.wit[min(31u - (uint32_t)__clz(len) - kHubBit0, kHubBits - 1)], 1u);
        }
        __syncthreads();
        if (tid < kHubBits && sm.wit[tid]) atomicAdd(&ctl->hubs[tid], sm.wit[tid]);
        team.meet(0u, sm.meet);
        if (!sm.meet.ok) return {};
        uint32_t above = 0, b = kHubBits;
        while (b > 0 && (above += ld_volatile_u32(&ctl->hubs[b - 1])) <= kHubsMax) --b;
        hot = 1u << (kHubBit0 + min(b, kHubBits - 1));
    }
    while (S > 0) {
        // one thread divides for the block: the division is a few hundred instructions, which
        // every warp of a full SM would pay for one after the other
        if (tid == 0) sm.threshold = peel_threshold(a.p, a.q, E, S);
        __syncthreads();
        const uint32_t T = sm.threshold;
        const uint32_t mark = kDead | (uint32_t)(r + 1);
        // ------------------------------------------------ phase 1: test + compact
        // the first round of a launch walks vertex ids in order (every vertex, or
        // every vertex a resumed peel has not failed yet) and writes the status map
        // whole, two words per warp; later rounds walk the alive list and set the
        // failures' bits
        const bool fresh = r == 0;                  // identity list, degrees from the rows
        const bool scan_all = !alive && resume;     // a resumed peel's first round: every vertex, failed ones skipped
        const bool by_id = fresh || scan_all;
        // thin: the last round removed less than 1/8 of the vertices; then this round collects the
        // next round's candidates (bound Bn), and it is lazy when the current list covers T
        // (unless the last collections were too long to be of use: see below)
        const bool thin = lazy_ok && !solo && !fresh && (S_prev - S) * 8 < S_prev && r >= cand_from;
        const bool lazy = thin && have_cands && !by_id && T <= B && cand_n * 4 < S;
        const uint32_t Bn = lazy ? B : (thin ? T + T / 128u : 0u);
        const uint64_t span = by_id ? (scan_all ? a.n : S) : (lazy ? cand_n : alive_len);
        const uint32_t* src = lazy ? cur_cand : alive;
        tested += span;
        lazy_rounds += lazy ? 1u : 0u;
        // a tile is `items` slices of TB (thread tid takes i = t + j TB + tid for j < items), four or
        // two where there is enough to test (their loads in flight together), else one; a list shorter
        // than the blocks' threads is spread over the blocks, `width` entries each (a hub's pieces
        // are written by its warp).  The first pass tests and marks, the second writes the lists at
        // the tile's reserved places
        const uint64_t threads = (uint64_t)size * TB;
        const uint32_t width = by_id || span >= threads ? TB : (uint32_t)((span + size - 1) / size);
        uint64_t X = 0, rows = 0;
        uint32_t nfail = 0, pushed = 0;  // this thread's failures; thread 0: pieces queued by the block
        auto test = [&](auto slices) {
            constexpr uint32_t items = decltype(slices)::value;
            for (uint64_t t = (uint64_t)team.rank * width * items; t < span; t += (uint64_t)size * width * items) {
                uint32_t fail_m = 0, surv_m = 0, cand_m = 0, nit = 0;
                uint32_t tv[items], td[items], tl[items];
                bool in[items];
#pragma unroll
                for (uint32_t j = 0; j < items; ++j) {
                    const uint64_t i = t + (uint64_t)j * TB + tid;
                    in[j] = tid < width && i < span;
                    tv[j] = in[j] ? (by_id ? (uint32_t)i : src[i]) : 0u;
                }
#pragma unroll
                for (uint32_t j = 0; j < items; ++j) {
                    // row lengths beside the states, not after the test: one round trip less
                    tl[j] = in[j] ? (uint32_t)(a.off[tv[j] + 1] - a.off[tv[j]]) : 0u;
                    td[j] = in[j] && !fresh ? a.st[tv[j]] : tl[j];
                }
#pragma unroll
                for (uint32_t j = 0; j < items; ++j) {
                    const uint32_t v = tv[j], d = td[j], len = tl[j];
                    const bool gone = (d & kDead) != 0;  // failed in an earlier round (a resumed peel's first, or a list
                                                         // left from before lazy rounds)
                    bool fail = false;
                    if (in[j] && scan_all && gone) rows += len;
                    if (in[j] && !gone) {
                        fail = d <= T;
                        if (fail) {
                            a.st[v] = mark;
                            X += d;
                            rows += len;
                            ++nfail;
                            nit += len <= a.chunk_len ? (len ? 1u : 0u) : (len + a.chunk_len - 1) / a.chunk_len;
                            fail_m |= 1u << j;
                            if (!by_id) atomicOr(&a.map[v >> 4], 1u << (2u * (v & 15u)));
                        } else {
                            if (!lazy) surv_m |= 1u << j;
                            if (thin && d <= Bn) cand_m |= 1u << j;
                            if (fresh) a.st[v] = d;
                        }
                    }
                    if (by_id) {
                        // each warp holds 32 consecutive ids starting at a multiple of 32
                        const uint32_t bd = __ballot_sync(kFullMask, fail || (in[j] && gone));
                        const uint32_t bh = __ballot_sync(kFullMask, in[j] && len >= hot);
                        const uint64_t i0 = t + (uint64_t)j * TB + (tid & ~31u);
                        if (lane == 0 && i0 < a.n) a.map[i0 >> 4] = spread16(bd) | (spread16(bh) << 1);
                        if (lane == 16 && i0 + 16 < a.n)
                            a.map[(i0 >> 4) + 1] = spread16(bd >> 16) | (spread16(bh >> 16) << 1);
                    }
                }
                // survivors go to the next list in id order within the tile (slice, then
                // warp, then lane), so the next round reads the states in order
                for (uint32_t j = 0; j < items; ++j) {
                    const uint32_t c = __popc(__ballot_sync(kFullMask, surv_m >> j & 1u));
                    if (lane == 0) sm.surv_at[j][warp] = c;
                }
                const uint32_t it_inc = warp_incl_scan(nit);
                if (lane == 31) sm.wit[warp] = it_inc;
                __syncthreads();
                if (tid < 32) {
                    // exclusive prefixes of the warps' pieces and of the (slice, warp)
                    // survivor counts, slice-major; the tile's share of both lists
                    const uint32_t c = tid < kW ? sm.wit[tid] : 0u;
                    const uint32_t ci = warp_incl_scan(c);
                    if (tid < kW) sm.wit[tid] = ci - c;
                    const uint32_t nt = __shfl_sync(kFullMask, ci, 31);
                    constexpr uint32_t per = (items * kW + 31) / 32;  // counts per lane, consecutive
                    uint32_t loc[per], sum = 0;
                    for (uint32_t q = 0; q < per; ++q) {
                        const uint32_t idx = tid * per + q;
                        loc[q] = idx < items * kW ? sm.surv_at[idx / kW][idx % kW] : 0u;
                        sum += loc[q];
                    }
                    const uint32_t inc = warp_incl_scan(sum);
                    const uint32_t nv = __shfl_sync(kFullMask, inc, 31);
                    uint32_t run = inc - sum;
                    for (uint32_t q = 0; q < per; ++q) {
                        const uint32_t idx = tid * per + q;
                        if (idx < items * kW) sm.surv_at[idx / kW][idx % kW] = run;
                        run += loc[q];
                    }
                    pushed += nt;
                    if (tid < 2) {
                        const uint32_t want = tid == 0 ? nt : nv;
                        unsigned long long b = 0;
                        if (solo) {
                            b = sm.cursor[tid];
                            sm.cursor[tid] = b + want;
                        } else if (want) {
                            b = atomicAdd(tid == 0 ? &ctl->items : &ctl->surv, (unsigned long long)want);
                        }
                        sm.base[tid] = b;
                    }
                }
                __syncthreads();
                uint64_t at = sm.base[0] + sm.wit[warp] + (it_inc - nit);
                const uint64_t v0 = sm.base[1] - surv_base;
#pragma unroll
                for (uint32_t j = 0; j < items; ++j) {
                    const uint32_t v = tv[j], len = tl[j];
                    uint32_t np = 0;
                    uint64_t b0 = 0;
                    if (fail_m >> j & 1u) {
                        b0 = a.off[v];
                        np = len <= a.chunk_len ? (len ? 1u : 0u) : (len + a.chunk_len - 1) / a.chunk_len;
                    }
                    if (np == 1) a.items[at] = b0 << kLenBits | len;
                    {
                        const uint32_t sb = __ballot_sync(kFullMask, surv_m >> j & 1u);
                        if (surv_m >> j & 1u) next[v0 + sm.surv_at[j][warp] + __popc(sb & lanemask_lt())] = v;
                        // candidates for the next round: one atomic per warp
                        const uint32_t cb = __ballot_sync(kFullMask, cand_m >> j & 1u);
                        if (cb) {
                            unsigned long long cbase = 0;
                            if (lane == 0) cbase = atomicAdd(&ctl->cand, (unsigned long long)__popc(cb));
                            cbase = __shfl_sync(kFullMask, cbase, 0);
                            if (cand_m >> j & 1u) next_cand[cbase - cand_base + __popc(cb & lanemask_lt())] = v;
                        }
                    }
                    // the pieces of the warp's long failures, written by the whole warp
                    // (a hub has hundreds of them)
                    for (uint32_t pend = __ballot_sync(kFullMask, np > 1); pend; pend &= pend - 1) {
                        const uint32_t o = __ffs(pend) - 1;
                        const uint32_t on = __shfl_sync(kFullMask, np, o);
                        const uint32_t ol = __shfl_sync(kFullMask, len, o);
                        const uint64_t ob = __shfl_sync(kFullMask, b0, o), oa = __shfl_sync(kFullMask, at, o);
                        for (uint32_t c = lane; c < on; c += 32) {
                            const uint32_t k = c * a.chunk_len;
                            a.items[oa + c] = (ob + k) << kLenBits | min(a.chunk_len, ol - k);
                        }
                    }
                    at += np;
                }
                __syncthreads();  // the tile's totals are read before the next tile writes its own
            }
        };
        if (span >= 4 * threads) test(std::integral_constant<uint32_t, 4>{});
        else if (!CL && span > threads) test(std::integral_constant<uint32_t, 2>{});
        else test(std::integral_constant<uint32_t, 1>{});
        {
            X = warp_sum(X);
            rows = warp_sum(rows);
            nfail = __reduce_add_sync(kFullMask, nfail);
            if (lane == 0 && (nfail || rows)) {
                atomicAdd(&sm.add[0], (unsigned long long)nfail);
                atomicAdd(&sm.add[1], (unsigned long long)X);
                atomicAdd(&sm.add[2], (unsigned long long)rows);
            }
        }
        __syncthreads();
        if (tid < 3) {
            const unsigned long long x = sm.add[tid];
            sm.add[tid] = 0;
            if (solo) sm.cum[tid] += x;
            else if (x) atomicAdd(tid == 0 ? &ctl->failed : tid == 1 ? &ctl->xsum : &ctl->rows, x);
        }
        const uint32_t got = team.meet(pushed, sm.meet);
        if (!sm.meet.ok) return {};
        stamp();
        if (S <= kLastMax) {
            // every vertex left has failed: no neighbour is left to take a degree from
            if (tid == 0) sm.last = (solo ? sm.cum[0] : ld_volatile_u64((const uint64_t*)&ctl->failed)) == a.n;
            __syncthreads();
            if (sm.last) {
                ++r;
                if (team.rank == 0 && tid == 0) {
                    if (!a.hist_S) {
                    } else if (r < a.hist_cap) a.hist_S[r] = a.hist_E[r] = 0;
                    else atomicOr(&ctl->err, ERR_CAPACITY);
                }
                S = E = 0;
                stamp();
                break;
            }
        }
        // ------------------------------------------------ phase 2: neighbour scan
        uint32_t ndec = 0;
        uint32_t* st = a.st;
        const uint32_t* map = a.map;
        {
            const uint64_t gw = (uint64_t)team.rank * kW + warp, nw = (uint64_t)size * kW;
            // pieces per warp and turn, the same for every turn.  Many turns: consecutive pieces
            // (neighbouring rows share sectors); few: pieces nw apart (a hub's pieces go to
            // different warps)
            const uint64_t turns = ((uint64_t)got + 32 * nw - 1) / (32 * nw);
            const uint32_t G = turns ? (uint32_t)((got + nw * turns - 1) / (nw * turns)) : 1u;
            const bool packed = turns > 2;
            const uint64_t s_lane = packed ? 1 : nw, s_warp = packed ? G : 1;
            for (uint64_t g0 = 0; g0 < got; g0 += nw * G) {
                const uint64_t i = g0 + lane * s_lane + gw * s_warp;
                uint64_t it = 0;
                if (lane < G && i < got) it = __ldcg(a.items + item_lo + i);
                const uint32_t len = (uint32_t)it & ((1u << kLenBits) - 1u);
                const uint32_t inc = warp_incl_scan(len);
                const uint32_t total = __shfl_sync(kFullMask, inc, 31);
                const uint32_t begin = inc - len;
                const uint64_t b0 = (it >> kLenBits) - begin;  // entry e of the group is adj[b0 + e] for its owner's b0
                uint64_t* const own = sm.own[warp];
                if (G > 1) {
                    __syncwarp();
                    const uint32_t nz = __ballot_sync(kFullMask, len != 0);
                    if (len) own[__popc(nz & lanemask_lt())] = b0;
                    __syncwarp();
                }
                for (uint32_t e0 = lane; e0 < ((total + 31u) & ~31u); e0 += 32 * kBatch) {
                    uint32_t u[kBatch], w[kBatch];
                    // owner: the last piece that starts at or before e, by counting the pieces' starts in a
                    // map of the step's positions (a five-step shuffle search per entry before: 1,500
                    // graphs in one batch 2.52 -> 2.37 ms, 3 10^6 vertices 689 -> 681 us)
                    const uint32_t e_lo = e0 - lane;
                    uint32_t before = G > 1 ? __popc(__ballot_sync(kFullMask, len != 0 && begin < e_lo)) : 0u;
                    const uint32_t rel = len != 0 && begin >= e_lo ? begin - e_lo : 0xffffffffu;
#pragma unroll
                    for (uint32_t j = 0; j < kBatch; ++j) {
                        const uint32_t e = e0 + 32 * j;
                        uint64_t ob;
                        if (G > 1) {
                            const uint32_t m = __reduce_or_sync(kFullMask, (rel >> 5) == j ? 1u << (rel & 31u) : 0u);
                            ob = own[before + __popc(m & (0xffffffffu >> (31u - lane))) - 1u];
                            before += __popc(m);
                        } else {
                            ob = __shfl_sync(kFullMask, b0, 0);
                        }
                        u[j] = e < total ? ld_stream(a.adj + ob + e) : 0xffffffffu;
                    }
#pragma unroll
                    for (uint32_t j = 0; j < kBatch; ++j) {
                        const bool valid = e0 + 32 * j < total;
#ifdef DSG_DEBUG_BOUNDS
                        if (valid && u[j] >= a.n) atomicOr(&ctl->err, ERR_RANGE);
                        w[j] = valid && u[j] < a.n ? map[u[j] >> 4] >> (2u * (u[j] & 15u)) : 1u;
#else
                        w[j] = valid ? map[u[j] >> 4] >> (2u * (u[j] & 15u)) : 1u;
#endif
                    }
#pragma unroll
                    for (uint32_t j = 0; j < kBatch; ++j) {
                        if (w[j] & 1u) continue;
                        // alive: one degree less (hubs' decrements combined in the block); in a thin
                        // round the decrement that takes a degree to the bound makes it a candidate
                        if ((w[j] & 2u) && agg_add(sm.agg, u[j])) {
                            sm.agg_used = 1;
                        } else if (thin) {
                            const uint32_t old = atomicSub(&st[u[j]], 1u);
                            if (old > Bn && old - 1u <= Bn) next_cand[atomicAdd(&ctl->cand, 1ull) - cand_base] = u[j];
                        } else {
                            atomicSub(&st[u[j]], 1u);
                        }
                        ++ndec;
                    }
                }
            }
        }
        ndec = __reduce_add_sync(kFullMask, ndec);
        if (lane == 0 && ndec) atomicAdd(&sm.add[3], (unsigned long long)ndec);
        __syncthreads();
        // flush the combined hub decrements
        if (sm.agg_used) {
            for (uint32_t i = tid; i < kAggSlots; i += TB) {
                uint32_t key = sm.agg.key[i];
                if (key != kAggEmpty) {
                    const uint32_t c = sm.agg.cnt[i];
                    if (thin) {
                        const uint32_t old = atomicSub(&st[key], c);
                        if (old > Bn && old - c <= Bn) next_cand[atomicAdd(&ctl->cand, 1ull) - cand_base] = key;
                    } else {
                        atomicSub(&st[key], c);
                    }
                    sm.agg.key[i] = kAggEmpty;
                    sm.agg.cnt[i] = 0;
                }
            }
        }
        if (tid == 0) {
            const unsigned long long x = sm.add[3];
            sm.add[3] = 0;
            if (solo) sm.cum[3] += x;
            else if (x) atomicAdd(&ctl->dec, x);
        }
        team.meet(0u, sm.meet);
        if (!sm.meet.ok) return {};
        stamp();
        if (tid == 0) sm.agg_used = 0;
        if (!solo) {
            if (tid < 5)
                sm.cum[tid] = ld_volatile_u64((const uint64_t*)(tid == 0   ? &ctl->failed
                                                                : tid == 1 ? &ctl->xsum
                                                                : tid == 2 ? &ctl->rows
                                                                : tid == 3 ? &ctl->dec
                                                                           : &ctl->cand));
            __syncthreads();
        }
        // edges removed so far: (X + D) / 2 summed over the rounds
        const uint64_t removed = (sm.cum[1] + sm.cum[3]) / 2;
        const uint64_t S1 = (uint64_t)a.n - sm.cum[0];
        const uint64_t E1 = a.m - removed;
        const uint64_t rows_left = 2 * a.m - sm.cum[2], cand_hi = sm.cum[4];
        ++r;
        if (team.rank == 0 && tid == 0) {
            sm.scanned = sm.cum[2];
            if (!a.hist_S) {
            } else if (r < a.hist_cap) {
                a.hist_S[r] = S1;
                a.hist_E[r] = E1;
            } else {
                atomicOr(&ctl->err, ERR_CAPACITY);
            }
        }
        if (S1 > 0 && (unsigned __int128)E1 * best_V > (unsigned __int128)best_E * S1) {
            best_round = r;
            best_E = E1;
            best_V = S1;
        }
        item_lo += got;
        if (!lazy) {  // a lazy round leaves the alive list as it was (its failures are skipped later)
            surv_base += S1;
            alive_len = S1;
            alive = next;
            next = (next == a.listA) ? a.listB : a.listA;
        }
        {
            if (thin) {
                uint32_t* t_ = cur_cand;
                cur_cand = next_cand;
                next_cand = t_;
                cand_n = cand_hi - cand_base;
                B = Bn;
                // a list that is no use to the next round (most degrees lie just above the threshold)
                // costs more than testing everyone: an atomic per warp of the alive list (nested shells
                // of 265,100 vertices: 12.5 us a round's test against 8).  Rest before the next try,
                // longer each time
                if (cand_n * 4 >= S1) {
                    cand_from = r + cand_rest;
                    cand_rest = min(2 * cand_rest, (uint64_t)64);
                } else {
                    cand_rest = 2;
                }
            }
            have_cands = thin;
            cand_base = cand_hi;
        }
        S_prev = S;
        S = S1;
        E = E1;
        if (r >= a.hist_cap) break;
        if (a.max_rounds && r - a.r0 >= a.max_rounds) break;  // pause: the state stays in st
        if (!CL && !solo && rows_left <= kSoloEntries && alive_len <= kSoloList) {
            // little is left: block 0 goes on alone
            if (team.rank != 0) return {};
            solo = true;
            size = team.size = 1;
            if (tid == 0) sm.cursor[0] = item_lo;
            if (tid == 1) sm.cursor[1] = surv_base;
        }
        __syncthreads();  // the round's sums are read before the next round changes them
    }
    if (team.rank == 0 && tid == 0) {
        ctl->stamps = nstamp;
        ctl->rounds = r;
        ctl->best_round = best_round;
        ctl->best_E = best_E;
        ctl->best_V = best_V;
        ctl->cur_S = S;
        ctl->cur_E = E;
        ctl->dec = sm.cum[3];
        ctl->tested = tested;
        ctl->lazy_rounds = lazy_rounds;
        ctl->scanned = sm.scanned;
    }
    return {r, best_round, best_E, best_V};
}

}  // namespace dsg
