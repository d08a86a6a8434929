// Algorithm 1 on one graph: launches, results, the side-by-side solve, the
// no-allocation variant, and peels that are paused and resumed.  The rounds
// are in peel_body.cuh.
#include <algorithm>
#include <cstdlib>
#include <string>
#include <thread>
#include <vector>

#include "dsg_common.cuh"
#include "dsg_kernels.cuh"
#include "peel_body.cuh"

namespace dsg {

template <int TB>
__global__ void __launch_bounds__(TB, 1024 / TB) peel_kernel(PeelArgs a) {
    __shared__ PeelSmem<TB> sm;
    Team<false> team{blockIdx.x, gridDim.x, a.ctl->bar, &a.ctl->err, a.limit_ns};
    peel_body<TB, false>(a, team, sm);
}

// The whole peel of a small graph by one cluster: the control block in shared
// memory (copied to a.ctl at the end), and the results written in the same
// launch (peel_round, set: nullable).  One block per SM: at 64 registers, for
// two, it spilled (10,000 vertices: kernel 65.5 against 61.3 us).
constexpr uint32_t kSmallTB = 512;

__global__ void __launch_bounds__(kSmallTB, 1) peel_cluster_kernel(PeelArgs a, uint32_t* peel_round, uint8_t* set) {
    __shared__ PeelSmem<kSmallTB> sm;
    __shared__ PeelCtl ctl;
    PeelCtl* const global = a.ctl;
    a.ctl = at_block0(&ctl);
    const uint32_t rank = cluster_rank(), tid = threadIdx.x;
    uint32_t* const words = reinterpret_cast<uint32_t*>(&ctl);
    if (rank == 0)
        for (uint32_t i = tid; i < sizeof(PeelCtl) / 4; i += kSmallTB) words[i] = 0;
    cluster_sync();
    const PeelOut o =
        peel_body<kSmallTB, true>(a, Team<true>{rank, kSmallBlocks, a.ctl->bar, &a.ctl->err, 0}, sm);
    for (uint32_t v = rank * kSmallTB + tid; v < a.n; v += kSmallBlocks * kSmallTB) {
        const uint32_t pr = __ldcg(a.st + v) & ~kDead;
        if (peel_round) peel_round[v] = pr;
        if (set) set[v] = pr > o.best_round ? 1 : 0;
    }
    cluster_sync();  // no block leaves while another reads block 0's shared memory
    if (rank == 0)
        for (uint32_t i = tid; i < sizeof(PeelCtl) / 4; i += kSmallTB) reinterpret_cast<uint32_t*>(global)[i] = words[i];
}

// Vertices plus row entries up to which one cluster peels (us, cluster / grid
// with its second launch for the results: work of 28,000 73 / 83, 113,000
// 81 / 86, 168,000 94 / 100, 244,000 81 / 83, 337,000 107 / 112, 372,000
// 106 / 89, 929,000 143 / 95).
constexpr uint64_t kSmallPeel = 250000;

// peel_round[v] = round v failed; set[v] = peel_round > best_round.
__global__ void peel_finish_kernel(uint32_t n, const uint32_t* __restrict__ st, const PeelCtl* __restrict__ ctl,
                                   uint32_t* __restrict__ peel_round, uint8_t* __restrict__ set) {
    uint64_t br = ctl->best_round;
    for (uint64_t v = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (uint64_t)gridDim.x * blockDim.x) {
        uint32_t pr = st[v] & ~kDead;
        if (peel_round) peel_round[v] = pr;
        if (set) set[v] = pr > br ? 1 : 0;
    }
}

// wrap_in (0: off): the meeting words start as if so many blocks had arrived
// that they pass 2^32 arrivals after that many rounds.
template <int TB>
static cudaError_t launch_peel(PeelArgs& a, uint32_t blocks_per_sm, cudaStream_t s, uint32_t max_grid,
                               uint32_t wrap_in = 0) {
    uint32_t grid = 1;
    cudaError_t e = coop_grid(peel_kernel<TB>, TB, 0, a.n, blocks_per_sm, &grid, max_grid);
    if (e != cudaSuccess) return e;
    if (wrap_in) {
        a.arrivals0 = (uint32_t)(((1ull << 32) / grid - wrap_in) * grid);
        const unsigned long long before = a.arrivals0;
        for (int w = 0; w < 2 && e == cudaSuccess; ++w)
            e = cudaMemcpyAsync(&a.ctl->bar[w][0], &before, sizeof(before), cudaMemcpyHostToDevice, s);
        if (e != cudaSuccess) return e;
    }
    void* params[] = {&a};
    LaunchScope ls("peel_rounds", s);
    return cudaLaunchCooperativeKernel((const void*)peel_kernel<TB>, dim3(grid), dim3(TB), params, 0, s);
}

// Entries of a row piece.
static uint32_t piece_len(const Tuning& tu) { return std::min<uint32_t>(tu.chunk_len, (1u << kLenBits) - 1u); }

// Run the peel; results land in the returned control block and, if given,
// in hist / peel_round / set (device pointers).
static dsg_status run_peel(const dsg_graph* g, uint32_t p, uint32_t q, uint64_t* hist_S_out, uint64_t* hist_E_out,
                           uint64_t hist_cap_out, uint32_t* peel_round_out, uint8_t* set_out, PeelCtl* ctl_host,
                           uint64_t* trace_dev = nullptr, uint64_t trace_cap = 0, uint32_t wrap_in = 0);

dsg_status peel_into(const dsg_graph* g, uint32_t p, uint32_t q, uint8_t* set_dev, uint64_t out4[4],
                     uint64_t* extra2) {
    PeelCtl c;
    dsg_status st;
    if (extra2 && g->n) {
        // the byte model's counters too: sum of |S_r| over the rounds (from the history) and the decrements
        const uint64_t cap = dsg_round_bound(g->n, p, q) + 1;
        std::vector<uint64_t> hs(cap);
        st = run_peel(g, p, q, hs.data(), nullptr, cap, nullptr, set_dev, &c);
        if (st != DSG_OK) return st;
        uint64_t sum = 0;
        for (uint64_t r = 0; r < c.rounds && r < cap; ++r) sum += hs[r];
        extra2[0] = sum;
        extra2[1] = c.dec;
    } else {
        st = run_peel(g, p, q, nullptr, nullptr, 0, nullptr, set_dev, &c);
    }
    if (st != DSG_OK) return st;
    out4[0] = g->n ? c.best_E : 0;
    out4[1] = g->n ? c.best_V : 0;
    out4[2] = c.rounds;
    out4[3] = c.best_round;
    return DSG_OK;
}

static dsg_status run_peel(const dsg_graph* g, uint32_t p, uint32_t q, uint64_t* hist_S_out, uint64_t* hist_E_out,
                           uint64_t hist_cap_out, uint32_t* peel_round_out, uint8_t* set_out, PeelCtl* ctl_host,
                           uint64_t* trace_dev, uint64_t trace_cap, uint32_t wrap_in) {
    cudaStream_t s = g->stream;
    const uint32_t n = g->n;
    Tuning tu = tuning_for(g, 0);
    if (g->force_block) tu.block = g->force_block;
    memset(ctl_host, 0, sizeof(PeelCtl));
    if (n == 0) {
        static const uint64_t zero = 0;
        if (hist_S_out && hist_cap_out) DSG_TRY_CUDA(copy_any(hist_S_out, &zero, sizeof(uint64_t), s));
        if (hist_E_out && hist_cap_out) DSG_TRY_CUDA(copy_any(hist_E_out, &zero, sizeof(uint64_t), s));
        DSG_TRY_CUDA(cudaStreamSynchronize(s));
        return DSG_OK;
    }
    uint64_t cap = dsg_round_bound(n, p, q) + 1;
    Scratch sc(s);
    PeelArgs a;
    a.n = n;
    a.m = g->m;
    a.p = p;
    a.q = q;
    a.off = g->off;
    a.adj = g->adj;
    a.hist_cap = cap;
    a.limit_ns = wait_limit_ns();
    a.chunk_len = piece_len(tu);
    const uint64_t item_cap = (uint64_t)n + (2 * g->m) / a.chunk_len + 1;
    a.hot_deg = tu.hot_deg;
    a.trace = trace_dev;
    a.trace_cap = trace_cap;
    a.r0 = a.S0 = a.E0 = a.best_round0 = a.best_E0 = a.best_V0 = a.max_rounds = a.arrivals0 = 0;
    const bool lazy = current_tuning().peel_lazy != 0;
    const bool pr_direct = peel_round_out && is_device_ptr(peel_round_out);
    const bool set_direct = set_out && is_device_ptr(set_out);
    uint32_t* pr_dev = peel_round_out && pr_direct ? peel_round_out : nullptr;
    uint8_t* set_dev = set_out && set_direct ? set_out : nullptr;
    {
        // one allocation for all of it
        size_t o = 0;
        auto carve = [&](size_t bytes) { const size_t at = o; o += (bytes + 255) & ~size_t(255); return at; };
        const size_t nb = (size_t)n * 4;
        const size_t o_ctl = carve(sizeof(PeelCtl)), o_st = carve(nb), o_a = carve(nb), o_b = carve(nb),
                     o_items = carve(item_cap * 8), o_map = carve(((size_t)n + 15) / 16 * 4),
                     o_ca = carve(lazy ? nb : 0), o_cb = carve(lazy ? nb : 0), o_hs = carve(cap * 8),
                     o_he = carve(cap * 8), o_pr = carve(peel_round_out && !pr_direct ? nb : 0),
                     o_set = carve(set_out && !set_direct ? n : 0);
        unsigned char* w;
        DSG_TRY_CUDA(sc.get(&w, o));
        a.ctl = reinterpret_cast<PeelCtl*>(w + o_ctl);
        a.st = reinterpret_cast<uint32_t*>(w + o_st);
        a.listA = reinterpret_cast<uint32_t*>(w + o_a);
        a.listB = reinterpret_cast<uint32_t*>(w + o_b);
        a.items = reinterpret_cast<uint64_t*>(w + o_items);
        a.map = reinterpret_cast<uint32_t*>(w + o_map);
        a.candA = lazy ? reinterpret_cast<uint32_t*>(w + o_ca) : nullptr;
        a.candB = lazy ? reinterpret_cast<uint32_t*>(w + o_cb) : nullptr;
        a.hist_S = reinterpret_cast<uint64_t*>(w + o_hs);
        a.hist_E = reinterpret_cast<uint64_t*>(w + o_he);
        if (peel_round_out && !pr_direct) pr_dev = reinterpret_cast<uint32_t*>(w + o_pr);
        if (set_out && !set_direct) set_dev = w + o_set;
    }
    const bool small = !wrap_in && n + 2 * g->m <= kSmallPeel && (g->max_blocks == 0 || g->max_blocks >= kSmallBlocks) &&
                       clusters_fit(peel_cluster_kernel, kSmallBlocks, kSmallTB, 0) > 0;
    if (small) {
        LaunchScope ls("peel_rounds", s);
        DSG_TRY_CUDA(launch_cluster(peel_cluster_kernel, kSmallBlocks, kSmallTB, 0, s, a, pr_dev, set_dev));
    } else {
        DSG_TRY_CUDA(cudaMemsetAsync(a.ctl, 0, sizeof(PeelCtl), s));
        cudaError_t e;
        switch (tu.block) {
            case 256: e = launch_peel<256>(a, tu.blocks_per_sm, s, g->max_blocks, wrap_in); break;
            case 1024: e = launch_peel<1024>(a, tu.blocks_per_sm, s, g->max_blocks, wrap_in); break;
            default: e = launch_peel<512>(a, tu.blocks_per_sm, s, g->max_blocks, wrap_in); break;
        }
        DSG_TRY_CUDA(e);
        if (pr_dev || set_dev) {
            uint64_t want = ((uint64_t)n + 255) / 256, cap_b = (uint64_t)dev_info().sms * 8;
            uint32_t blocks = (uint32_t)(want < cap_b ? want : cap_b);
            LaunchScope ls("peel_finish", s);
            peel_finish_kernel<<<blocks, 256, 0, s>>>(n, a.st, a.ctl, pr_dev, set_dev);
            DSG_TRY_CUDA(cudaGetLastError());
        }
    }
    DSG_TRY_CUDA(cudaMemcpyAsync(ctl_host, a.ctl, sizeof(PeelCtl), cudaMemcpyDeviceToHost, s));
    DSG_TRY_CUDA(cudaStreamSynchronize(s));
    dsg_status st = status_from_err(ctl_host->err, "bahmani peel");
    if (st != DSG_OK) return st;
    uint64_t R = ctl_host->rounds;
    if (hist_S_out || hist_E_out) {
        uint64_t k = R + 1 < hist_cap_out ? R + 1 : hist_cap_out;
        if (hist_S_out) DSG_TRY_CUDA(copy_any(hist_S_out, a.hist_S, k * sizeof(uint64_t), s));
        if (hist_E_out) DSG_TRY_CUDA(copy_any(hist_E_out, a.hist_E, k * sizeof(uint64_t), s));
    }
    if (peel_round_out && !pr_direct) DSG_TRY_CUDA(copy_any(peel_round_out, pr_dev, (size_t)n * 4, s));
    if (set_out && !set_direct) DSG_TRY_CUDA(copy_any(set_out, set_dev, (size_t)n, s));
    DSG_TRY_CUDA(cudaStreamSynchronize(s));
    return DSG_OK;
}

}  // namespace dsg

using namespace dsg;

extern "C" {

dsg_status dsg_bahmani(const dsg_graph* g, uint32_t eps_num, uint32_t eps_den, uint8_t* out_set, uint64_t* out_E,
                       uint64_t* out_V) {
    clear_error();
    DSG_CHECK_ARG(g, "graph is NULL");
    DSG_CHECK_ARG(eps_den != 0, "eps_den must be positive");
    DSG_TRY_CUDA(cudaSetDevice(g->device));
    PeelCtl c;
    dsg_status st = run_peel(g, eps_num, eps_den, nullptr, nullptr, 0, nullptr, out_set, &c);
    if (st != DSG_OK) return st;
    if (out_E) *out_E = g->n ? c.best_E : 0;
    if (out_V) *out_V = g->n ? c.best_V : 0;
    return DSG_OK;
}

// Peels at several eps and the core numbers of one graph.  The two kinds of
// solve are independent, so they may run side by side: the peels on one
// internal stream and the core numbers on another (from a second host thread,
// since each solve waits for its stream), each kernel with 1024-thread blocks
// on at most half the SMs -- one block per SM, so the two grids fit the GPU
// together.  Both streams start after the graph's stream, and the graph's
// stream waits for both before the call returns.
dsg_status dsg_solve(const dsg_graph* g, uint32_t count, const uint32_t* eps_num, const uint32_t* eps_den,
                     uint8_t* const* out_sets, uint64_t* out_E, uint64_t* out_V, uint32_t* out_core) {
    clear_error();
    DSG_CHECK_ARG(g, "graph is NULL");
    DSG_CHECK_ARG(count == 0 || (eps_num && eps_den), "eps arrays are NULL");
    for (uint32_t i = 0; i < count; ++i) DSG_CHECK_ARG(eps_den[i] != 0, "eps_den must be positive");
    DSG_TRY_CUDA(cudaSetDevice(g->device));
    auto peels = [&](const dsg_graph* h) -> dsg_status {
        for (uint32_t i = 0; i < count; ++i) {
            PeelCtl c;
            dsg_status st =
                run_peel(h, eps_num[i], eps_den[i], nullptr, nullptr, 0, nullptr, out_sets ? out_sets[i] : nullptr, &c);
            if (st != DSG_OK) return st;
            if (out_E) out_E[i] = g->n ? c.best_E : 0;
            if (out_V) out_V[i] = g->n ? c.best_V : 0;
        }
        return DSG_OK;
    };
    // side by side only pays when the peels are a fair share of the work:
    // each kind then runs on half the GPU; when the autotuned times of this
    // graph's size class say the core numbers dominate, run one after the
    // other with the whole GPU each
    double peel_ms = 0, core_ms = 0;
    const bool tuned = tuned_times(g, &peel_ms, &core_ms);
    const bool mostly_core = tuned && count * peel_ms < 0.25 * core_ms;
    if (count == 0 || !out_core || g->n == 0 || mostly_core) {
        dsg_status st = peels(g);
        if (st != DSG_OK || !out_core) return st;
        return run_kcore(g, out_core, nullptr, 0);
    }
    const uint32_t sms = (uint32_t)dev_info().sms;
    // two streams and three events per calling thread and device, made once
    struct SideBySide {
        int device = -1;
        cudaStream_t sa = nullptr, sb = nullptr;
        cudaEvent_t ev0 = nullptr, eva = nullptr, evb = nullptr;
    };
    static thread_local SideBySide cache[16];
    SideBySide& sbs = cache[g->device & 15];
    if (sbs.device != g->device) {
        DSG_TRY_CUDA(cudaStreamCreateWithFlags(&sbs.sa, cudaStreamNonBlocking));
        DSG_TRY_CUDA(cudaStreamCreateWithFlags(&sbs.sb, cudaStreamNonBlocking));
        DSG_TRY_CUDA(cudaEventCreateWithFlags(&sbs.ev0, cudaEventDisableTiming));
        DSG_TRY_CUDA(cudaEventCreateWithFlags(&sbs.eva, cudaEventDisableTiming));
        DSG_TRY_CUDA(cudaEventCreateWithFlags(&sbs.evb, cudaEventDisableTiming));
        sbs.device = g->device;
    }
    cudaStream_t sa = sbs.sa, sb = sbs.sb;
    cudaEvent_t ev0 = sbs.ev0, eva = sbs.eva, evb = sbs.evb;
    DSG_TRY_CUDA(cudaEventRecord(ev0, g->stream));
    DSG_TRY_CUDA(cudaStreamWaitEvent(sa, ev0, 0));
    DSG_TRY_CUDA(cudaStreamWaitEvent(sb, ev0, 0));
    dsg_graph va = *g, vb = *g;
    va.owns = vb.owns = false;
    va.stream = sa;
    vb.stream = sb;
    va.force_block = vb.force_block = 1024;
    // the peels' share of the SMs: DSG_SOLVE_PEEL_PERMILLE if set, else from
    // the autotuned times (each side's share of the summed time, within
    // [1/4, 3/4]), else as if the core numbers took as long as eight peels
    // (R-MAT 2^20, three peels, from host memory: 6.72 ms at 0.25, 6.82 at 0.3,
    // 7.49 at half; Chung-Lu 3 10^6 9.48 / 8.98 / 9.63; Erdos-Renyi 5 10^5
    // 1.80 / 1.78 / 1.89)
    double peel_frac = std::min(0.5, std::max(0.15, count / (count + 8.0)));
    if (tuned && count * peel_ms + core_ms > 0)
        peel_frac = std::min(0.75, std::max(0.25, count * peel_ms / (count * peel_ms + core_ms)));
    if (const char* e = getenv("DSG_SOLVE_PEEL_PERMILLE")) {
        const long pm = strtol(e, nullptr, 10);
        if (pm > 0 && pm < 1000) peel_frac = pm / 1000.0;
    }
    va.max_blocks = std::max<uint32_t>(1, (uint32_t)(sms * peel_frac + 0.5));
    if (va.max_blocks >= sms) va.max_blocks = sms > 1 ? sms - 1 : 1;
    vb.max_blocks = sms - va.max_blocks > 0 ? sms - va.max_blocks : 1;
    dsg_status st_core = DSG_OK;
    std::string err_core;
    std::thread th([&] {
        cudaSetDevice(g->device);
        st_core = run_kcore(&vb, out_core, nullptr, 0);
        if (st_core != DSG_OK) err_core = dsg_last_error();
    });
    dsg_status st = peels(&va);
    th.join();
    cudaEventRecord(eva, sa);
    cudaEventRecord(evb, sb);
    cudaStreamWaitEvent(g->stream, eva, 0);
    cudaStreamWaitEvent(g->stream, evb, 0);
    if (st != DSG_OK) return st;
    if (st_core != DSG_OK) {
        set_error("%s", err_core.c_str());
        return st_core;
    }
    return DSG_OK;
}

dsg_status dsg_bahmani_trace(const dsg_graph* g, uint32_t eps_num, uint32_t eps_den, dsg_trace* t) {
    clear_error();
    DSG_CHECK_ARG(g, "graph is NULL");
    DSG_CHECK_ARG(t, "trace is NULL");
    DSG_CHECK_ARG(eps_den != 0, "eps_den must be positive");
    DSG_TRY_CUDA(cudaSetDevice(g->device));
    PeelCtl c;
    dsg_status st = run_peel(g, eps_num, eps_den, t->hist_S, t->hist_E, t->hist_cap, t->peel_round, t->out_set, &c);
    if (st != DSG_OK) return st;
    t->rounds = c.rounds;
    t->best_round = c.best_round;
    t->best_E = g->n ? c.best_E : 0;
    t->best_V = g->n ? c.best_V : 0;
    t->edges_scanned = g->n ? c.scanned : 0;
    t->decrements = g->n ? c.dec : 0;
    t->tested = g->n ? c.tested : 0;
    t->lazy_rounds = g->n ? c.lazy_rounds : 0;
    if (t->hist_cap < c.rounds + 1 && (t->hist_S || t->hist_E)) {
        set_error("bahmani_trace: history needs %llu slots, got %llu", (unsigned long long)(c.rounds + 1),
                  (unsigned long long)t->hist_cap);
        return DSG_EOVERFLOW;
    }
    return DSG_OK;
}

// Phase timestamps of one peel (debug/analysis): ts[i] = %globaltimer after
// the i-th grid barrier (ts[0] = kernel start).  *count = stamps taken.
dsg_status dsg_debug_peel_trace(const dsg_graph* g, uint32_t eps_num, uint32_t eps_den, uint64_t* ts, uint64_t cap,
                                uint64_t* count) {
    clear_error();
    DSG_CHECK_ARG(g && ts && cap, "graph/ts/cap");
    DSG_CHECK_ARG(eps_den != 0, "eps_den must be positive");
    DSG_TRY_CUDA(cudaSetDevice(g->device));
    Scratch sc(g->stream);
    uint64_t* dts;
    DSG_TRY_CUDA(sc.get(&dts, cap));
    PeelCtl c;
    dsg_status st = run_peel(g, eps_num, eps_den, nullptr, nullptr, 0, nullptr, nullptr, &c, dts, cap);
    if (st != DSG_OK) return st;
    uint64_t k = c.stamps < cap ? c.stamps : cap;
    DSG_TRY_CUDA(copy_any(ts, dts, k * 8, g->stream));
    DSG_TRY_CUDA(cudaStreamSynchronize(g->stream));
    if (count) *count = c.stamps;
    return DSG_OK;
}

uint32_t dsg_debug_meet_count(uint64_t word, uint32_t high, uint32_t arrivals, uint32_t blocks) {
    return meet_count(word, high, arrivals, blocks);
}

dsg_status dsg_debug_peel_wrap(const dsg_graph* g, uint32_t eps_num, uint32_t eps_den, uint32_t wrap_in,
                               uint32_t* peel_round, uint8_t* out_set, uint64_t out4[4]) {
    clear_error();
    DSG_CHECK_ARG(g && out4, "graph / out4 is NULL");
    DSG_CHECK_ARG(eps_den != 0, "eps_den must be positive");
    DSG_CHECK_ARG(wrap_in >= 1 && wrap_in <= 1u << 20, "wrap_in must be in [1, 2^20]");
    DSG_TRY_CUDA(cudaSetDevice(g->device));
    PeelCtl c;
    dsg_status st = run_peel(g, eps_num, eps_den, nullptr, nullptr, 0, peel_round, out_set, &c, nullptr, 0, wrap_in);
    if (st != DSG_OK) return st;
    out4[0] = g->n ? c.best_E : 0;
    out4[1] = g->n ? c.best_V : 0;
    out4[2] = c.rounds;
    out4[3] = c.best_round;
    return DSG_OK;
}

}  // extern "C"

// ===================================================== no-allocation variant
//
// Some callers cannot allocate device memory at the moment they want a peel:
// code running under an allocator they do not own (a host application whose
// memory pool is reserved up front, a framework that forbids allocation on
// its hot path), or code that must not risk cudaMalloc's implicit device
// synchronisation.  dsg_bahmani_noalloc serves them: it runs the same
// persistent peel kernel as dsg_bahmani, but every scratch array lives in one
// fixed buffer that belongs to this library file -- a static device array of
// kNoAllocScratchBytes, reserved on each GPU that loads this code and held
// until the process exits.  The caller passes the graph and the outputs.
#include <mutex>

namespace dsg {

constexpr size_t kNoAllocScratchBytes = 64ull << 20;  // 64 MiB per device

static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocScratchBytes];

// Device address of g_noalloc_scratch.  Host code may not use the symbol
// itself as an address (on the host it names a shadow variable), so the
// address is looked up with cudaGetSymbolAddress, with the device current,
// the first time a call runs in a CUDA context.  The cache is keyed on the
// context's id, not on the device ordinal: after a context is destroyed and
// made again (cudaDeviceReset, a released primary context) the module is
// loaded again and the array may sit elsewhere, so the new context looks it
// up afresh.
struct NoAllocSlot {
    unsigned long long ctx_id = 0;  // 0: empty
    unsigned char* addr = nullptr;
};
static std::mutex g_noalloc_mu;
static NoAllocSlot g_noalloc_slots[64];

static dsg_status noalloc_scratch(unsigned char** out) {
    int dev = 0;
    DSG_TRY_CUDA(cudaGetDevice(&dev));
    DSG_CHECK_ARG(dev >= 0 && dev < 64, "device ordinal above 63");
    const unsigned long long id = current_ctx_id();
    std::lock_guard<std::mutex> lk(g_noalloc_mu);
    NoAllocSlot& slot = g_noalloc_slots[dev];
    if (id == 0 || slot.ctx_id != id) {
        void* p = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e != cudaSuccess || !p) {
            set_error("bahmani_noalloc: cudaGetSymbolAddress of the static scratch failed: %s",
                      cudaGetErrorString(e));
            return DSG_ECUDA;
        }
        slot.addr = static_cast<unsigned char*>(p);
        slot.ctx_id = id;
    }
    *out = slot.addr;
    return DSG_OK;
}

static size_t align256(size_t b) { return (b + 255) & ~size_t(255); }

template <int TB>
static cudaError_t launch_peel_noalloc(PeelArgs& a, uint32_t blocks_per_sm, cudaStream_t s) {
    uint32_t grid = 1;
    cudaError_t e = coop_grid(peel_kernel<TB>, TB, 0, a.n, blocks_per_sm, &grid);
    if (e != cudaSuccess) return e;
    void* params[] = {&a};
    LaunchScope ls("peel_rounds", s);
    return cudaLaunchCooperativeKernel((const void*)peel_kernel<TB>, dim3(grid), dim3(TB), params, 0, s);
}

}  // namespace dsg

extern "C" dsg_status dsg_bahmani_noalloc(uint32_t n, const uint64_t* off, const uint32_t* adj, uint32_t eps_num,
                                          uint32_t eps_den, uint8_t* out_set, uint64_t* out_E, uint64_t* out_V,
                                          void* stream) {
    clear_error();
    DSG_CHECK_ARG(eps_den != 0, "eps_den must be positive");
    DSG_CHECK_ARG(n < 0x80000000u, "n must be below 2^31");
    DSG_CHECK_ARG(off && is_device_ptr(off), "off must be a device pointer");
    DSG_CHECK_ARG(!out_set || is_device_ptr(out_set), "out_set must be a device pointer (or NULL)");
    cudaStream_t s = (cudaStream_t)stream;
    uint64_t total = 0;
    DSG_TRY_CUDA(cudaMemcpyAsync(&total, off + n, sizeof(uint64_t), cudaMemcpyDeviceToHost, s));
    DSG_TRY_CUDA(cudaStreamSynchronize(s));
    DSG_CHECK_ARG(total % 2 == 0, "off[n] must be even for a symmetric CSR");
    DSG_CHECK_ARG(total == 0 || (adj && is_device_ptr(adj)), "adj must be a device pointer");
    if (n == 0) {
        if (out_E) *out_E = 0;
        if (out_V) *out_V = 0;
        return DSG_OK;
    }
    const Tuning tu = current_tuning();
    const uint64_t m = total / 2;
    const uint64_t cap = dsg_round_bound(n, eps_num, eps_den) + 1;
    const uint64_t chunk_cap = (uint64_t)n + (2 * m) / piece_len(tu) + 1;
    const size_t b_list = align256((size_t)n * 4);
    const size_t b_chunk = align256((size_t)chunk_cap * 8);
    const size_t b_hist = align256((size_t)cap * 8);
    constexpr size_t b_ctl = 1280;  // the control block's share (a part of the documented limit)
    static_assert(sizeof(PeelCtl) <= b_ctl, "the control block's share");
    const size_t b_map = align256(((size_t)n + 15) / 16 * 4);
    const size_t need = 4 * b_list + b_chunk + b_map + 2 * b_hist + b_ctl;
    if (need > kNoAllocScratchBytes) {
        set_error("bahmani_noalloc: this graph needs %zu bytes of scratch, above the fixed %zu-byte buffer "
                  "(use dsg_bahmani)", need, (size_t)kNoAllocScratchBytes);
        return DSG_EINVAL;
    }
    unsigned char* base = nullptr;
    dsg_status st = noalloc_scratch(&base);
    if (st != DSG_OK) return st;
    PeelArgs a;
    a.n = n;
    a.m = m;
    a.p = eps_num;
    a.q = eps_den;
    a.off = off;
    a.adj = adj;
    size_t o = 0;
    a.st = reinterpret_cast<uint32_t*>(base + o); o += b_list;
    a.listA = reinterpret_cast<uint32_t*>(base + o); o += b_list;
    a.listB = reinterpret_cast<uint32_t*>(base + o); o += b_list;
    a.items = reinterpret_cast<uint64_t*>(base + o); o += b_chunk;
    a.map = reinterpret_cast<uint32_t*>(base + o); o += b_map;
    a.candA = nullptr;  // no lazy rounds: every round tests the whole alive list
    a.candB = nullptr;
    a.hist_S = reinterpret_cast<uint64_t*>(base + o); o += b_hist;
    a.hist_E = reinterpret_cast<uint64_t*>(base + o); o += b_hist;
    a.ctl = reinterpret_cast<PeelCtl*>(base + o);
    a.hist_cap = cap;
    a.limit_ns = wait_limit_ns();
    a.chunk_len = piece_len(tu);
    a.hot_deg = tu.hot_deg;
    a.trace = nullptr;
    a.trace_cap = 0;
    a.r0 = a.S0 = a.E0 = a.best_round0 = a.best_E0 = a.best_V0 = a.max_rounds = a.arrivals0 = 0;
    // The buffer keeps whatever the previous call left; only the control
    // block must start at zero (every other array is written before it is read).
    DSG_TRY_CUDA(cudaMemsetAsync(a.ctl, 0, sizeof(PeelCtl), s));
    cudaError_t e;
    switch (tu.block) {
        case 256: e = launch_peel_noalloc<256>(a, tu.blocks_per_sm, s); break;
        case 1024: e = launch_peel_noalloc<1024>(a, tu.blocks_per_sm, s); break;
        default: e = launch_peel_noalloc<512>(a, tu.blocks_per_sm, s); break;
    }
    DSG_TRY_CUDA(e);
    if (out_set) {
        uint64_t want = ((uint64_t)n + 255) / 256, cap_b = (uint64_t)dev_info().sms * 8;
        uint32_t blocks = (uint32_t)(want < cap_b ? want : cap_b);
        {
            LaunchScope ls("peel_finish", s);
            peel_finish_kernel<<<blocks, 256, 0, s>>>(n, a.st, a.ctl, nullptr, out_set);
        }
        DSG_TRY_CUDA(cudaGetLastError());
    }
    PeelCtl c;
    DSG_TRY_CUDA(cudaMemcpyAsync(&c, a.ctl, sizeof(PeelCtl), cudaMemcpyDeviceToHost, s));
    DSG_TRY_CUDA(cudaStreamSynchronize(s));
    st = status_from_err(c.err, "bahmani_noalloc");
    if (st != DSG_OK) return st;
    if (out_E) *out_E = c.best_E;
    if (out_V) *out_V = c.best_V;
    return DSG_OK;
}

// ========================================================= snapshot / resume
//
// Algorithm 1's state between two rounds is small: each vertex's state word
// (its degree inside S_r, or the round it failed in), the round r, |S_r|,
// |E(S_r)|, the best round so far with its (E, V), and the history of
// (|S_t|, |E(S_t)|).  A paused peel keeps that state on the device between
// launches; a snapshot writes it to host memory, and resuming rebuilds it on
// a handle of the same graph, so a long peel (eps = 0 on a graph that peels
// slowly) can be checkpointed, moved or continued later with the same result.
struct dsg_peel_state {
    const dsg_graph* g = nullptr;
    uint32_t p = 0, q = 1;
    uint64_t r = 0, S = 0, E = 0, best_round = 0, best_E = 0, best_V = 0, cap = 0;
    bool done = false;
    dsg::Tuning tu;
    uint32_t *st = nullptr, *listA = nullptr, *listB = nullptr, *map = nullptr, *candA = nullptr, *candB = nullptr;
    uint64_t *items = nullptr, *hist_S = nullptr, *hist_E = nullptr;
    dsg::PeelCtl* ctl = nullptr;
};

namespace dsg {

static constexpr uint64_t kSnapMagic = 0x314c454550475344ull;  // "DSGPEEL1"
static constexpr uint64_t kSnapHeaderWords = 16;

static void peel_state_release(dsg_peel_state* ps) {
    if (!ps) return;
    cudaStream_t s = ps->g ? ps->g->stream : nullptr;
    void* bufs[] = {ps->st,    ps->listA, ps->listB,  ps->items,  ps->map,
                    ps->candA, ps->candB, ps->hist_S, ps->hist_E, ps->ctl};
    for (void* b : bufs)
        if (b) dev_free(b, s);
    if (s) cudaStreamSynchronize(s);
    delete ps;
}

// A new state on g (device arrays allocated, scalars at round 0).
static dsg_status peel_state_new(const dsg_graph* g, uint32_t p, uint32_t q, dsg_peel_state** out) {
    dsg_peel_state* ps = new dsg_peel_state();
    ps->g = g;
    ps->p = p;
    ps->q = q;
    ps->tu = tuning_for(g, 0);
    if (g->force_block) ps->tu.block = g->force_block;
    const uint32_t n = g->n;
    ps->cap = n ? dsg_round_bound(n, p, q) + 1 : 1;
    const uint64_t item_cap = (uint64_t)n + (2 * g->m) / piece_len(ps->tu) + 1;
    ps->S = n;
    ps->E = g->m;
    ps->best_E = g->m;
    ps->best_V = n;
    ps->done = n == 0;
    cudaStream_t s = g->stream;
    const size_t nb = ((size_t)(n ? n : 1) * 4 + 255) & ~size_t(255);
    cudaError_t e = dev_alloc((void**)&ps->st, nb, s);
    if (e == cudaSuccess) e = dev_alloc((void**)&ps->listA, nb, s);
    if (e == cudaSuccess) e = dev_alloc((void**)&ps->listB, nb, s);
    if (e == cudaSuccess) e = dev_alloc((void**)&ps->candA, nb, s);
    if (e == cudaSuccess) e = dev_alloc((void**)&ps->candB, nb, s);
    if (e == cudaSuccess) e = dev_alloc((void**)&ps->items, item_cap * 8, s);
    if (e == cudaSuccess) e = dev_alloc((void**)&ps->map, (((size_t)(n ? n : 1) + 15) / 16 * 4 + 255) & ~size_t(255), s);
    if (e == cudaSuccess) e = dev_alloc((void**)&ps->hist_S, ps->cap * 8, s);
    if (e == cudaSuccess) e = dev_alloc((void**)&ps->hist_E, ps->cap * 8, s);
    if (e == cudaSuccess) e = dev_alloc((void**)&ps->ctl, sizeof(PeelCtl), s);
    if (e != cudaSuccess) {
        set_error("peel state: %s", cudaGetErrorString(e));
        peel_state_release(ps);
        return e == cudaErrorMemoryAllocation ? DSG_ENOMEM : DSG_ECUDA;
    }
    *out = ps;
    return DSG_OK;
}

// Run up to max_rounds rounds (0: to the end) from where ps stands.
static dsg_status peel_state_run(dsg_peel_state* ps, uint64_t max_rounds) {
    if (ps->done) return DSG_OK;
    const dsg_graph* g = ps->g;
    cudaStream_t s = g->stream;
    PeelArgs a;
    a.n = g->n;
    a.m = g->m;
    a.p = ps->p;
    a.q = ps->q;
    a.off = g->off;
    a.adj = g->adj;
    a.st = ps->st;
    a.listA = ps->listA;
    a.listB = ps->listB;
    a.items = ps->items;
    a.map = ps->map;
    const bool lazy_on = current_tuning().peel_lazy != 0;
    a.candA = lazy_on ? ps->candA : nullptr;
    a.candB = lazy_on ? ps->candB : nullptr;
    a.hist_S = ps->hist_S;
    a.hist_E = ps->hist_E;
    a.hist_cap = ps->cap;
    a.ctl = ps->ctl;
    a.limit_ns = wait_limit_ns();
    a.chunk_len = piece_len(ps->tu);
    a.hot_deg = ps->tu.hot_deg;
    a.trace = nullptr;
    a.trace_cap = 0;
    a.r0 = ps->r;
    a.S0 = ps->S;
    a.E0 = ps->E;
    a.best_round0 = ps->best_round;
    a.best_E0 = ps->best_E;
    a.best_V0 = ps->best_V;
    a.max_rounds = max_rounds;
    a.arrivals0 = 0;
    PeelCtl init;
    memset(&init, 0, sizeof(init));
    init.failed = (uint64_t)g->n - ps->S;  // the counters the kernel derives S and E from
    init.xsum = 2 * (g->m - ps->E);
    DSG_TRY_CUDA(cudaMemcpyAsync(ps->ctl, &init, sizeof(PeelCtl), cudaMemcpyHostToDevice, s));
    cudaError_t e;
    switch (ps->tu.block) {
        case 256: e = launch_peel<256>(a, ps->tu.blocks_per_sm, s, g->max_blocks); break;
        case 1024: e = launch_peel<1024>(a, ps->tu.blocks_per_sm, s, g->max_blocks); break;
        default: e = launch_peel<512>(a, ps->tu.blocks_per_sm, s, g->max_blocks); break;
    }
    DSG_TRY_CUDA(e);
    PeelCtl c;
    DSG_TRY_CUDA(cudaMemcpyAsync(&c, ps->ctl, sizeof(PeelCtl), cudaMemcpyDeviceToHost, s));
    DSG_TRY_CUDA(cudaStreamSynchronize(s));
    dsg_status st = status_from_err(c.err, "peel");
    if (st != DSG_OK) return st;
    ps->r = c.rounds;
    ps->S = c.cur_S;
    ps->E = c.cur_E;
    ps->best_round = c.best_round;
    ps->best_E = c.best_E;
    ps->best_V = c.best_V;
    ps->done = ps->S == 0;
    return DSG_OK;
}

static uint64_t snapshot_bytes(const dsg_peel_state* ps) {
    return (kSnapHeaderWords + 2 * (ps->r + 1)) * 8 + (uint64_t)ps->g->n * 4;
}

}  // namespace dsg

extern "C" {

dsg_status dsg_peel_begin(const dsg_graph* g, uint32_t eps_num, uint32_t eps_den, dsg_peel_state** out) {
    clear_error();
    DSG_CHECK_ARG(g && out, "graph / out is NULL");
    DSG_CHECK_ARG(eps_den != 0, "eps_den must be positive");
    DSG_TRY_CUDA(cudaSetDevice(g->device));
    dsg_peel_state* ps = nullptr;
    dsg_status st = peel_state_new(g, eps_num, eps_den, &ps);
    if (st != DSG_OK) return st;
    const uint64_t h[2] = {g->n, g->m};
    cudaError_t e = cudaMemcpyAsync(ps->hist_S, &h[0], 8, cudaMemcpyHostToDevice, g->stream);
    if (e == cudaSuccess) e = cudaMemcpyAsync(ps->hist_E, &h[1], 8, cudaMemcpyHostToDevice, g->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(g->stream);
    if (e != cudaSuccess) {
        set_error("peel_begin: %s", cudaGetErrorString(e));
        peel_state_release(ps);
        return DSG_ECUDA;
    }
    *out = ps;
    return DSG_OK;
}

dsg_status dsg_peel_advance(dsg_peel_state* ps, uint32_t max_rounds, uint64_t* rounds, uint32_t* done) {
    clear_error();
    DSG_CHECK_ARG(ps, "state is NULL");
    DSG_TRY_CUDA(cudaSetDevice(ps->g->device));
    dsg_status st = peel_state_run(ps, max_rounds);
    if (st != DSG_OK) return st;
    if (rounds) *rounds = ps->r;
    if (done) *done = ps->done ? 1u : 0u;
    return DSG_OK;
}

dsg_status dsg_peel_snapshot_size(const dsg_peel_state* ps, uint64_t* bytes) {
    clear_error();
    DSG_CHECK_ARG(ps && bytes, "state / bytes is NULL");
    *bytes = snapshot_bytes(ps);
    return DSG_OK;
}

dsg_status dsg_peel_snapshot(const dsg_peel_state* ps, void* buf, uint64_t bytes) {
    clear_error();
    DSG_CHECK_ARG(ps && buf, "state / buffer is NULL");
    DSG_CHECK_ARG(bytes >= snapshot_bytes(ps), "buffer smaller than dsg_peel_snapshot_size");
    DSG_TRY_CUDA(cudaSetDevice(ps->g->device));
    uint64_t* w = static_cast<uint64_t*>(buf);
    const uint64_t hl = ps->r + 1;
    const uint64_t h[kSnapHeaderWords] = {kSnapMagic, 1, ps->g->n, ps->g->m, ps->p, ps->q, ps->r, ps->S, ps->E,
                                          ps->best_round, ps->best_E, ps->best_V, hl, 0, 0, 0};
    memcpy(w, h, sizeof(h));
    cudaStream_t s = ps->g->stream;
    DSG_TRY_CUDA(copy_any(w + kSnapHeaderWords, ps->hist_S, hl * 8, s));
    DSG_TRY_CUDA(copy_any(w + kSnapHeaderWords + hl, ps->hist_E, hl * 8, s));
    uint32_t* words = reinterpret_cast<uint32_t*>(w + kSnapHeaderWords + 2 * hl);
    if (ps->r > 0) {
        if (ps->g->n) DSG_TRY_CUDA(copy_any(words, ps->st, (size_t)ps->g->n * 4, s));
    } else {
        memset(words, 0, (size_t)ps->g->n * 4);  // before the first round the state words are not used
    }
    DSG_TRY_CUDA(cudaStreamSynchronize(s));
    return DSG_OK;
}

dsg_status dsg_peel_resume(const dsg_graph* g, const void* buf, uint64_t bytes, dsg_peel_state** out) {
    clear_error();
    DSG_CHECK_ARG(g && buf && out, "graph / buffer / out is NULL");
    DSG_CHECK_ARG(bytes >= kSnapHeaderWords * 8, "buffer shorter than a snapshot header");
    const uint64_t* w = static_cast<const uint64_t*>(buf);
    DSG_CHECK_ARG(w[0] == kSnapMagic && w[1] == 1, "not a peel snapshot (magic / version)");
    DSG_CHECK_ARG(w[2] == g->n && w[3] == g->m, "the snapshot was taken on a graph of another size");
    DSG_CHECK_ARG(w[5] != 0 && w[4] <= 0xffffffffull && w[5] <= 0xffffffffull, "bad eps in the snapshot");
    const uint64_t r = w[6], hl = w[12];
    DSG_CHECK_ARG(hl == r + 1, "bad history length in the snapshot");
    DSG_CHECK_ARG(bytes >= (kSnapHeaderWords + 2 * hl) * 8 + (uint64_t)g->n * 4, "snapshot truncated");
    DSG_CHECK_ARG(w[7] <= g->n && w[8] <= g->m && w[9] <= r && w[11] <= g->n, "inconsistent snapshot scalars");
    DSG_TRY_CUDA(cudaSetDevice(g->device));
    dsg_peel_state* ps = nullptr;
    dsg_status st = peel_state_new(g, (uint32_t)w[4], (uint32_t)w[5], &ps);
    if (st != DSG_OK) return st;
    if (hl > ps->cap) {
        set_error("peel_resume: the snapshot has %llu rounds, more than the bound %llu for its eps",
                  (unsigned long long)r, (unsigned long long)(ps->cap - 1));
        peel_state_release(ps);
        return DSG_EINVAL;
    }
    ps->r = r;
    ps->S = w[7];
    ps->E = w[8];
    ps->best_round = w[9];
    ps->best_E = w[10];
    ps->best_V = w[11];
    ps->done = ps->S == 0;
    cudaStream_t s = g->stream;
    cudaError_t e = copy_any(ps->hist_S, w + kSnapHeaderWords, hl * 8, s);
    if (e == cudaSuccess) e = copy_any(ps->hist_E, w + kSnapHeaderWords + hl, hl * 8, s);
    if (e == cudaSuccess && r > 0 && g->n)
        e = copy_any(ps->st, reinterpret_cast<const uint32_t*>(w + kSnapHeaderWords + 2 * hl), (size_t)g->n * 4, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) {
        set_error("peel_resume: %s", cudaGetErrorString(e));
        peel_state_release(ps);
        return DSG_ECUDA;
    }
    *out = ps;
    return DSG_OK;
}

dsg_status dsg_peel_finish(dsg_peel_state* ps, uint8_t* out_set, uint64_t* out_E, uint64_t* out_V,
                           uint64_t* out_rounds, uint64_t* hist_S, uint64_t* hist_E, uint64_t hist_cap) {
    clear_error();
    DSG_CHECK_ARG(ps, "state is NULL");
    DSG_TRY_CUDA(cudaSetDevice(ps->g->device));
    dsg_status st = peel_state_run(ps, 0);
    if (st != DSG_OK) return st;
    const dsg_graph* g = ps->g;
    cudaStream_t s = g->stream;
    const uint32_t n = g->n;
    if (out_set && n) {
        Scratch sc(s);
        uint8_t* set_dev = out_set;
        const bool direct = is_device_ptr(out_set);
        if (!direct) DSG_TRY_CUDA(sc.get(&set_dev, n));
        PeelCtl c;
        memset(&c, 0, sizeof(c));
        c.best_round = ps->best_round;
        DSG_TRY_CUDA(cudaMemcpyAsync(ps->ctl, &c, sizeof(PeelCtl), cudaMemcpyHostToDevice, s));
        uint64_t want = ((uint64_t)n + 255) / 256, cap_b = (uint64_t)dev_info().sms * 8;
        {
            LaunchScope ls("peel_finish", s);
            peel_finish_kernel<<<(uint32_t)(want < cap_b ? want : cap_b), 256, 0, s>>>(n, ps->st, ps->ctl, nullptr,
                                                                                       set_dev);
        }
        DSG_TRY_CUDA(cudaGetLastError());
        if (!direct) DSG_TRY_CUDA(copy_any(out_set, set_dev, n, s));
        DSG_TRY_CUDA(cudaStreamSynchronize(s));
    }
    const uint64_t R = ps->r;
    if (hist_S || hist_E) {
        const uint64_t k = R + 1 < hist_cap ? R + 1 : hist_cap;
        if (hist_S && k) DSG_TRY_CUDA(copy_any(hist_S, ps->hist_S, k * 8, s));
        if (hist_E && k) DSG_TRY_CUDA(copy_any(hist_E, ps->hist_E, k * 8, s));
        DSG_TRY_CUDA(cudaStreamSynchronize(s));
    }
    if (out_E) *out_E = n ? ps->best_E : 0;
    if (out_V) *out_V = n ? ps->best_V : 0;
    if (out_rounds) *out_rounds = R;
    if ((hist_S || hist_E) && hist_cap < R + 1) {
        set_error("peel_finish: history needs %llu slots, got %llu", (unsigned long long)(R + 1),
                  (unsigned long long)hist_cap);
        return DSG_EOVERFLOW;
    }
    return DSG_OK;
}

void dsg_peel_free(dsg_peel_state* ps) {
    if (ps && ps->g) cudaSetDevice(ps->g->device);
    peel_state_release(ps);
}

}  // extern "C"
