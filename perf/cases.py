"""Workloads of the densest-subgraph library, one dict of plain values each.

A case names a task (which public calls a program makes), a graph family and
its sizes.  Graphs are drawn on the GPU from the seed: uniform pairs (er),
R-MAT (rmat), power-law Chung-Lu (cl), and nested shells around a clique
(onion, the long tail of thin rounds).

  peel    Algorithm 1 on a resident graph: bahmani(), or bahmani_trace()
  kcore   core numbers of a resident graph
  step    raw pairs on the GPU -> from_edges + bahmani + kcore
  solve   raw pairs in pinned host memory -> from_edges + solve (peels at
          three eps and the core numbers), results to pinned host memory
  cbds    densest core and its augmentation from core numbers in hand
  batch   BatchSolver over many packed graphs, with or without core numbers
  serve   a burst of requests through a running Server
"""
import math

import numpy as np
import torch

import paper_2103_00154_gb300 as dsg

DEV = "cuda"


# -------------------------------------------------------------------- cases
def listed():
    return [
        # the smallest call: one peel of a 10^4-vertex graph kept on the GPU,
        # as an interactive query makes it (launches and waits count)
        dict(name="peel_small", task="peel", trace=False, family="er", n=10_000, m=50_000, block=100, pblock=0.5,
             p=1, q=10),
        # the same graph from its raw pairs: a whole small analysis per call
        dict(name="step_small", task="step", family="er", n=10_000, m=50_000, block=100, pblock=0.5, p=1, q=10),
        # a peel with its full history on a mid-size social graph of ragged size
        dict(name="peel_social", task="peel", trace=True, family="cl", n=3_000_017, m=40_000_003, gamma=2.1,
             mean=26.7, wmax=40_000.0, p=1, q=100),
        # a graph whose peel is a long tail of thin rounds (about one per shell)
        dict(name="peel_tail", task="peel", trace=False, family="onion", n=262_144, d=64, core=160, p=1, q=1000),
        # core numbers alone, an ordinary web-graph size
        dict(name="kcore_web", task="kcore", family="cl", n=700_001, m=5_600_000, gamma=2.3, mean=16.0,
             wmax=30_000.0),
        # core numbers of a skewed R-MAT graph (hubs at low ids, many empty rows)
        dict(name="kcore_rmat", task="kcore", family="rmat", n=1 << 18, m=1 << 22),
        # a one-off analysis from host memory: pairs in, sets and core numbers out
        dict(name="solve_rmat20", task="solve", family="rmat", n=1 << 20, m=1 << 24),
        # densest core with augmentation for a graph whose core numbers are known
        dict(name="cbds_web", task="cbds", family="cl", n=2_000_003, m=30_000_000, gamma=2.1, mean=30.0,
             wmax=30_000.0),
        # many small communities at once
        dict(name="batch_many", task="batch", graphs=1500, n_lo=1_000, n_hi=100_000, cores=False, p=1, q=10),
        # uneven batch up to a million vertices, core numbers too
        dict(name="batch_cores", task="batch", graphs=96, n_lo=1_000, n_hi=1_000_000, cores=True, p=1, q=10),
        # a burst of mixed requests at a running server
        dict(name="serve_burst", task="serve", graphs=64, n_lo=1_000, n_hi=300_000),
        # the largest single graph: 2^24 vertices, 2^28 raw pairs
        dict(name="step_largest", task="step", family="cl", n=1 << 24, m=1 << 28, gamma=2.1, mean=32.0, wmax=1e5,
             p=1, q=10),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    task = rng.choice(["peel", "peel", "kcore", "kcore", "step", "step", "solve", "cbds", "batch", "serve"])
    p, q = rng.choice([(1, 1000), (1, 100), (1, 10), (1, 2), (1, 1)])
    if task in ("batch", "serve"):
        lo = _log(rng, 500, 5_000)
        if task == "serve":
            return dict(task=task, graphs=rng.randrange(8, 97), n_lo=lo, n_hi=_log(rng, 20_000, 300_000))
        cores = rng.random() < 0.5
        hi = _log(rng, 20_000, 200_000)
        return dict(task=task, graphs=_log(rng, 16, 600 if cores else 1200), n_lo=lo, n_hi=hi, cores=cores, p=p, q=q)
    c = dict(task=task, family=rng.choice(["er", "rmat", "cl", "cl"]))
    n = _log(rng, 3_000, 4_000_000) | rng.randrange(2)
    mean = rng.uniform(6.0, 40.0)
    if task == "peel":
        c.update(trace=rng.random() < 0.5)
        if rng.random() < 0.2:
            c.update(family="onion", n=_log(rng, 20_000, 600_000), d=rng.randrange(16, 80), core=rng.randrange(90, 200),
                     p=1, q=1000)
            return c
    if task in ("peel", "step"):
        c.update(p=p, q=q)
    if c["family"] == "rmat":
        n = 1 << min(21, max(12, n.bit_length()))
    c.update(n=n, m=int(n * mean / 2))
    if c["family"] == "cl":
        c.update(gamma=round(rng.uniform(2.05, 2.6), 2), mean=mean, wmax=float(int(rng.uniform(0.3, 20.0) * math.sqrt(mean * n))))
    if c["family"] == "er":
        c.update(block=max(2, math.isqrt(n) * rng.randrange(1, 4) // 2), pblock=round(rng.uniform(0.2, 0.6), 2))
    return c


# ------------------------------------------------------------------- graphs
def _gen(seed, k=0):
    return torch.Generator(device=DEV).manual_seed((seed * 1_000_003 + k * 7_919 + 12_345) % (1 << 62))


def _er(n, m, gen):
    return torch.randint(0, n, (2, m), generator=gen, device=DEV, dtype=torch.int32)


def _block(n, k, prob, gen):
    """Each pair of k spread-out vertices with probability prob."""
    at = torch.arange(k, device=DEV) * max(1, n // k) + int(torch.randint(0, max(1, n // k), (1,), generator=gen, device=DEV))
    i, j = torch.triu_indices(k, k, 1, device=DEV)
    keep = torch.rand(i.numel(), generator=gen, device=DEV) < prob
    return torch.stack([at[i[keep]], at[j[keep]]]).to(torch.int32)


def _rmat(n, m, gen, a=0.57, b=0.19, c=0.19):
    x = torch.zeros(2, m, dtype=torch.int32, device=DEV)
    for _ in range(n.bit_length() - 1):
        u = torch.rand(m, generator=gen, device=DEV)
        x[0] = x[0] * 2 + (u >= a + b)
        x[1] = x[1] * 2 + ((u >= a) & (u < a + b) | (u >= a + b + c))
    return x


def _chung_lu(n, m, gamma, mean, wmax, gen):
    """Endpoints with probability ~ (i + i0)^(-1/(gamma-1)), i0 such that the
    largest weight is wmax / mean times the average one."""
    e = 1.0 - 1.0 / (gamma - 1.0)
    lo, hi = 1e-3, 10.0 * n
    for _ in range(100):
        i0 = math.sqrt(lo * hi)
        avg = ((i0 + n) ** e - i0 ** e) / (e * n)
        lo, hi = (i0, hi) if i0 ** (e - 1.0) / avg > wmax / mean else (lo, i0)
    w0, w1 = i0 ** e, (i0 + n) ** e
    x = torch.empty(2, m, dtype=torch.int32, device=DEV)
    flat = x.view(-1)
    for a in range(0, 2 * m, 1 << 26):
        u = torch.rand(min(1 << 26, 2 * m - a), generator=gen, device=DEV, dtype=torch.float64)
        flat[a:a + u.numel()] = (u.mul_(w1 - w0).add_(w0).pow_(1.0 / e).sub_(i0)).clamp_(0, n - 1).to(torch.int32)
    return x


def _onion(n, d, core, gen):
    """Nested shells around a clique, each vertex with d edges into the shell
    inside; vertex ids shuffled."""
    sizes = [core]
    while sum(sizes) < n:
        sizes.append(-(-sizes[-1] * (d + 1) // d))
    total, base = sum(sizes), 0
    parts = [torch.triu_indices(core, core, 1, device=DEV)]
    for inner, size in zip(sizes, sizes[1:]):
        e = torch.arange(size * d, device=DEV)
        parts.append(torch.stack([base + inner + e // d, base + e % inner]))
        base += inner
    ids = torch.randperm(total, generator=gen, device=DEV)
    return total, ids[torch.cat(parts, 1)].to(torch.int32)


def _pairs(c, seed):
    """(n, pairs) of a single-graph case: int32 [2, m] on the GPU."""
    gen, n = _gen(seed), c["n"]
    if c["family"] == "onion":
        return _onion(n, c["d"], c["core"], gen)
    if c["family"] == "rmat":
        return n, _rmat(n, c["m"], gen)
    if c["family"] == "cl":
        return n, _chung_lu(n, c["m"], c["gamma"], c["mean"], c["wmax"], gen)
    return n, torch.cat([_er(n, c["m"], gen), _block(n, c["block"], c["pblock"], gen)], 1)


def _sizes(c):
    """The vertex counts of a batch or burst: spread over their logarithm, the same for every seed."""
    g = c["graphs"]
    f = [(i * 0.6180339887498949) % 1.0 for i in range(1, g)]
    return [c["n_hi"]] + [int(c["n_lo"] * (c["n_hi"] / c["n_lo"]) ** x) for x in f]


def _members(c, seed):
    """The pairs of each graph of a batch or burst: even ones uniform with mean
    degree 8, odd ones power-law with mean degree 16, each with a dense block."""
    for i, n in enumerate(_sizes(c)):
        gen = _gen(seed, i + 1)
        base = _er(n, 4 * n, gen) if i % 2 == 0 else _chung_lu(n, 8 * n, 2.3, 16.0, math.sqrt(16.0 * n), gen)
        yield n, torch.cat([base, _block(n, math.isqrt(n), 0.3, gen)], 1)


def _csr(n, pairs):
    """Sorted, symmetric, loop-free CSR (int64 offsets, int64 neighbours)."""
    u, v = pairs[0].long(), pairs[1].long()
    keep = u != v
    u, v = u[keep], v[keep]
    key = torch.unique(torch.cat([u * n + v, v * n + u]))
    off = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    off[1:] = torch.bincount(key // n, minlength=n).cumsum(0)
    return off, key % n


def _packed(c, seed):
    """(vtx_base, off, adj) with ids counted over the whole batch."""
    base, parts = [0], []
    for n, pairs in _members(c, seed):
        parts.append(pairs.long() + base[-1])
        base.append(base[-1] + n)
    off, adj = _csr(base[-1], torch.cat(parts, 1))
    return torch.tensor(base, device=DEV), off, adj


# -------------------------------------------------------------- prepare, run
def _eps_of(i):
    return (1, 100) if i % 2 == 0 else (1, 10)


SOLVE_EPS = [(1, 1000), (1, 10), (1, 1)]


def prepare(case, seed):
    task, st = case["task"], {"case": case, "stream": torch.cuda.current_stream()}
    if task == "batch":
        base, off, adj = _packed(case, seed)
        n = int(base[-1])
        owner = torch.repeat_interleave(base[:-1], base.diff())
        local = (adj - owner[torch.repeat_interleave(off.diff())]).to(torch.int32)
        g = case["graphs"]
        st["solver"] = dsg.BatchSolver(base, off, local, [(case["p"], case["q"])] * g,
                                       np.ones(g, np.uint8) if case["cores"] else None)
        st["mask"] = torch.empty(n, dtype=torch.uint8, device=DEV)
        st["core"] = torch.empty(n, dtype=torch.int32, device=DEV) if case["cores"] else None
        return st
    if task == "serve":
        st["graphs"] = [(n, x[0].cpu().pin_memory(), x[1].cpu().pin_memory()) for n, x in _members(case, seed)]
        n = sum(_sizes(case))
        st["mask"] = np.zeros(n, np.uint8)
        st["core"] = np.zeros(n, np.uint32)
        st["server"] = dsg.Server()
        return st
    n, pairs = _pairs(case, seed)
    st["n"] = n
    if task == "solve":
        st["pairs"] = (pairs[0].cpu().pin_memory(), pairs[1].cpu().pin_memory())
        st["masks"] = [torch.empty(n, dtype=torch.uint8).pin_memory() for _ in SOLVE_EPS]
        st["core"] = torch.empty(n, dtype=torch.int32).pin_memory()
        return st
    if task == "step":
        st["pairs"] = (pairs[0].contiguous(), pairs[1].contiguous())
    else:
        st["graph"] = dsg.Graph.from_edges(n, pairs[0].contiguous(), pairs[1].contiguous(), stream=st["stream"])
    st["mask"] = torch.empty(n, dtype=torch.uint8, device=DEV)
    st["core"] = torch.empty(n, dtype=torch.int32, device=DEV)
    if task == "cbds":
        st["graph"].kcore(out=st["core"])
    if task == "peel" and case["trace"]:
        st["peel_round"] = torch.empty(n, dtype=torch.int32, device=DEV)
    return st


def run(state):
    c = state["case"]
    task = c["task"]
    if task == "peel" and c["trace"]:
        t = state["graph"].bahmani_trace(c["p"], c["q"], peel_round=state["peel_round"], out_set=state["mask"])
        return {"mask": t.mask, "peel_round": t.peel_round, "E": t.E, "V": t.V, "rounds": t.rounds,
                "best_round": t.best_round, "hist_S": t.hist_S.view(np.int64), "hist_E": t.hist_E.view(np.int64)}
    if task == "peel":
        mask, E, V = state["graph"].bahmani(c["p"], c["q"], out_set=state["mask"])
        return {"mask": mask, "E": E, "V": V}
    if task == "kcore":
        return {"core": state["graph"].kcore(out=state["core"])}
    if task == "cbds":
        r = state["graph"].cbds(core=state["core"], out_set=state["mask"])
        return {"k_star": r.k_star, "E_core": r.E_core, "V_core": r.V_core, "E": r.E, "V": r.V,
                "n_legit": r.n_legit, "mask": r.mask}
    if task == "step":
        g = dsg.Graph.from_edges(state["n"], *state["pairs"], stream=state["stream"])
        mask, E, V = g.bahmani(c["p"], c["q"], out_set=state["mask"])
        core = g.kcore(out=state["core"])
        m = g.m
        g.close()
        return {"m": m, "mask": mask, "E": E, "V": V, "core": core}
    if task == "solve":
        g = dsg.Graph.from_edges(state["n"], *state["pairs"], stream=state["stream"])
        res, core = g.solve(SOLVE_EPS, out_sets=state["masks"], out_core=state["core"])
        m = g.m
        g.close()
        return {"m": m, "masks": [r[0] for r in res], "E": [r[1] for r in res], "V": [r[2] for r in res], "core": core}
    if task == "batch":
        E, V, R, BR = state["solver"].solve(out_set=state["mask"], core=state["core"], stream=state["stream"])
        out = {"E": E.view(np.int64), "V": V.view(np.int64), "rounds": R.view(np.int64),
               "best_round": BR.view(np.int64), "mask": state["mask"]}
        if c["cores"]:
            out["core"] = state["core"]
        return out
    srv, tickets, at = state["server"], [], 0
    for i, (n, src, dst) in enumerate(state["graphs"]):
        p, q = _eps_of(i)
        core = state["core"][at:at + n] if i % 4 < 2 else None
        tickets.append(srv.submit(n, src, dst, p, q, want_core=core is not None, out_set=state["mask"][at:at + n],
                                  core=core, borrow=True))
        at += n
    got = [srv.wait(t) for t in tickets]
    out = {k: np.array([r[k] for r in got], np.int64) for k in ("m", "E", "V", "rounds", "best_round")}
    return dict(out, mask=state["mask"], core=state["core"].view(np.int32))


# --------------------------------------------------------------------- work
def work(case):
    """Inputs read once, outputs written once (integers only: no flops)."""
    task = case["task"]
    if task in ("batch", "serve"):
        ns = _sizes(case)
        raw = sum((4 if i % 2 == 0 else 8) * n + 0.15 * n for i, n in enumerate(ns))
        if task == "serve":
            return {"bytes": 8.0 * raw + 3.0 * sum(ns), "flops": 0}
        return {"bytes": 8.0 * raw + (13.0 if case["cores"] else 9.0) * sum(ns), "flops": 0}
    n = case["n"]
    raw = case["d"] * n if case["family"] == "onion" else case["m"]
    if task == "step":
        return {"bytes": 8.0 * raw + 5.0 * n, "flops": 0}
    if task == "solve":
        return {"bytes": 8.0 * raw + 7.0 * n, "flops": 0}
    out = {"peel": 5 if case.get("trace") else 1, "kcore": 4, "cbds": 5}[task]
    return {"bytes": 8.0 * raw + (8.0 + out) * n, "flops": 0}


# -------------------------------------------------------------------- exact
def _row_entries(off, rows):
    """Positions of all entries of the given rows."""
    cnt = off[rows + 1] - off[rows]
    first = torch.repeat_interleave(off[rows] - (cnt.cumsum(0) - cnt), cnt)
    return first + torch.arange(first.numel(), device=DEV)


def _peel64(base, off, adj, p, q):
    """Algorithm 1 on every graph of a batch at once (p, q: one per graph)."""
    g, n = base.numel() - 1, off.numel() - 1
    size = base.diff()
    gid = torch.repeat_interleave(torch.arange(g, device=DEV), size)
    deg = off.diff()
    owner = torch.repeat_interleave(torch.arange(n, device=DEV), deg)
    S, E = size.clone(), (off[base[1:]] - off[base[:-1]]) // 2
    best = torch.stack([torch.zeros_like(S), E, S])
    R, gone = torch.zeros_like(S), torch.zeros(n, dtype=torch.int64, device=DEV)
    hist, r = [(S, E)], 0
    while bool((S > 0).any()):
        fail = (gone == 0) & (deg * (q * S)[gid] <= (2 * (p + q) * E)[gid])
        r += 1
        R[S > 0] = r
        gone[fail] = r
        alive = gone == 0
        keep = alive[owner] & alive[adj]
        deg = torch.bincount(owner[keep], minlength=n)
        S = torch.zeros_like(S).index_add_(0, gid, alive.long())
        E = torch.zeros_like(E).index_add_(0, gid, deg * alive) // 2
        hist.append((S, E))
        up = (S > 0) & (E * best[2] > best[1] * S)
        best = torch.where(up, torch.stack([torch.full_like(S, r), E, S]), best)
    return gone, R, best, hist, (gone > best[0][gid]).to(torch.uint8)


def _core64(off, adj):
    """Core numbers: repeated removal of the vertices of least remaining degree."""
    n = off.numel() - 1
    deg = off.diff()
    left = torch.ones(n, dtype=torch.bool, device=DEV)
    core = torch.zeros(n, dtype=torch.int64, device=DEV)
    rem = torch.arange(n, device=DEV)
    while rem.numel():
        k = int(deg[rem].min())
        front = rem[deg[rem] <= k]
        while front.numel():
            left[front] = False
            core[front] = k
            u = adj[_row_entries(off, front)]
            u = u[left[u]]
            deg.index_add_(0, u, torch.full_like(u, -1))
            u = u[deg[u] <= k]
            front = torch.unique(u)
        rem = rem[left[rem]]
    return core


def _cbds64(off, adj, core):
    n = off.numel() - 1
    owner = torch.repeat_interleave(torch.arange(n, device=DEV), off.diff())
    tail = lambda x: x.flip(0).cumsum(0).flip(0)  # noqa: E731
    V = tail(torch.bincount(core)).tolist()
    E = [e // 2 for e in tail(torch.bincount(torch.minimum(core[owner], core[adj]), minlength=len(V))).tolist()]
    k = 0
    for i in range(1, len(V)):
        if E[i] * V[k] > E[k] * V[i]:
            k = i
    inside = core >= k
    cnt = torch.bincount(owner[inside[adj]], minlength=n)
    legit = (core * V[k] > E[k]) & ~inside & (cnt * V[k] > E[k])
    extra = int(cnt[legit].sum()) + int((legit[owner] & legit[adj]).sum()) // 2
    nleg = int(legit.sum())
    return {"k_star": k, "E_core": E[k], "V_core": V[k], "E": E[k] + extra, "V": V[k] + nleg, "n_legit": nleg,
            "mask": (inside | legit).to(torch.uint8)}


def exact(case, seed):
    """What run() returns, by plain torch in 64 bits; None above 2^27 raw pairs."""
    task = case["task"]
    if task in ("batch", "serve"):
        base, off, adj = _packed(case, seed)
        g, n = base.numel() - 1, off.numel() - 1
        eps = [_eps_of(i) if task == "serve" else (case["p"], case["q"]) for i in range(g)]
        p, q = torch.tensor(eps, device=DEV).T
        _, R, best, _, mask = _peel64(base, off, adj, p, q)
        out = {"E": best[1], "V": best[2], "rounds": R, "best_round": best[0], "mask": mask}
        if task == "serve":
            out["m"] = (off[base[1:]] - off[base[:-1]]) // 2
        if task == "serve" or case["cores"]:
            out["core"] = _core64(off, adj)
            if task == "serve":
                asked = torch.arange(g, device=DEV) % 4 < 2
                out["core"] *= torch.repeat_interleave(asked, base.diff())
            out["core"] = out["core"].to(torch.int32)
        return {k: v.cpu().numpy() if task == "serve" or v.dtype == torch.int64 else v for k, v in out.items()}
    if case.get("m", 0) > 1 << 27:
        return None
    n, pairs = _pairs(case, seed)
    off, adj = _csr(n, pairs)
    m = adj.numel() // 2
    if task == "kcore":
        return {"core": _core64(off, adj).to(torch.int32)}
    if task == "cbds":
        return _cbds64(off, adj, _core64(off, adj))
    base = torch.tensor([0, n], device=DEV)
    one = lambda x: torch.tensor([x], device=DEV)  # noqa: E731
    if task == "solve":
        got = [_peel64(base, off, adj, one(p), one(q)) for p, q in SOLVE_EPS]
        return {"m": m, "masks": [x[4].cpu() for x in got], "E": [int(x[2][1]) for x in got],
                "V": [int(x[2][2]) for x in got], "core": _core64(off, adj).to(torch.int32).cpu()}
    gone, R, best, hist, mask = _peel64(base, off, adj, one(case["p"]), one(case["q"]))
    out = {"mask": mask, "E": int(best[1]), "V": int(best[2])}
    if task == "step":
        return dict(out, m=m, core=_core64(off, adj).to(torch.int32))
    if case["trace"]:
        S, E = (torch.cat(x).cpu().numpy() for x in zip(*hist))
        out.update(peel_round=gone.to(torch.int32), rounds=int(R), best_round=int(best[0]), hist_S=S, hist_E=E)
    return out
