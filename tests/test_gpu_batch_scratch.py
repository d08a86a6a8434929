"""Scratch of a batch: one large graph among hundreds of small ones does not
make every block's share as large as its own, a batch runs with fewer blocks
or clusters where there is no memory for all, and a server's batches stay
within what their requests were admitted with.  Results against the oracle."""
import numpy as np
import pytest

import inputs
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2103_00154_gb300 as dsg  # noqa: E402
from paper_2103_00154_gb300 import _native as N  # noqa: E402


class Meter:
    """Allocator hook: bytes live and their peak; allocations above `limit` are refused."""

    def __init__(self, limit=None):
        self.live, self.peak, self.largest, self.refused, self.limit, self.size = 0, 0, 0, 0, limit, {}
        self.hooks = (N.ALLOC_FN(self._alloc), N.FREE_FN(self._free))

    def _alloc(self, nbytes, ctx, stream):
        nbytes = max(int(nbytes), 1)
        if self.limit is not None and nbytes > self.limit:
            self.refused += 1
            return None
        p = torch.cuda.caching_allocator_alloc(nbytes, torch.cuda.current_device(), int(stream or 0))
        self.size[p] = nbytes
        self.live += nbytes
        self.peak = max(self.peak, self.live)
        self.largest = max(self.largest, nbytes)
        return p

    def _free(self, p, ctx, stream):
        self.live -= self.size.pop(int(p))
        torch.cuda.caching_allocator_delete(int(p))

    def __enter__(self):
        dsg.lib().dsg_set_allocator(self.hooks[0], self.hooks[1], None)
        return self

    def __exit__(self, *exc):
        dsg.lib().dsg_set_allocator(N.ALLOC_FN(), N.FREE_FN(), None)


@pytest.fixture(autouse=True)
def _default_tuning():
    dsg.set_tuning()
    dsg.tune_clear()
    yield
    dsg.set_tuning()


def _solve(csrs, meter, cores):
    vb, off, adj = dsg.pack_batch([(c.off, c.adj) for c in csrs], device="cuda")
    solver = dsg.BatchSolver(vb, off, adj, [(1, 10)] * len(csrs), np.ones(len(csrs), np.uint8) if cores else None)
    out_set = torch.zeros(solver.N, dtype=torch.uint8, device="cuda")
    core = torch.zeros(solver.N, dtype=torch.int32, device="cuda") if cores else None
    with meter:
        E, V, R, BR = solver.solve(out_set=out_set, core=core)
    base, sets = vb.cpu().numpy(), out_set.cpu().numpy()
    for g, c in enumerate(csrs):
        want = oracle.bahmani(c, 1, 10)
        assert (int(E[g]), int(V[g]), int(R[g]), int(BR[g])) == (want.E, want.V, want.rounds, want.best_round), g
        np.testing.assert_array_equal(sets[base[g]:base[g + 1]], want.mask, err_msg=f"graph {g}")
        if cores:
            got = core[int(base[g]):int(base[g + 1])].cpu().numpy().view(np.uint32)
            np.testing.assert_array_equal(got, oracle.kcore_bz(c), err_msg=f"graph {g}")
    return solver.N, int(off[-1])


def test_one_large_graph_among_small_ones():
    # the large graph sits in the middle of the packing; every graph in the block-per-graph launch
    small = [inputs.random_small(200 + i % 90, 0.05, i) for i in range(400)]
    raws = small[:200] + [inputs.chung_lu(1 << 19, 1 << 20, 2.3, 4.0, 3000.0, 7)] + small[200:]
    csrs = [oracle.from_raw(r) for r in raws]
    dsg.set_tuning(batch_split=0xffffffff)
    meter = Meter()
    n, entries = _solve(csrs, meter, cores=True)
    # 20 bytes a vertex, 1/32 an entry, under 2 KB of rounding in a small slab, and the call's tables
    assert meter.peak <= 20 * n + entries // 32 + 304 * (20 * 300 + 2048) + (1 << 20)


@pytest.mark.parametrize("cores", [False, True], ids=["peel", "cores"])
def test_fewer_teams_where_memory_is_short(cores):
    # clusters (20 mid-size graphs) beside blocks (small ones, one of them sparse and wide)
    raws = [inputs.batch_graph(i, n_lo=20_000, n_hi=60_000) for i in range(20)]
    raws += [inputs.random_small(100 + i, 0.1, i) for i in range(60)] + [inputs.path(30_000), inputs.empty(50_000)]
    csrs = [oracle.from_raw(r) for r in raws]
    free = Meter()
    _solve(csrs, free, cores)
    tight = Meter(limit=free.largest // 3)
    _solve(csrs, tight, cores)
    assert tight.refused > 0


def test_server_stays_within_what_it_admitted():
    raws = [inputs.random_small(300, 0.05, i) for i in range(150)]
    raws.insert(40, inputs.er_block(n=200_000, m=200_000, k=50, p=0.5, seed=3))
    csrs = [oracle.from_raw(r) for r in raws]
    charge = sum(64 * len(r.src) + 96 * r.n + (64 << 10) for r in raws)
    meter = Meter()
    with meter:
        with dsg.Server() as srv:
            sets = [np.zeros(r.n, np.uint8) for r in raws]
            cores = [np.zeros(r.n, np.uint32) for r in raws]
            tickets = [srv.submit(r.n, r.src, r.dst, 1, 10, want_core=True, out_set=s, core=k)
                       for r, s, k in zip(raws, sets, cores)]
            got = [srv.wait(t) for t in tickets]
    for g, (c, r) in enumerate(zip(csrs, got)):
        want = oracle.bahmani(c, 1, 10)
        assert (r["E"], r["V"], r["rounds"]) == (want.E, want.V, want.rounds), g
        np.testing.assert_array_equal(sets[g], want.mask)
        np.testing.assert_array_equal(cores[g], oracle.kcore_bz(c))
    assert meter.peak <= charge
