"""A batch's graph of more than 2^20 vertices runs on the whole GPU wherever
its few edges put it in the order by work; the others keep their blocks and
clusters.  Every graph against the oracle, and the count the call reports."""
import numpy as np
import pytest

import inputs
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2103_00154_gb300 as dsg  # noqa: E402


@pytest.mark.parametrize("wide,on_grid", [((1 << 20) + 1, 1), (1 << 20, 0)])
def test_sparse_graph_behind_denser_ones(wide, on_grid):
    raws = [inputs.rmat(15, 1 << 20, seed=i) for i in range(6)]
    raws += [inputs.er_pairs(wide, 50_000, 3), inputs.path(500), inputs.empty(0), inputs.complete(40)]
    csrs = [oracle.from_raw(r) for r in raws]
    work = [2 * c.m + c.n for c in csrs]
    assert work[6] < min(work[:6]) and max(work) < sum(work) / 4
    dsg.set_tuning()
    dsg.tune_clear()
    vb, off, adj = dsg.pack_batch([(c.off, c.adj) for c in csrs], device="cuda")
    solver = dsg.BatchSolver(vb, off, adj, [(1, 10)] * len(raws), np.ones(len(raws), np.uint8))
    out_set = torch.zeros(solver.N, dtype=torch.uint8, device="cuda")
    core = torch.zeros(solver.N, dtype=torch.int32, device="cuda")
    stats = np.zeros(4, np.uint64)
    E, V, R, BR = solver.solve(out_set=out_set, core=core, stats=stats)
    assert int(stats[3]) == on_grid
    base, sets, cores = vb.cpu().numpy(), out_set.cpu().numpy(), core.cpu().numpy().view(np.uint32)
    for g, c in enumerate(csrs):
        want = oracle.bahmani(c, 1, 10)
        assert (int(E[g]), int(V[g]), int(R[g]), int(BR[g])) == (want.E, want.V, want.rounds, want.best_round), g
        lo, hi = int(base[g]), int(base[g + 1])
        np.testing.assert_array_equal(sets[lo:hi], want.mask)
        np.testing.assert_array_equal(cores[lo:hi], oracle.kcore_bz(c))
