"""Batches whose graphs fall into the different classes: a block each, a
cluster each (few graphs: 16 blocks; more: 8), the whole GPU, and all of them
side by side; graphs just below and above the line between block and cluster,
empty and one-vertex graphs between them, core numbers for some.  Every graph
against the oracle alone."""
import numpy as np
import pytest

import inputs
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2103_00154_gb300 as dsg  # noqa: E402


@pytest.fixture(autouse=True)
def _default_tuning():
    dsg.set_tuning()
    dsg.tune_clear()
    yield


def _line(extra):
    # 2m + n = 2^17 + extra: a cycle with a tail of isolated vertices
    n = 40_000
    m = ((1 << 17) + extra - n) // 2
    v = np.arange(m, dtype=np.int64)
    return inputs.RawGraph(n, (v % n).astype(np.uint32), ((v % n + 1 + v // n) % n).astype(np.uint32), f"line{extra}")


SMALL = [inputs.empty(0), inputs.empty(1), inputs.complete(9), inputs.star(700), inputs.path(513),
         inputs.er_block(n=3000, m=9000, k=40, p=0.5, seed=1)]
MID = [inputs.batch_graph(i, n_lo=20_000, n_hi=60_000) for i in range(20)]
SETS = {
    "blocks": SMALL * 3,
    "line": SMALL + [_line(0), _line(2), _line(-2)],
    "few_clusters": SMALL + MID[:9],
    "many_clusters": MID + SMALL,
    "grid_and_rest": SMALL + MID[:3] + [inputs.rmat(17, 1 << 21, seed=3)],
    "one": [inputs.chung_lu(1 << 15, 1 << 19, 2.1, 32.0, 9000.0, 3)],
}


@pytest.mark.parametrize("cores", [False, True], ids=["peel", "cores"])
@pytest.mark.parametrize("name", list(SETS))
def test_every_class(name, cores):
    csrs = [oracle.from_raw(r) for r in SETS[name]]
    eps = [[(1, 10), (1, 1000), (0, 1), (1, 1)][i % 4] for i in range(len(csrs))]
    want_core = np.array([1 if i % 3 else 0 for i in range(len(csrs))], np.uint8)
    vb, off, adj = dsg.pack_batch([(c.off, c.adj) for c in csrs], device="cuda")
    solver = dsg.BatchSolver(vb, off, adj, eps, want_core if cores else None)
    out_set = torch.zeros(max(solver.N, 1), dtype=torch.uint8, device="cuda")
    core = torch.full((max(solver.N, 1),), -1, dtype=torch.int32, device="cuda") if cores else None
    stats = np.zeros(4, np.uint64)
    for _ in range(2):
        E, V, R, BR = solver.solve(out_set=out_set, core=core, stats=stats)
    sets, base = out_set.cpu().numpy(), vb.cpu().numpy()
    got = core.cpu().numpy().view(np.uint32) if cores else None
    scanned = 0
    for g, (c, (p, q)) in enumerate(zip(csrs, eps)):
        want = oracle.bahmani(c, p, q)
        assert (int(E[g]), int(V[g]), int(R[g]), int(BR[g])) == (want.E, want.V, want.rounds, want.best_round), g
        lo, hi = int(base[g]), int(base[g + 1])
        np.testing.assert_array_equal(sets[lo:hi], want.mask, err_msg=f"graph {g}")
        if cores:
            exp = oracle.kcore_bz(c) if want_core[g] else np.full(c.n, 0xffffffff, np.uint32)
            np.testing.assert_array_equal(got[lo:hi], exp, err_msg=f"graph {g}")
        scanned += int(want.hist_S[:want.rounds].sum())
    assert int(stats[0]) == scanned and int(stats[2]) == sum(2 * c.m for c in csrs)
