"""The peel's round machinery at the sizes where it changes course: one block
or several (511 .. 513 vertices), lists shorter and longer than the grid's
threads, rows at the edges of a row piece, block 0 going on alone with little
left (and not), a last round that removes everything, hubs counted before the
first round (2^20 vertices) or not.  Everything against the oracle."""
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
    dsg.set_tuning()


CASES = [
    inputs.random_small(511, 0.02, 1), inputs.random_small(513, 0.02, 2), inputs.random_small(1500, 0.2, 3),
    inputs.star(255), inputs.star(256), inputs.star(257), inputs.star(70_000), inputs.complete(300),
    inputs.disjoint_cliques([255, 256, 257, 258, 514, 2]), inputs.onion(30_000, 16, 60),
    inputs.er_block(n=20_000, m=70_000, k=150, p=0.5, seed=3), inputs.rmat(16, 1 << 19, seed=4),
    inputs.chung_lu((1 << 20) - 1, 1 << 22, 2.1, 8.0, 60_000.0, 5),
    inputs.chung_lu((1 << 20) + 1, 1 << 22, 2.1, 8.0, 60_000.0, 6),
    inputs.union(inputs.star(140_000), inputs.er_pairs(1 << 20, 1 << 20, 7)),
]


@pytest.mark.parametrize("block", [256, 512, 1024])
@pytest.mark.parametrize("pq", [(1, 10), (1, 1000), (0, 1)], ids=lambda t: f"{t[0]}_{t[1]}")
@pytest.mark.parametrize("raw", CASES, ids=lambda r: r.name)
def test_rounds(raw, pq, block):
    c = oracle.from_raw(raw)
    want = oracle.bahmani(c, *pq)
    dsg.set_tuning(block=block)
    g = dsg.Graph.from_csr(raw.n, c.off, c.adj)
    tr = g.bahmani_trace(*pq)
    assert (tr.rounds, tr.best_round, tr.E, tr.V) == (want.rounds, want.best_round, want.E, want.V)
    np.testing.assert_array_equal(tr.hist_S, want.hist_S)
    np.testing.assert_array_equal(tr.hist_E, want.hist_E)
    np.testing.assert_array_equal(tr.peel_round, want.peel_round)
    np.testing.assert_array_equal(tr.mask, want.mask)
    g.close()


@pytest.mark.parametrize("d,core", [(64, 160), (16, 60)])
def test_candidate_lists_that_are_no_use(d, core):
    # nested shells whose degrees all lie just above the threshold: every candidate list would hold
    # nearly every vertex, so collecting rests; the rounds stay the same, with lists on and off
    raw = inputs.onion(40_000, d, core)
    c = oracle.from_raw(raw)
    want = oracle.bahmani(c, 1, 1000)
    for lazy in (True, False):
        dsg.set_tuning(peel_lazy=lazy)
        g = dsg.Graph.from_csr(raw.n, c.off, c.adj)
        tr = g.bahmani_trace(1, 1000)
        assert (tr.rounds, tr.best_round, tr.E, tr.V) == (want.rounds, want.best_round, want.E, want.V)
        np.testing.assert_array_equal(tr.peel_round, want.peel_round)
        np.testing.assert_array_equal(tr.hist_E, want.hist_E)
        g.close()
