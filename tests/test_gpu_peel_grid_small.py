"""The grid-wide peel on graphs small enough for a cluster (the grid capped
below the cluster's 16 blocks): one block or several at every block size,
tiles and pieces at their edges, block 0 going on alone, with and without
candidate lists.  Against the oracle."""
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
    inputs.random_small(255, 0.04, 1), inputs.random_small(257, 0.04, 2), inputs.random_small(511, 0.02, 1),
    inputs.random_small(513, 0.02, 2), inputs.random_small(1023, 0.02, 3), inputs.random_small(1025, 0.02, 4),
    inputs.star(255), inputs.star(256), inputs.star(257), inputs.star(70_000), inputs.complete(300),
    inputs.onion(5_000, 16, 60), inputs.er_block(n=20_000, m=70_000, k=150, p=0.5, seed=3),
]


@pytest.mark.parametrize("blocks", [1, 2, 15])
@pytest.mark.parametrize("block", [256, 512, 1024])
@pytest.mark.parametrize("pq", [(1, 10), (1, 1000), (0, 1)], ids=lambda t: f"{t[0]}_{t[1]}")
@pytest.mark.parametrize("raw", CASES, ids=lambda r: r.name)
def test_rounds(raw, pq, block, blocks):
    c = oracle.from_raw(raw)
    want = oracle.bahmani(c, *pq)
    dsg.set_tuning(block=block, peel_lazy=blocks != 2)
    g = dsg.Graph.from_csr(raw.n, c.off, c.adj)
    g.set_max_blocks(blocks)
    tr = g.bahmani_trace(*pq)
    g.close()
    assert (tr.rounds, tr.best_round, tr.E, tr.V) == (want.rounds, want.best_round, want.E, want.V)
    np.testing.assert_array_equal(tr.hist_S, want.hist_S)
    np.testing.assert_array_equal(tr.hist_E, want.hist_E)
    np.testing.assert_array_equal(tr.peel_round, want.peel_round)
    np.testing.assert_array_equal(tr.mask, want.mask)
