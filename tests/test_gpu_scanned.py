"""The trace's count of adjacency entries read: every row of a vertex that
failed before the last round, and the last round's only where more than 2^16
vertices were left; none where the first round removes everything."""
import numpy as np
import pytest

import inputs
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2103_00154_gb300 as dsg  # noqa: E402

CASES = [inputs.complete(300), inputs.complete(2), inputs.empty(7), inputs.star(1000), inputs.path(2000),
         inputs.er_block(n=20_000, m=70_000, k=150, p=0.5, seed=3), inputs.rmat(16, 1 << 19, seed=4),
         inputs.onion(30_000, 16, 60), inputs.cycle(1 << 16), inputs.cycle((1 << 16) + 1)]


@pytest.mark.parametrize("blocks", [0, 1, 3])
@pytest.mark.parametrize("pq", [(1, 10), (0, 1)], ids=lambda t: f"{t[0]}_{t[1]}")
@pytest.mark.parametrize("raw", CASES, ids=lambda r: r.name)
def test_entries_read(raw, pq, blocks):
    c = oracle.from_raw(raw)
    want = oracle.bahmani(c, *pq)
    g = dsg.Graph.from_csr(c.n, c.off, c.adj)
    g.set_max_blocks(blocks)
    tr = g.bahmani_trace(*pq)
    g.close()
    assert (tr.rounds, tr.E, tr.V) == (want.rounds, want.E, want.V)
    deg = np.diff(c.off.astype(np.int64))
    last = want.peel_round == want.rounds
    skipped = int(deg[last].sum()) if c.n and last.sum() <= 1 << 16 else 0
    assert tr.edges_scanned == 2 * c.m - skipped
