"""A paused peel resumed by one block (at most 256 vertices, or the grid capped
at one): the removed vertices and edges it starts from are the pause's, so
thresholds, history and best set are the uninterrupted peel's."""
import numpy as np
import pytest

import inputs
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2103_00154_gb300 as dsg  # noqa: E402

CASES = [inputs.random_small(33, 0.2, 1), inputs.random_small(255, 0.05, 2), inputs.random_small(256, 0.1, 3),
         inputs.path(200), inputs.disjoint_cliques([40, 30, 20, 10, 5]), inputs.onion(5000, 16, 60)]


@pytest.mark.parametrize("pq", [(0, 1), (1, 1000), (1, 10)], ids=lambda t: f"{t[0]}_{t[1]}")
@pytest.mark.parametrize("raw", CASES, ids=lambda r: r.name)
def test_paused_after_every_round(raw, pq):
    c = oracle.from_raw(raw)
    want = oracle.bahmani(c, *pq)
    g = dsg.Graph.from_csr(c.n, c.off, c.adj)
    g.set_max_blocks(1)
    for start in range(1, min(want.rounds, 12)):
        st = dsg.PeelState.begin(g, *pq)
        st.advance(start)
        snap = st.snapshot()
        st.close()
        st = dsg.PeelState.resume(g, snap)
        tr = st.finish()
        st.close()
        assert (tr.rounds, tr.E, tr.V) == (want.rounds, want.E, want.V), start
        np.testing.assert_array_equal(tr.hist_S, want.hist_S)
        np.testing.assert_array_equal(tr.hist_E, want.hist_E)
        np.testing.assert_array_equal(tr.mask, want.mask)
    g.close()
