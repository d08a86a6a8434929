"""Core numbers by the bitwise search (the vertices left for it, or the whole
graph when it is small enough): rows at the edges of a row piece (128 entries)
and of a warp's 32 pieces, graphs whose core numbers need one to eleven bits,
one block up to the whole grid, the largest graph it takes whole and the
smallest it does not, rows of more pieces than a key can say, thin and wide
cascades.  Every core number against the
oracle, the level counters against the core numbers."""
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


def _bipartite(a, b):
    i, j = np.meshgrid(np.arange(a), a + np.arange(b), indexing="ij")
    return inputs.RawGraph(a + b, i.ravel().astype(np.uint32), j.ravel().astype(np.uint32), f"K{a},{b}")


CASES = [
    inputs.complete(2), inputs.complete(33), inputs.disjoint_cliques([127, 128, 129, 130, 3]),
    inputs.disjoint_cliques([1024, 513, 257, 2]),
    _bipartite(3, 127), _bipartite(3, 128), _bipartite(2, 129), _bipartite(5, 32 * 128 + 1),
    inputs.star(127), inputs.star(128), inputs.star(129), inputs.star(4 * 128 + 1), inputs.star(131070),
    inputs.path(700), inputs.cycle(1000), inputs.onion(6000, 16, 40), inputs.empty(131072),
    inputs.star((8191 * 128) + 1), inputs.star(1_200_000), inputs.rmat(12, 1 << 17, seed=5), inputs.chung_lu(32768, 1 << 18, 2.1, 16.0, 9000.0, 9),
    inputs.chung_lu(32769, 1 << 18, 2.1, 16.0, 9000.0, 9), inputs.random_small(400, 0.5, 3),
]


@pytest.mark.parametrize("tail", [131072, 65536, 2048, 100])
@pytest.mark.parametrize("raw", CASES, ids=lambda r: r.name)
def test_core_numbers(raw, tail):
    c = oracle.from_raw(raw)
    want = oracle.kcore_bz(c)
    dsg.set_tuning(kcore_tail=tail)
    g = dsg.Graph.from_csr(raw.n, c.off, c.adj)
    np.testing.assert_array_equal(g.kcore(), want)
    core, st = g.kcore_counters()
    np.testing.assert_array_equal(core, want)
    # a level is run for every core number that occurs; all vertices are scanned at least once
    assert st["levels"] == len(np.unique(want))
    assert st["rem_scanned"] >= raw.n
    g.set_max_blocks(3)
    np.testing.assert_array_equal(g.kcore(), want)
    g.close()
