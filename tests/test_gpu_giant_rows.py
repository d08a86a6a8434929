"""Rows above 8,192 entries: cut into ranges (at most 64, of about 5,000
entries), the ranges sorted by any block and put back in order.  Lengths at the
edges of the number of ranges, rows too skewed for ranges beside rows that are
not, many rows at once; built in one launch and by buckets (above 1,500,000
pairs).  The CSR against the oracle's."""
import numpy as np
import pytest

import inputs
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2103_00154_gb300 as dsg  # noqa: E402


def _raw(name, n, rows, fill):
    """rows: (vertex, neighbours); fill random pairs besides."""
    rng = np.random.default_rng(len(rows))
    src = np.concatenate([np.full(len(x), v) for v, x in rows] + [rng.integers(0, n, fill)]).astype(np.uint32)
    dst = np.concatenate([x for _, x in rows] + [rng.integers(0, n, fill)]).astype(np.uint32)
    p = rng.permutation(src.size)
    return inputs.RawGraph(n, src[p], dst[p], name)


def _spread(n, lens, seed):
    rng = np.random.default_rng(seed)
    return [(v, rng.choice(n - 64, d, replace=False) + 64) for v, d in enumerate(lens)]


N = 400_000
CASES = {
    "two and three ranges": (N, _spread(N, [8193, 9999, 10_000, 10_001, 15_000, 15_001], 1)),
    "63, 64 and more": (N, _spread(N, [314_999, 315_001, 320_000, 320_001, 390_000], 2)),
    "one id again and again": (N, [(0, np.full(30_000, 5)), (1, np.arange(100, 20_100)), (2, np.repeat(np.arange(64, 20_064), 2))]),
    "many rows": (N, _spread(N, [17_000] * 60, 3)),
}


@pytest.mark.parametrize("fill", [0, 1_600_000])
@pytest.mark.parametrize("name", CASES)
def test_csr(name, fill):
    n, rows = CASES[name]
    raw = _raw(name, n, rows, fill)
    c = oracle.from_raw(raw)
    g = dsg.Graph.from_edges(raw.n, raw.src, raw.dst)
    off, adj = g.csr()
    np.testing.assert_array_equal(off, c.off)
    np.testing.assert_array_equal(adj, c.adj)
    g.close()
