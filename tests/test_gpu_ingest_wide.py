"""Ingest of few pairs over many vertices (up to 6,000,000, the most that the
one-launch path takes): sizes around the line between its cluster and its
grid, pair counts on both sides of the cluster's, the last vertices isolated
or not, and the same through a server.  The CSR against the oracle's."""
import numpy as np
import pytest

import inputs
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2103_00154_gb300 as dsg  # noqa: E402


def _sparse(n, m, top=None):
    rng = np.random.default_rng(n + m)
    return inputs.RawGraph(n, rng.integers(0, top or n, m).astype(np.uint32),
                           rng.integers(0, top or n, m).astype(np.uint32), f"n{n}_m{m}{'_low' if top else ''}")


CASES = [_sparse(65_536, 10), _sparse(65_537, 10), _sparse(65_536, 16_384), _sparse(65_537, 16_384),
         _sparse(300_000, 10_000), _sparse(5_000_000, 10), _sparse(5_000_000, 10_000), _sparse(5_000_000, 20_000),
         _sparse(5_000_000, 20_000, top=500), _sparse(6_000_000, 16_384), _sparse(6_000_001, 16_384),
         inputs.empty(6_000_000)]


@pytest.mark.parametrize("raw", CASES, ids=lambda r: r.name)
def test_csr(raw):
    c = oracle.from_raw(raw)
    src, dst = (torch.from_numpy(x.view(np.int32)).cuda() for x in (raw.src, raw.dst))
    g = dsg.Graph.from_edges(raw.n, src, dst)
    off, adj = g.csr()
    np.testing.assert_array_equal(off, c.off)
    np.testing.assert_array_equal(adj, c.adj)
    g.close()


def test_served():
    raws = [_sparse(5_000_000, 10_000), _sparse(300_000, 10_000), _sparse(5_000_000, 20_000, top=500)]
    with dsg.Server() as srv:
        sets = [np.zeros(r.n, np.uint8) for r in raws]
        tickets = [srv.submit(r.n, r.src, r.dst, 1, 10, out_set=s) for r, s in zip(raws, sets)]
        got = [srv.wait(t) for t in tickets]
    for raw, s, r in zip(raws, sets, got):
        want = oracle.bahmani(oracle.from_raw(raw), 1, 10)
        assert (r["E"], r["V"], r["rounds"]) == (want.E, want.V, want.rounds)
        np.testing.assert_array_equal(s, want.mask)
