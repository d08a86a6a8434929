"""Calls where the scratch of today's faster way cannot be had but that of the
plainer one can: core numbers go back to the levels alone (whole graphs, and
what the levels leave of larger ones), a batch's clusters to blocks.  An
allocator hook refuses whatever is larger than a limit; results against the
oracle."""
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


class Refuse:
    """Allocator hook that refuses allocations above `limit` bytes."""

    def __init__(self, limit):
        self.limit, self.refused = limit, 0
        self.hooks = (N.ALLOC_FN(self._alloc), N.FREE_FN(lambda p, c, s: torch.cuda.caching_allocator_delete(int(p))))

    def _alloc(self, nbytes, ctx, stream):
        if nbytes > self.limit:
            self.refused += 1
            return None
        return torch.cuda.caching_allocator_alloc(max(int(nbytes), 1), torch.cuda.current_device(), int(stream or 0))

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


@pytest.mark.parametrize("host", [False, True], ids=["device", "host"])
@pytest.mark.parametrize("raw,tail,limit", [
    (inputs.chung_lu(200_000, 2_000_000, 2.2, 20.0, 5000.0, 3), 65536, 8 << 20),
    (inputs.union(inputs.path(100_000), inputs.block(100_000, 1500, 0.9, 4)), 2048, 3 << 19),
], ids=["whole", "tail"])
def test_core_numbers(raw, tail, limit, host):
    c = oracle.from_raw(raw)
    want = oracle.kcore_bz(c)
    g = dsg.Graph.from_csr(c.n, c.off, c.adj)
    dsg.set_tuning(kcore_tail=tail)
    out = np.zeros(c.n, np.uint32) if host else torch.zeros(c.n, dtype=torch.int32, device="cuda")
    with Refuse(limit) as hook:
        g.kcore(out=out)
    assert hook.refused > 0
    np.testing.assert_array_equal(out if host else out.cpu().numpy().view(np.uint32), want)
    assert dsg.lib().dsg_last_error() == b""
    with Refuse(1 << 16) as hook, pytest.raises(dsg.DsgError) as e:
        g.kcore(out=out)
    assert e.value.status == N.DSG_ENOMEM
    np.testing.assert_array_equal(g.kcore(), want)  # the calls after it have all they need
    g.close()


def test_batch_clusters_become_blocks():
    raws = [inputs.batch_graph(i, n_lo=20_000, n_hi=60_000) for i in range(6)] + [inputs.path(400), inputs.complete(20)]
    csrs = [oracle.from_raw(r) for r in raws]
    vb, off, adj = dsg.pack_batch([(c.off, c.adj) for c in csrs], device="cuda")
    base = vb.cpu().numpy()
    solver = dsg.BatchSolver(vb, off, adj, [(1, 10)] * len(raws), np.ones(len(raws), np.uint8))
    mask = torch.zeros(solver.N, dtype=torch.uint8, device="cuda")
    core = torch.zeros(solver.N, dtype=torch.int32, device="cuda")
    # below a cluster's slab (84 bytes a vertex), above a block's (20)
    with Refuse(20 * int(np.diff(base).max()) + (1 << 19)) as hook:
        E, V, _, _ = solver.solve(out_set=mask, core=core)
    assert hook.refused > 0
    mask, core = mask.cpu().numpy(), core.cpu().numpy().view(np.uint32)
    for i, c in enumerate(csrs):
        want = oracle.bahmani(c, 1, 10)
        assert (int(E[i]), int(V[i])) == (want.E, want.V)
        np.testing.assert_array_equal(mask[base[i]:base[i + 1]], want.mask)
        np.testing.assert_array_equal(core[base[i]:base[i + 1]], oracle.kcore_bz(c))
