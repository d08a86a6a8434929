"""Peels whose blocks pass the 2^32nd arrival on their meeting words (the
words and the blocks' counters start a few rounds short of it): every block
size, grids up to the whole GPU, rounds before and after.  Against the
oracle."""
import ctypes

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

CASES = [(inputs.onion(60_000, 16, 60), (1, 1000)), (inputs.rmat(16, 1 << 19, seed=4), (1, 100)),
         (inputs.path(30_000), (0, 1)), (inputs.chung_lu((1 << 20) + 1, 1 << 22, 2.1, 8.0, 60_000.0, 6), (1, 100))]


@pytest.mark.parametrize("wrap_in", [1, 2, 5])
@pytest.mark.parametrize("block", [256, 512, 1024])
@pytest.mark.parametrize("raw,pq", CASES, ids=lambda x: getattr(x, "name", None))
def test_peel_across_the_wrap(raw, pq, block, wrap_in):
    c = oracle.from_raw(raw)
    want = oracle.bahmani(c, *pq)
    dsg.set_tuning(block=block)
    try:
        g = dsg.Graph.from_csr(raw.n, c.off, c.adj)
        pr, mask = np.zeros(c.n, np.uint32), np.zeros(c.n, np.uint8)
        out = (ctypes.c_uint64 * 4)()
        N.check(dsg.lib().dsg_debug_peel_wrap(g._h, *pq, wrap_in, N.ptr(pr), N.ptr(mask), out), "peel_wrap")
        g.close()
    finally:
        dsg.set_tuning()
    assert tuple(out) == (want.E, want.V, want.rounds, want.best_round)
    np.testing.assert_array_equal(pr, want.peel_round)
    np.testing.assert_array_equal(mask, want.mask)
