"""Batches with graphs in both launches (clusters beside blocks, on a second
stream) from many short-lived threads, several at once: every result equals
the oracle's."""
import threading

import numpy as np
import pytest

import inputs
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2103_00154_gb300 as dsg  # noqa: E402


@pytest.mark.parametrize("at_once", [1, 6])
def test_short_lived_threads(at_once):
    dsg.set_tuning()
    dsg.tune_clear()
    raws = [inputs.batch_graph(i, n_lo=20_000, n_hi=40_000) for i in range(3)] + [inputs.path(300), inputs.complete(30)]
    csrs = [oracle.from_raw(r) for r in raws]
    wants = [oracle.bahmani(c, 1, 10) for c in csrs]
    mask = np.concatenate([w.mask for w in wants])
    core = np.concatenate([oracle.kcore_bz(c) for c in csrs])
    vb, off, adj = dsg.pack_batch([(c.off, c.adj) for c in csrs], device="cuda")
    ok = []

    def one():
        stream = torch.cuda.Stream()
        with torch.cuda.stream(stream):
            solver = dsg.BatchSolver(vb, off, adj, [(1, 10)] * len(raws), np.ones(len(raws), np.uint8))
            m, k = np.zeros(solver.N, np.uint8), np.zeros(solver.N, np.uint32)
            E, V, _, _ = solver.solve(out_set=m, core=k, stream=stream)
        ok.append([(int(e), int(v)) for e, v in zip(E, V)] == [(w.E, w.V) for w in wants]
                  and np.array_equal(m, mask) and np.array_equal(k, core))

    for _ in range(8):
        threads = [threading.Thread(target=one) for _ in range(at_once)]
        for t in threads:
            t.start()
        for t in threads:
            t.join()
    assert ok == [True] * (8 * at_once)
