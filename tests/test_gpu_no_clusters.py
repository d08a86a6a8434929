"""Where a GPU has no room for a thread-block cluster (here: told so by
DSG_CLUSTERS=0, in a process of its own) the calls that would launch one go to
the grid and block launches beside them and give the same results."""
import os
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SCRIPT = """
import ctypes
import numpy as np
import torch
import inputs, oracle
import paper_2103_00154_gb300 as dsg

def launches():
    buf = ctypes.create_string_buffer(1 << 16)
    dsg.lib().dsg_profile_report(buf, 1 << 16)
    return {l.split()[0]: int(l.split()[1]) for l in buf.value.decode().splitlines()}

dsg.lib().dsg_profile_enable(1)
for raw in [inputs.er_block(n=3000, m=9000, k=40, p=0.5, seed=1), inputs.star(300), inputs.empty(9),
            inputs.rmat(14, 1 << 16, seed=2)]:
    c = oracle.from_raw(raw)
    want = oracle.bahmani(c, 1, 10)
    g = dsg.Graph.from_edges(raw.n, raw.src, raw.dst)
    off, adj = g.csr()
    assert np.array_equal(off, c.off) and np.array_equal(adj, c.adj)
    tr = g.bahmani_trace(1, 10)
    assert (tr.rounds, tr.best_round, tr.E, tr.V) == (want.rounds, want.best_round, want.E, want.V)
    assert np.array_equal(tr.peel_round, want.peel_round) and np.array_equal(tr.mask, want.mask)
    assert np.array_equal(g.kcore(), oracle.kcore_bz(c))
    g.close()
assert launches().get("peel_finish") == 4  # the cluster writes its results itself
raws = [inputs.batch_graph(i, n_lo=20_000, n_hi=60_000) for i in range(6)] + [inputs.path(50), inputs.complete(9)]
csrs = [oracle.from_raw(r) for r in raws]
vb, off, adj = dsg.pack_batch([(c.off, c.adj) for c in csrs], device="cuda")
solver = dsg.BatchSolver(vb, off, adj, [(1, 10)] * len(raws), np.ones(len(raws), np.uint8))
mask, core = np.zeros(solver.N, np.uint8), np.zeros(solver.N, np.uint32)
E, V, R, BR = solver.solve(out_set=mask, core=core)
base = vb.cpu().numpy()
with dsg.Server() as srv:
    tickets = [srv.submit(r.n, r.src, r.dst, 1, 10) for r in raws]
    served = [srv.wait(t) for t in tickets]
for i, c in enumerate(csrs):
    want = oracle.bahmani(c, 1, 10)
    lo, hi = int(base[i]), int(base[i + 1])
    assert (int(E[i]), int(V[i]), int(R[i])) == (want.E, want.V, want.rounds)
    assert (served[i]["E"], served[i]["V"], served[i]["rounds"]) == (want.E, want.V, want.rounds)
    assert np.array_equal(mask[lo:hi], want.mask) and np.array_equal(core[lo:hi], oracle.kcore_bz(c))
seen = launches()
assert ("batch_clusters" in seen) == (CLUSTERS == 1), seen
print("done")
"""


@pytest.mark.parametrize("clusters", [0, 1])
def test_same_results(clusters):
    script = SCRIPT.replace("CLUSTERS", str(clusters))
    if clusters:
        script = script.replace('assert launches().get("peel_finish") == 4', 'assert "peel_finish" not in launches()')
    env = dict(os.environ, DSG_CLUSTERS=str(clusters), PYTHONPATH=ROOT)
    r = subprocess.run([sys.executable, "-c", script], cwd=ROOT, env=env, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "done" in r.stdout, r.stdout + r.stderr
