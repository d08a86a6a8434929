"""Many ingest threads with inputs that one launch takes (up to 1.5 million
pairs, or many vertices) beside big requests: the grids they launch, whose
blocks wait for one another, fit the GPU together.  Against the oracle."""
import pytest

import inputs
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2103_00154_gb300 as dsg  # noqa: E402


@pytest.mark.parametrize("threads", [1, 8, 200])
def test_ingest_threads_and_big_requests(threads):
    raws = [inputs.er_pairs(50_000 + i, 1_400_000, i) for i in range(3)]
    raws += [inputs.er_pairs(2_000_000, 60_000, 9), inputs.chung_lu(1 << 17, 1_200_000, 2.2, 18.0, 5000.0, 4)]
    csrs = [oracle.from_raw(r) for r in raws]
    wants = [oracle.bahmani(c, 1, 10) for c in csrs]
    bad = inputs.RawGraph(raws[0].n, raws[0].src, raws[0].dst.copy(), "bad")
    bad.dst[77] = bad.n  # its launch's share of the GPU comes back too
    with dsg.Server(ingest_threads=threads, big_work=2_000_000) as srv:
        tickets = []
        for _ in range(4):
            tickets += [(i, srv.submit(r.n, r.src, r.dst, 1, 10, borrow=True)) for i, r in enumerate(raws)]
            tickets.append((None, srv.submit(bad.n, bad.src, bad.dst, 1, 10, borrow=True)))
        for i, t in tickets:
            r = srv.wait(t)
            if i is None:
                assert r["status"] != 0
            else:
                assert (r["status"], r["m"], r["E"], r["V"]) == (0, csrs[i].m, wants[i].E, wants[i].V)
