"""Ingest of small inputs in one launch: pair counts around the lines between
cluster, grid and the bucketed path, rows at the edges of every way to sort
them (8/16/32 entries, a warp's 64 .. 1,024, a block's 16,384, longer), loops,
repeats in both orientations, empty rows, a bad id.  The CSR against the
oracle's, byte for byte."""
import numpy as np
import pytest

import inputs
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2103_00154_gb300 as dsg  # noqa: E402


def _rows(lens, n, seed, dup=False):
    """Vertex i < len(lens) gets lens[i] distinct neighbours among the others."""
    rng = np.random.default_rng(seed)
    k = len(lens)
    src = np.repeat(np.arange(k, dtype=np.uint32), lens)
    dst = np.concatenate([k + rng.choice(n - k, size=d, replace=False) for d in lens]).astype(np.uint32)
    if dup:  # some pairs again, the other way round, and loops
        again = rng.choice(src.size, size=src.size // 3, replace=False)
        loops = rng.integers(0, n, 50).astype(np.uint32)
        src, dst = (np.concatenate([src, dst[again], loops]), np.concatenate([dst, src[again], loops]))
    p = rng.permutation(src.size)
    return inputs.RawGraph(n, src[p], dst[p], f"rows{max(lens)}{'dup' if dup else ''}")


def _count(m):
    rng = np.random.default_rng(m)
    n = max(50, m // 7)
    return inputs.RawGraph(n, rng.integers(0, n, m).astype(np.uint32), rng.integers(0, n, m).astype(np.uint32), f"m{m}")


CASES = [
    inputs.empty(1), inputs.empty(700), inputs.complete(2), inputs.star(3), _count(1), _count(33),
    _count(16384), _count(16385), _count(16384 + 1024), _count(1_500_000), _count(1_500_001),
    _rows([1, 7, 8, 9, 15, 16, 17, 31, 32, 33, 63, 64, 65, 127, 128, 129], 400, 1),
    _rows([1, 7, 8, 9, 15, 16, 17, 31, 32, 33, 63, 64, 65, 127, 128, 129], 400, 2, dup=True),
    _rows([255, 256, 257, 511, 512, 513, 1023, 1024, 1025, 2047, 2048, 2049], 9000, 3, dup=True),
    _rows([4096, 4097, 8192, 8193, 16383, 16384, 16385], 60_000, 4),
    _rows([12_000, 15_000, 40_000, 20_000], 70_000, 5, dup=True),
    inputs.star(100_000), inputs.rmat(16, 1 << 20, seed=9),
]


@pytest.mark.parametrize("device", [False, True], ids=["host", "device"])
@pytest.mark.parametrize("raw", CASES, ids=lambda r: r.name)
def test_csr(raw, device):
    c = oracle.from_raw(raw)
    src, dst = raw.src, raw.dst
    if device:
        src, dst = (torch.from_numpy(x.view(np.int32)).cuda() for x in (src, dst))
    g = dsg.Graph.from_edges(raw.n, src, dst)
    off, adj = g.csr()
    np.testing.assert_array_equal(off, c.off)
    np.testing.assert_array_equal(adj, c.adj)
    g.close()


@pytest.mark.parametrize("m", [10, 16384, 30_000])
def test_bad_id_is_refused(m):
    raw = _count(m)
    src = raw.src.copy()
    src[m // 2] = raw.n
    with pytest.raises(dsg.DsgError):
        dsg.Graph.from_edges(raw.n, src, raw.dst)
    g = dsg.Graph.from_edges(raw.n, raw.src, raw.dst)
    assert g.m == oracle.from_raw(raw).m
    g.close()
