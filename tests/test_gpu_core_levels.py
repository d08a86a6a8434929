"""Core numbers level by level: the vertices that reach the level while a block
drains are collected in a list of the block (1,024) and claimed between two
drains; what does not fit the list is claimed at once and queued."""
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


def _layered(first, ring):
    """`first` vertices with 2 * ring neighbours each of their own, these in a ring joined to the `ring` nearest on each
    side: all of the ring falls to degree 2 * ring as the first, found by one block's scan, are drained."""
    fan = 2 * ring
    a, i = np.repeat(np.arange(first), fan), np.arange(first * fan)
    src = np.concatenate([a] + [first + i] * ring).astype(np.uint32)
    dst = np.concatenate([first + i] + [first + (i + d) % i.size for d in range(1, ring + 1)]).astype(np.uint32)
    return inputs.RawGraph(first + i.size, src, dst, f"layered{first},{ring}")


CASES = [_layered(100, 4), _layered(127, 4), _layered(128, 4), _layered(129, 4), _layered(256, 4), _layered(1000, 3),
         inputs.path(3000), inputs.star(1025), inputs.onion(6000, 16, 40), inputs.chung_lu(20000, 1 << 18, 2.1, 16.0, 9000.0, 9)]


@pytest.mark.parametrize("block", [256, 512, 1024])
@pytest.mark.parametrize("raw", CASES, ids=lambda r: r.name)
def test_level_lists(raw, block):
    want = oracle.kcore_bz(oracle.from_raw(raw))
    dsg.set_tuning(block=block, kcore_tail=0)
    g = dsg.Graph.from_edges(raw.n, raw.src, raw.dst)
    for blocks in (0, 1, 3):
        g.set_max_blocks(blocks)
        core, st = g.kcore_counters()
        np.testing.assert_array_equal(core, want)
        assert st["levels"] >= len(np.unique(want))  # a level may find that its vertices fell lower meanwhile
