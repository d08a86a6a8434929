"""Block sizes that nobody has given follow the rule by graph size and kernel,
also after set_tuning() has set other values or the defaults again; a given
block size holds until then.  One peel and one level-by-level core-number run
on either side of the line against the oracle."""
import numpy as np
import pytest

import inputs
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2103_00154_gb300 as dsg  # noqa: E402

LINE = 1 << 19


@pytest.fixture(autouse=True)
def _default_tuning():
    dsg.set_tuning()
    dsg.tune_clear()
    yield
    dsg.set_tuning()


@pytest.mark.parametrize("n", [LINE - 1, LINE])
def test_rule_given_and_back(n):
    raw = inputs.chung_lu(n, 1 << 21, 2.1, 8.0, 20_000.0, 5)
    c = oracle.from_raw(raw)
    rule = {"peel": 1024 if n >= LINE else 512, "kcore": 256}
    g = dsg.Graph.from_csr(n, c.off, c.adj)
    blocks = lambda: {k: g.tuning(k)["block"] for k in rule}  # noqa: E731
    assert blocks() == rule
    for given in (256, 512, 1024):
        dsg.set_tuning(block=given)
        assert blocks() == {"peel": given, "kcore": given}
        dsg.set_tuning(chunk_len=128)
        assert blocks() == rule and g.tuning("peel")["chunk_len"] == 128
    dsg.set_tuning(kcore_tail=0)
    want = oracle.bahmani(c, 1, 10)
    mask, E, V = g.bahmani(1, 10)
    assert (E, V) == (want.E, want.V)
    np.testing.assert_array_equal(mask, want.mask)
    np.testing.assert_array_equal(g.kcore(), oracle.kcore_bz(c))
    g.close()
