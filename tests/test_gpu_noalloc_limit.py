"""The largest graph that dsg_bahmani_noalloc takes: the nine arrays that the
header lists, 64 MiB together, to the byte."""
import ctypes

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2103_00154_gb300 as dsg  # noqa: E402
from paper_2103_00154_gb300 import _native as N  # noqa: E402

LIMIT = 64 << 20


def _need(n, p, q):
    up = lambda b: (b + 255) // 256 * 256  # noqa: E731
    return 4 * up(4 * n) + up(8 * (n + 1)) + up((n + 15) // 16 * 4) + 2 * up(8 * (dsg.round_bound(n, p, q) + 1)) + 1280


@pytest.mark.parametrize("p,q", [(1, 1), (1, 10), (0, 1)])
def test_limit(p, q):
    dsg.set_tuning()
    lo, hi = 1, 1 << 23
    while hi - lo > 1:  # the last n that fits
        mid = (lo + hi) // 2
        lo, hi = (mid, hi) if _need(mid, p, q) <= LIMIT else (lo, mid)
    E, V = ctypes.c_uint64(), ctypes.c_uint64()
    off = torch.zeros(hi + 1, dtype=torch.int64, device="cuda")
    for n, want in [(lo, N.DSG_OK), (hi, N.DSG_EINVAL)]:
        st = dsg.lib().dsg_bahmani_noalloc(n, off.data_ptr(), None, p, q, None, ctypes.byref(E), ctypes.byref(V), None)
        assert st == want
    assert (E.value, V.value) == (0, lo)
