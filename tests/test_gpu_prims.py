"""The device-wide primitives themselves, called by their C++ names: the
one-block scan and its successor at their limits, and key sorts in one
cluster launch at the edges of its CTAs, past its 65536 keys and in
the passes of whole tiles."""
import ctypes

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

P, I64 = ctypes.c_void_p, ctypes.c_int64


@pytest.fixture(scope="module")
def solver():
    import paper_1708_07544_gb300 as pkg

    h = torch.zeros(2, 2, dtype=torch.float64, device="cuda")
    e = torch.zeros(2, 2, 2, 2, dtype=torch.float64, device="cuda")
    with pkg.HCISolver(2, 1, 1, h, e) as s:
        yield s


def _fn(name, *types):
    from paper_1708_07544_gb300 import _abi

    f = getattr(_abi.load(), name)
    f.argtypes, f.restype = types, ctypes.c_int
    return f


@pytest.mark.parametrize("n", [1, 2, 31, 1024, 8191, 8192, 8193, 16383, 16384, 16385, 32769, 300_001])
@pytest.mark.parametrize("in_place", [False, True])
def test_scan(solver, n, in_place):
    scan = _fn("_Z8scan_i64P7hci_ctxPKlPllS3_", P, P, P, I64, P)
    v = np.random.default_rng(n).integers(0, 1 << 40, n)
    d = torch.tensor(v, device="cuda")
    out = d if in_place else torch.full((n + 1,), -7, dtype=torch.int64, device="cuda")
    tot = torch.full((1,), -7, dtype=torch.int64, device="cuda")
    torch.cuda.synchronize()
    assert scan(solver.ctx, d.data_ptr(), out.data_ptr(), n, tot.data_ptr()) == 0
    torch.cuda.synchronize()
    c = np.cumsum(v)
    assert np.array_equal(out[:n].cpu().numpy(), np.concatenate([[0], c[:-1]]))
    assert int(tot) == c[-1]
    if not in_place:
        assert int(out[n]) == -7


@pytest.mark.parametrize("n", [2, 33, 1023, 1024, 1025, 2049, 4097, 8191, 8192, 8193, 16385, 32768, 32769, 65535, 65536, 65537])
@pytest.mark.parametrize("bits_a,bits_b", [(64, 64), (5, 0), (12, 44), (3, 9)])
def test_sort(solver, n, bits_a, bits_b):
    sort = _fn("_Z9sort_keysP7hci_ctxPmS1_lii", P, P, P, I64, ctypes.c_int, ctypes.c_int)
    r = np.random.default_rng(n + bits_a)
    lim_a, lim_b = (1 << bits_a) - 1, (1 << bits_b) - 1
    k = np.empty((n, 2), np.uint64)
    k[:, 0] = r.integers(0, lim_a, n, np.uint64, endpoint=True)
    # few distinct low words: long runs of equal digits; unsorted words ride along
    k[:, 1] = r.integers(0, min(lim_b, 300), n, np.uint64, endpoint=True) << np.uint64(max(0, bits_b - 9)) if bits_b else \
        np.arange(n, dtype=np.uint64)
    d = torch.tensor(k.astype(np.int64), device="cuda")
    tmp = torch.empty_like(d)
    torch.cuda.synchronize()
    assert sort(solver.ctx, d.data_ptr(), tmp.data_ptr(), n, bits_a, bits_b) == 0
    torch.cuda.synchronize()
    o = np.lexsort((k[:, 1], k[:, 0])) if bits_b else np.argsort(k[:, 0], kind="stable")
    assert np.array_equal(d.cpu().numpy().astype(np.uint64), k[o])
