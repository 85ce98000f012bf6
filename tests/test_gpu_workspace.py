"""Workspaces of a context that is used many times: on small spaces its
buffers are pieces of one slab, and pieces given back are used again, so that
repeated calls ask the device's allocator for nothing."""
import ctypes

import numpy as np
import pytest
import torch

import hci_inputs as hi

pytestmark = pytest.mark.gpu

USED_CURRENT, USED_HIGH = 7, 8      # cudaMemPoolAttrUsedMemCurrent, cudaMemPoolAttrUsedMemHigh


class Pool:
    """Bytes in use of the device's default stream-ordered pool."""

    def __init__(self):
        from paper_1708_07544_gb300 import _abi

        self.rt = _abi.load()         # the CUDA runtime is among its dependencies
        self.pool = ctypes.c_void_p()
        assert self.rt.cudaDeviceGetDefaultMemPool(ctypes.byref(self.pool), torch.cuda.current_device()) == 0

    def get(self, attr):
        v = ctypes.c_uint64(0)
        assert self.rt.cudaMemPoolGetAttribute(self.pool, ctypes.c_int(attr), ctypes.byref(v)) == 0
        return v.value

    def taken_by(self, fn):
        """Most that was in use during fn beyond what was before it."""
        torch.cuda.synchronize()
        zero = ctypes.c_uint64(0)
        assert self.rt.cudaMemPoolSetAttribute(self.pool, ctypes.c_int(USED_HIGH), ctypes.byref(zero)) == 0
        before = self.get(USED_CURRENT)
        fn()
        torch.cuda.synchronize()
        return self.get(USED_HIGH) - before


@pytest.mark.parametrize("roots", [1, 2])
def test_repeated_solves_stay_on_the_slab(roots):
    import paper_1708_07544_gb300 as pkg

    inst = hi.random_tiny(5, 2, 2, 11)
    with pkg.HCISolver(5, 2, 2, torch.tensor(inst.h).cuda(), torch.tensor(inst.eri).cuda(), inst.e_core) as s:
        out_k = torch.empty(256, 2, dtype=torch.int64, device="cuda")
        out_c = torch.empty(256 * roots, dtype=torch.float64, device="cuda")
        nv, it = ctypes.c_int64(0), ctypes.c_int(0)
        e = (ctypes.c_double * roots)()
        L = pkg.load()

        def solve():
            if roots == 1:
                st = L.hci_solve(s.ctx, 1e-4, 30, 1e-10, 400, out_k.data_ptr(), out_c.data_ptr(), 256, ctypes.byref(nv),
                                 ctypes.cast(e, ctypes.POINTER(ctypes.c_double)), ctypes.byref(it))
            else:
                st = L.hci_solve_roots(s.ctx, roots, 1e-4, 30, 1e-10, 400, out_k.data_ptr(), out_c.data_ptr(), 256,
                                       ctypes.byref(nv), e, ctypes.byref(it))
            assert st == 0, pkg.hci_last_error(s.ctx)
            torch.cuda.synchronize()
            n = nv.value
            return out_k[:n].cpu().numpy().copy(), out_c[: n * roots].cpu().numpy().copy(), np.array(e[:])

        want = solve()
        for _ in range(4):
            solve()
        pool = Pool()
        early = pool.taken_by(solve)
        for _ in range(100):
            got = solve()
        # pieces used again hold what they should
        assert np.array_equal(got[0], want[0]) and np.allclose(got[2], want[2], rtol=0, atol=1e-9)
        assert np.abs(np.abs(got[1]) - np.abs(want[1])).max() < 1e-7
        late = pool.taken_by(solve)
    assert late == early == 0
