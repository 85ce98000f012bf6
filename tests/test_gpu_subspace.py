"""The subspace eigenproblem of Davidson at its edges: every subspace size up
to the restart, exactly and nearly degenerate lowest states (where the FP32
stages give way to the FP64 Jacobi), and large energy offsets, against a dense
eigensolver on the oracle's Hamiltonian."""
import numpy as np
import pytest
import torch

import hci_inputs as hi
import oracle

pytestmark = pytest.mark.gpu


def _solver(inst):
    import paper_1708_07544_gb300 as pkg

    dev = torch.device("cuda")
    return pkg.HCISolver(inst.norb, inst.nalpha, inst.nbeta, torch.tensor(inst.h, device=dev),
                         torch.tensor(inst.eri, device=dev), inst.e_core)


def _check(inst, keys, tol=1e-10, start=None):
    H = oracle.hamiltonian(inst, keys).toarray()
    w = np.linalg.eigvalsh(H)
    kt = torch.tensor(keys.astype(np.int64), device="cuda")
    with _solver(inst) as s:
        e, c, _ = s.davidson(kt, start, tol, 2000)
        sig = s.sigma(kt, c)
    r = float((sig - e * c).norm())
    # residual bound: tol, and the rounding of a product of norm |E|
    assert r <= tol + 1e-14 * max(1.0, abs(e)) * np.sqrt(len(keys))
    # Ritz value within the residual of an eigenvalue, and the lowest one found
    assert abs(e - w[0]) <= tol + 1e-13 * max(1.0, abs(w[0]))


@pytest.mark.parametrize("nV", [1, 2, 3, 7, 8, 9, 16, 17, 24, 25, 26, 60])
def test_subspace_sizes(nV):
    inst = hi.random_tiny(6, 3, 2, 5)
    keys = hi.random_det_keys(6, 3, 2, nV, 3)
    _check(inst, keys)


@pytest.mark.parametrize("split", [0.0, 1e-13, 1e-9, 1e-6, 1e-4])
def test_close_lowest_states(split):
    # two uncoupled groups with the same spectrum up to `split`: orbitals 0-2
    # and 3-5 hold the same one-electron matrix and no two-electron terms
    inst = hi.random_tiny(6, 1, 0, 2)
    blk = inst.h[:3, :3]
    inst.h = np.zeros((6, 6))
    inst.h[:3, :3] = blk
    inst.h[3:, 3:] = blk + split * np.eye(3)
    inst.eri = np.zeros_like(inst.eri)
    keys = np.array([[1 << p, 0] for p in range(6)], dtype=np.uint64)
    g = torch.Generator().manual_seed(1)
    _check(inst, keys, start=torch.randn(6, generator=g, dtype=torch.float64).cuda())


@pytest.mark.parametrize("offset", [0.0, -1e3, 1e6])
def test_energy_offset(offset):
    inst = hi.random_tiny(6, 3, 3, 9)
    inst.e_core += offset
    keys = hi.random_det_keys(6, 3, 3, 200, 4)
    H = oracle.hamiltonian(inst, keys).toarray()
    kt = torch.tensor(keys.astype(np.int64), device="cuda")
    with _solver(inst) as s:
        e, c, _ = s.davidson(kt, None, max(1e-10, 1e-13 * abs(offset)), 2000)
    assert abs(e - np.linalg.eigvalsh(H)[0]) <= 1e-12 * max(1.0, abs(offset)) * 10


@pytest.mark.parametrize("maxit", [1, 3, 4, 5, 9])
def test_tolerance_never_met(maxit):
    # neither a negative tolerance nor NaN is met by any residual: maxit steps,
    # and the same Ritz pair from both
    inst = hi.random_tiny(6, 3, 3, 9)
    keys = hi.random_det_keys(6, 3, 3, 200, 4)
    kt = torch.tensor(keys.astype(np.int64), device="cuda")
    out = {}
    for tol in (-1.0, float("nan")):
        with _solver(inst) as s:
            out[str(tol)] = s.davidson(kt, None, tol, maxit, allow_unconverged=True)
    (e0, c0, i0), (e1, c1, i1) = out.values()
    assert i0 == i1 == maxit
    assert e0 == e1 and torch.equal(c0, c1)


@pytest.mark.parametrize("offset", [0.0, -1e3, 1e6, -3e7])
def test_energy_offset_to_rounding(offset):
    # the subspace problem is shifted by its first element, so an offset costs
    # the rounding of the diagonal, the products and the Rayleigh quotient
    # (some ulps of the offset) and no more: against the spectrum without it
    inst = hi.random_tiny(6, 3, 3, 9)
    keys = hi.random_det_keys(6, 3, 3, 200, 4)
    H = oracle.hamiltonian(inst, keys).toarray()
    w = np.linalg.eigvalsh(H)
    inst.e_core += offset
    kt = torch.tensor(keys.astype(np.int64), device="cuda")
    tol = max(1e-10, 1e-13 * abs(offset))
    with _solver(inst) as s:
        e, c, _ = s.davidson(kt, None, tol, 2000)
    c = c.cpu().numpy()
    assert abs((e - offset) - w[0]) <= 1e-14 * abs(offset) + 1e-11
    r = np.linalg.norm(H @ c - (e - offset) * c)
    assert r <= tol + 1e-14 * max(1.0, abs(offset)) * np.sqrt(len(keys))


def test_converged_start_queues_nothing():
    # a call from the converged state takes one step and launches no iteration
    # behind it (8 kernels each)
    from paper_1708_07544_gb300 import _abi

    inst = hi.random_tiny(6, 3, 3, 9)
    keys = hi.random_det_keys(6, 3, 3, 200, 4)
    kt = torch.tensor(keys.astype(np.int64), device="cuda")
    with _solver(inst) as s:
        e, c, _ = s.davidson(kt)
        before = _abi.hci_launch_count()
        e2, c2, it = s.davidson(kt, c)
        launches = _abi.hci_launch_count() - before
        # a tighter tolerance goes on from there
        e3, c3, it3 = s.davidson(kt, c, 1e-12)
    assert it == 1 and launches <= 30
    assert abs(e2 - e) <= 1e-12 and it3 > 1 and abs(e3 - e) <= 1e-11
