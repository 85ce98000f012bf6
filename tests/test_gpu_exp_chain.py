"""The matrix chains of the rotation (exponential, its adjoint, the n x n
products) at every cluster form (one CTA up to 16 orbitals, several above), at
ragged block sizes and over the number of squarings, against the oracle and a
library exponential; the adjoint contraction for every accumulator form."""
import numpy as np
import pytest
import scipy.linalg as sl
import torch

import hci_inputs as hi
import oracle

pytestmark = pytest.mark.gpu


def _run(n, kap, seed=3):
    import paper_1708_07544_gb300 as pkg

    inst = hi.df_instance(n, 2 * n, seed=seed, name=f"df{n}")
    t = lambda a: torch.tensor(np.ascontiguousarray(a), device="cuda")  # noqa: E731
    g = np.random.default_rng(seed)
    r1 = g.standard_normal((n, n))
    r1 = r1 + r1.T
    r2 = g.standard_normal((n,) * 4)
    r2 = r2 + r2.transpose(2, 3, 0, 1)
    r2 = r2 + r2.transpose(1, 0, 3, 2)
    fwd = pkg.hci_rotate(t(kap), t(inst.h), t(inst.eri))
    bwd = pkg.hci_rotate_backward(t(kap), t(inst.h), t(inst.eri), t(r1), t(r2))
    return inst, r1, r2, [x.cpu().numpy() for x in fwd], [x.cpu().numpy() for x in bwd]


@pytest.mark.parametrize("n", [1, 2, 3, 10, 16, 17, 19, 33, 45, 46, 64])
def test_chain_every_form(n):
    kap = hi.random_kappa(n, seed=n, sigma=0.05)
    inst, r1, r2, (U, h2, _), (dh, _, dk) = _run(n, kap)
    ref = sl.expm(kap)
    assert np.abs(U - ref).max() <= 1e-14 * n
    assert np.abs(h2 - ref.T @ inst.h @ ref).max() <= 1e-13 * max(1.0, np.abs(inst.h).max()) * n
    assert np.abs(dh - ref @ r1 @ ref.T).max() <= 1e-13 * n * np.abs(r1).max()
    if n <= 33:
        g = oracle.gradient(inst, kap, r1, r2)
        scale = max(1.0, np.abs(g["dkappa"]).max())
        assert np.abs(dk - g["dkappa"]).max() <= 1e-12 * scale * n


# |kappa|_1 from far below 1/2 (no squaring) to several squarings; a general
# (not antisymmetric) kappa too
@pytest.mark.parametrize("norm", [1e-9, 0.499, 0.501, 3.0, 40.0])
@pytest.mark.parametrize("n", [7, 22])
@pytest.mark.parametrize("anti", [True, False])
def test_squarings(n, norm, anti):
    k = np.random.default_rng(n).standard_normal((n, n))
    k = k - k.T if anti else k
    k *= norm / np.abs(k).sum(0).max()
    if not anti and norm > 5.0:
        k *= 0.1
    inst, r1, r2, (U, _, _), (_, _, dk) = _run(n, k)
    ref = sl.expm(k)
    assert np.abs(U - ref).max() <= 1e-13 * max(1.0, norm) * max(1.0, np.abs(ref).max())
    g = oracle.gradient(inst, k, r1, r2)
    scale = max(1.0, np.abs(g["dkappa"]).max())
    assert np.abs(dk - g["dkappa"]).max() <= 1e-11 * max(1.0, norm) * scale


def test_infinite_kappa_refused():
    import paper_1708_07544_gb300 as pkg

    k = torch.zeros(5, 5, dtype=torch.float64, device="cuda")
    k[1, 2] = float("inf")
    h, e = torch.eye(5, dtype=torch.float64, device="cuda"), torch.zeros((5,) * 4, dtype=torch.float64, device="cuda")
    with pytest.raises(pkg.HCIError):
        pkg.hci_rotate(k, h, e)
    with pytest.raises(pkg.HCIError):
        pkg.hci_rotate_backward(k, h, e, h, e)


# blocks of a CTA that end in the middle of a warp (5 x 5 to 16 x 16 less a
# ragged edge): every product's loop ends thread by thread before the
# cluster's barrier.  Without two-electron integrals the whole gradient comes
# from the chains: dE/dU = h U g1^T + h^T U g1, dkappa = L_exp(kappa^T, dE/dU).
@pytest.mark.parametrize("n", [18, 21, 26, 31, 37, 50, 63])
@pytest.mark.parametrize("sigma", [0.01, 0.4])
def test_ragged_blocks(n, sigma):
    import paper_1708_07544_gb300 as pkg

    g = np.random.default_rng(n)
    kap = hi.random_kappa(n, seed=n, sigma=sigma)
    h, r1 = g.standard_normal((n, n)), g.standard_normal((n, n))
    h, r1 = h + h.T, r1 + r1.T
    t = lambda a: torch.tensor(np.ascontiguousarray(a), device="cuda")  # noqa: E731
    zero = torch.zeros((n,) * 4, dtype=torch.float64, device="cuda")
    U, h2, _ = (x.cpu().numpy() for x in pkg.hci_rotate(t(kap), t(h), zero))
    dh, _, dk = (x.cpu().numpy() for x in pkg.hci_rotate_backward(t(kap), t(h), zero, t(r1), zero))
    ref = sl.expm(kap)
    assert np.abs(U - ref).max() <= 1e-14 * n * max(1.0, np.abs(kap).sum(0).max())
    assert np.abs(h2 - ref.T @ h @ ref).max() <= 1e-13 * n * np.abs(h).max()
    assert np.abs(dh - ref @ r1 @ ref.T).max() <= 1e-13 * n * np.abs(r1).max()
    G = h @ ref @ r1.T + h.T @ ref @ r1
    want = sl.expm_frechet(kap.T, G, compute_expm=False)
    assert np.abs(dk - want).max() <= 1e-13 * n * max(1.0, np.abs(kap).sum(0).max()) * np.abs(want).max()


# a refused call leaves its outputs as they were (eri_out may be eri itself)
@pytest.mark.parametrize("n", [5, 20])
@pytest.mark.parametrize("noalloc", [False, True])
def test_refused_rotation_keeps_its_outputs(n, noalloc):
    from paper_1708_07544_gb300 import _abi

    L = _abi.load()
    dev = {"dtype": torch.float64, "device": "cuda"}
    k = torch.zeros(n, n, **dev)
    k[1, 2] = float("inf")
    h, eri = torch.randn(n, n, **dev), torch.randn(n, n, n, n, **dev)
    outs = [torch.full((n, n), 7.0, **dev), torch.full((n, n), 7.0, **dev), eri]
    keep = [o.clone() for o in outs]
    torch.cuda.synchronize()
    f = L.hci_rotate_noalloc if noalloc else L.hci_rotate
    assert f(n, k.data_ptr(), h.data_ptr(), eri.data_ptr(), *[o.data_ptr() for o in outs], None) == _abi.HCI_ERR_INVALID
    for o, w in zip(outs, keep):
        assert torch.equal(o, w)
    # backward: an infinite kappa, then an infinite dE/dU (dh and deri are done by then)
    g = [torch.full((n, n), 7.0, **dev), torch.full((n,) * 4, 7.0, **dev), torch.full((n, n), 7.0, **dev)]
    r1, r2 = torch.randn(n, n, **dev), torch.randn(n, n, n, n, **dev)
    torch.cuda.synchronize()
    back = lambda kap, rdm1: L.hci_rotate_backward(n, kap.data_ptr(), h.data_ptr(), eri.data_ptr(), rdm1.data_ptr(),  # noqa: E731
                                                   r2.data_ptr(), *[o.data_ptr() for o in g], None)
    assert back(k, r1) == _abi.HCI_ERR_INVALID
    assert all(bool((o == 7.0).all()) for o in g)
    r1[0, 0] = float("inf")
    assert back(torch.zeros(n, n, **dev), r1) == _abi.HCI_ERR_INVALID
    assert bool((g[2] == 7.0).all())
