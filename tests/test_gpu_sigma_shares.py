"""The stored product where a warp's equal share of the connections cuts rows:
spaces from one determinant up, rows longer than several shares (a determinant
connected to the whole space), unconnected determinants (empty rows, the last
ones among them), against the oracle's rows."""
import numpy as np
import pytest
import torch

import hci_inputs as hi
import oracle

pytestmark = pytest.mark.gpu


def _check(inst, keys, seed=1, grow=0):
    import paper_1708_07544_gb300 as pkg

    dev = lambda k: torch.tensor(np.ascontiguousarray(k).astype(np.int64), device="cuda")  # noqa: E731
    c = hi.random_vector(len(keys), seed)
    ref = oracle.sigma_rows(inst, keys, c, np.arange(len(keys)))
    with pkg.HCISolver(inst.norb, inst.nalpha, inst.nbeta, torch.tensor(inst.h, device="cuda"),
                       torch.tensor(inst.eri, device="cuda"), inst.e_core) as s:
        if grow:      # the graph extended from a part of the space
            part = np.sort(np.random.default_rng(2).choice(len(keys), grow, replace=False))
            s.sigma(dev(keys[part]), torch.ones(grow, dtype=torch.float64, device="cuda"))
        out = s.sigma(dev(keys), torch.tensor(c, device="cuda"))
        again = s.sigma(dev(keys), torch.tensor(c, device="cuda"))
    assert torch.equal(out, again)
    assert np.abs(out.cpu().numpy() - ref).max() <= 1e-11 * max(1.0, np.abs(ref).max())


@pytest.mark.parametrize("nV", [1, 2, 3, 5, 33, 100, 700, 4000])
@pytest.mark.parametrize("grow", [0, 1])
def test_random_spaces(nV, grow):
    inst = hi.random_tiny(10, 5, 4, 77)
    _check(inst, hi.random_det_keys(10, 5, 4, nV, 5), grow=grow if nV > 1 else 0)


# every single and double of one determinant: its row holds the whole space
@pytest.mark.parametrize("n,na,nb", [(8, 4, 4), (12, 6, 5)])
def test_one_long_row(n, na, nb):
    inst = hi.random_tiny(n, na, nb, 9)
    k0 = hi.aufbau_key(na, nb)
    new, _, _ = oracle.select(inst, k0, np.ones(1), 0.0)
    keys = np.concatenate([k0, new])
    _check(inst, keys[np.lexsort((keys[:, 1], keys[:, 0]))])


# determinants three or more electrons apart: every row empty, or only a few
@pytest.mark.parametrize("linked", [0, 3])
def test_empty_rows(linked):
    inst = hi.random_tiny(16, 4, 4, 4)
    blocks = [0b1111, 0b11110000, 0b111100000000, 0b1111000000000000]
    keys = [(a, b) for a in blocks for b in blocks if (a, b) != (15, 15)]
    keys = [(a, b) for a, b in keys]
    keys += [(0b1111, (0b111 | (1 << (4 + k)))) for k in range(linked)]
    keys = np.array(sorted(set(keys)), dtype=np.uint64)
    _check(inst, keys)


# more connections than a share per warp: blocks of 16 warps with one and with
# several shares each, on every determinant of 8 electrons
@pytest.mark.parametrize("n", [11, 12])
def test_several_shares(n):
    import paper_1708_07544_gb300 as pkg
    from itertools import combinations

    inst = hi.random_tiny(n, 4, 4, 5)
    strings = sorted(sum(1 << p for p in o) for o in combinations(range(n), 4))
    keys = np.array([(a, b) for a in strings for b in strings], dtype=np.uint64)
    c, d = hi.random_vector(len(keys), 1), hi.random_vector(len(keys), 2)
    rows = np.unique(np.concatenate([np.arange(4), np.random.default_rng(3).integers(0, len(keys), 24),
                                     len(keys) - 1 - np.arange(4)]))
    ref = oracle.sigma_rows(inst, keys, c, rows)
    kt = torch.tensor(keys.astype(np.int64), device="cuda")
    ct, dt = torch.tensor(c, device="cuda"), torch.tensor(d, device="cuda")
    with pkg.HCISolver(inst.norb, inst.nalpha, inst.nbeta, torch.tensor(inst.h, device="cuda"),
                       torch.tensor(inst.eri, device="cuda"), inst.e_core) as s:
        hc, hd = s.sigma(kt, ct), s.sigma(kt, dt)
        assert s.stats()["graph_nnz"] > 8e7
    assert np.abs(hc.cpu().numpy()[rows] - ref).max() <= 1e-11 * max(1.0, np.abs(ref).max())
    # H is symmetric: every row and column
    a, b = float(dt @ hc), float(ct @ hd)
    assert abs(a - b) <= 1e-12 * float(dt.norm() * hc.norm() + ct.norm() * hd.norm())


# around the size from which rows are cut across shares: the determinant whose
# row holds nearly the whole space, and four empty rows, the last of the space
# among them
@pytest.mark.parametrize("nV", [2047, 2048, 2049, 2600])
@pytest.mark.parametrize("grow", [0, 40, 2000])
def test_long_and_empty_rows_where_rows_are_first_cut(nV, grow):
    inst = hi.random_tiny(16, 6, 5, 6)
    k0 = hi.aufbau_key(6, 5)
    new, _, _ = oracle.select(inst, k0, np.ones(1), 0.0)
    # more than two electrons from one another and from the aufbau determinant's neighbours
    far = [(0b111111 << 10, b << 6) for b in (0b11111, 0b1111100000)]
    far = np.array(far + [(a, 0b11111 << 11) for a in (0b111111 << 6, 0b111 << 13 | 0b111 << 6)], np.uint64)
    near = new[np.sort(np.random.default_rng(nV).choice(len(new), nV - 1 - len(far), replace=False))]
    keys = np.unique(np.concatenate([k0, near, far]), axis=0)
    lens = np.diff(oracle.hamiltonian(inst, keys).indptr) - 1
    assert len(keys) == nV and lens.max() == nV - 1 - len(far) and (lens == 0).sum() == 4 and lens[-1] == 0
    _check(inst, keys, grow=grow)


# a product on a small space with its graph cached: the content hash, the two
# orders of the vectors and the product itself
@pytest.mark.parametrize("nV", [1, 30, 400, 2048])
def test_launches_of_a_small_product(nV):
    import paper_1708_07544_gb300 as pkg
    from paper_1708_07544_gb300 import _abi

    inst = hi.random_tiny(10, 5, 4, 77)
    keys = hi.random_det_keys(10, 5, 4, nV, 5)
    kt = torch.tensor(keys.astype(np.int64), device="cuda")
    c = torch.ones(nV, dtype=torch.float64, device="cuda")
    with pkg.HCISolver(inst.norb, inst.nalpha, inst.nbeta, torch.tensor(inst.h, device="cuda"),
                       torch.tensor(inst.eri, device="cuda"), inst.e_core) as s:
        s.sigma(kt, c)
        before = _abi.hci_launch_count()
        s.sigma(kt, c)
        assert _abi.hci_launch_count() - before == 4
