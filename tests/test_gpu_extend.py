"""Rows moved and appended to in chunks of entries when a space grows (rows
shorter and longer than a chunk, rows without entries, a pool that is packed
anew), and the diagonal as its difference from the aufbau determinant, against
the oracle."""
import numpy as np
import pytest
import torch

import hci_inputs as hi
import oracle

pytestmark = pytest.mark.gpu


def _solver(inst):
    import paper_1708_07544_gb300 as pkg

    return pkg.HCISolver(inst.norb, inst.nalpha, inst.nbeta, torch.tensor(inst.h, device="cuda"),
                         torch.tensor(inst.eri, device="cuda"), inst.e_core)


def _sigma(s, keys, c):
    return s.sigma(torch.tensor(keys.astype(np.int64), device="cuda"), torch.tensor(c, device="cuda")).cpu().numpy()


# 5 of 10 and 4 of 10 electrons: a row has up to 995 connections; 7 of 14: up
# to 3283, longer than a chunk
@pytest.mark.parametrize("norb,na,nb", [(10, 5, 4), (14, 7, 7)])
@pytest.mark.parametrize("sizes", [(1, 2), (3, 40, 41), (900, 1000, 5000), (20, 4000, 4300, 9000)])
def test_growing_space(norb, na, nb, sizes):
    inst = hi.random_tiny(norb, na, nb, 12)
    allk = hi.random_det_keys(norb, na, nb, sizes[-1], 4)
    order = np.random.default_rng(2).permutation(len(allk))
    with _solver(inst) as s:
        for n in sizes:
            keys = allk[np.sort(order[:n])]
            c = hi.random_vector(n, 3)
            rows = np.unique(np.linspace(0, n - 1, 60).astype(np.int64))
            ref = oracle.sigma_rows(inst, keys, c, rows)
            out = _sigma(s, keys, c)[rows]
            # some 3e3 terms of order 1 per row
            assert np.abs(out - ref).max() <= 1e-12 * max(1.0, np.abs(ref).max())
        assert s.stats()["graph_builds"] == len(sizes)


@pytest.mark.parametrize("norb,na,nb", [(1, 1, 0), (2, 1, 1), (10, 5, 4), (16, 3, 13), (16, 16, 16)])
def test_diagonal(norb, na, nb):
    inst = hi.random_tiny(norb, na, nb, 6)
    full = (1 << norb) - 1
    # aufbau, its spin-swapped and its complement (far from the reference)
    ks = {((1 << na) - 1, (1 << nb) - 1), ((full << (norb - na)) & full, (full << (norb - nb)) & full)}
    for k in sorted(ks):
        keys = np.array([k], dtype=np.uint64)
        ref = float(oracle.diag(inst, keys)[0])
        with _solver(inst) as s:
            out = float(_sigma(s, keys, np.ones(1))[0])
        # up to 1024 pairs of integrals of order 1, summed in FP64 on both sides
        assert abs(out - ref) <= 1e-12 * max(1.0, abs(ref))
