"""The tiled radix scatter at the edges of its 4096-entry tiles (beta-major
order of a space, read back through H c) and the hash grouping of the
perturbative pairs where keys share a hash (few hash bits for few pairs) and
past that size, against the oracle."""
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


@pytest.mark.parametrize("nV", [2, 255, 257, 4095, 4096, 4097, 8193])
def test_sort_tile_edges(nV):
    inst = hi.random_tiny(10, 5, 4, 12)
    keys = hi.random_det_keys(10, 5, 4, nV, 21)
    c = hi.random_vector(nV, 3)
    ref = oracle.sigma_rows(inst, keys, c, np.arange(nV))
    with _solver(inst) as s:
        out = s.sigma(torch.tensor(keys.astype(np.int64), device="cuda"), torch.tensor(c, device="cuda"))
    # at most ~2e3 terms of order 1 per row
    assert np.abs(out.cpu().numpy() - ref).max() <= 1e-12 * max(1.0, np.abs(ref).max())


# pairs: every single and double of every determinant, from about 1.4e3 to
# 1.4e5 of them (the hash widens past 4096 pairs)
@pytest.mark.parametrize("nV", [1, 2, 3, 4, 6, 100])
@pytest.mark.parametrize("rdms", [False, True])
def test_pt2_groups(nV, rdms):
    inst = hi.random_tiny(10, 5, 5, 31, h_scale=0.3)
    keys = hi.random_det_keys(10, 5, 5, nV, 8)
    c = hi.random_vector(nV, 5)
    e0 = float(oracle.diag(inst, keys).min()) - 40.0
    e2, n = oracle.pt2(inst, keys, c, -1.0, e0)[:2]
    kt, ct = torch.tensor(keys.astype(np.int64), device="cuda"), torch.tensor(c, device="cuda")
    with _solver(inst) as s:
        out = s.pt2(kt, ct, -1.0, e0, rdms=rdms)
        split = s.pt2(kt, ct, -1.0, e0, max_pairs=700, rdms=rdms)
    for o in (out, split):
        assert o[1] == n
        assert abs(o[0] - e2) <= 1e-11 * abs(e2)
    if rdms:
        ref = oracle.pt2_rdm(inst, keys, c, -1.0, e0)
        for a, b in zip(out[2], ref):
            assert np.abs(a.cpu().numpy() - b).max() <= 1e-10
