"""Selection and screened pairs at the edges of the 32-wide queues of the walk
and of the singles (32 determinants fetched at a time, 32 queued singles
evaluated at a time), with coefficients over six orders of magnitude, zeros
among them, and more than 32 orbitals: the selected set against the oracle's
enumeration, bit for bit but for its listed ties, and E2 with its pairs."""
import numpy as np
import pytest
import torch

import hci_inputs as hi
import oracle

pytestmark = pytest.mark.gpu


def _problem(norb, na, nb, nV):
    inst = hi.random_tiny(norb, na, nb, 100 + norb)
    keys = hi.random_det_keys(norb, na, nb, nV, nV + 3)
    rng = np.random.default_rng(nV)
    c = rng.choice([-1.0, 1.0], len(keys)) * 10.0 ** rng.uniform(-6, 0, len(keys))
    c[:: 7] = 0.0
    c[len(keys) // 2] = 0.5
    return inst, keys, c


def _dev(a):
    return torch.tensor(np.ascontiguousarray(a).astype(np.int64) if a.dtype == np.uint64 else a, device="cuda")


def _solver(inst):
    import paper_1708_07544_gb300 as pkg

    return pkg.HCISolver(inst.norb, inst.nalpha, inst.nbeta, _dev(inst.h), _dev(inst.eri), inst.e_core)


SPACES = [(12, 6, 5, 1), (12, 6, 5, 31), (12, 6, 5, 32), (12, 6, 5, 33), (12, 6, 5, 65), (12, 6, 5, 1025), (33, 3, 2, 40),
          (40, 1, 0, 20), (9, 9, 4, 12), (9, 0, 4, 12)]


@pytest.mark.parametrize("space", SPACES)
@pytest.mark.parametrize("eps1", [1e-4, 2e-2, 10.0])
def test_selection(space, eps1):
    inst, keys, c = _problem(*space)
    want, _, ties = oracle.select(inst, keys, c, eps1)
    with _solver(inst) as s:
        got = s.select(eps1, _dev(keys), _dev(c)).cpu().numpy().view(np.uint64).reshape(-1, 2)
    as_set = lambda k: set(map(tuple, np.asarray(k).tolist()))  # noqa: E731
    assert as_set(got) - as_set(ties) == as_set(want) - as_set(ties)
    assert len(as_set(got)) == len(got)


@pytest.mark.parametrize("space", SPACES)
@pytest.mark.parametrize("eps2", [1e-3, 0.0, -1.0])
def test_screened_pairs(space, eps2):
    inst, keys, c = _problem(*space)
    if space[0] > 30 and eps2 <= 0.0:
        pytest.skip("every pair of many orbitals")
    e0 = float(oracle.diag(inst, keys).min()) - 60.0
    e2, n = oracle.pt2(inst, keys, c, eps2, e0)
    with _solver(inst) as s:
        got = s.pt2(_dev(keys), _dev(c), eps2, e0)
    assert got[1] == n
    assert abs(got[0] - e2) <= 1e-11 * max(abs(e2), 1e-12)


# several determinants per fetch, fewer than 32: about one fetch per warp of
# the chip (9728 warps on 152 multiprocessors)
@pytest.mark.parametrize("nV", [9000, 9729, 20000, 60001])
def test_selection_of_wider_queues(nV):
    inst, keys, c = _problem(12, 6, 5, nV)
    want, _, ties = oracle.select(inst, keys, c, 0.3)
    with _solver(inst) as s:
        got = s.select(0.3, _dev(keys), _dev(c)).cpu().numpy().view(np.uint64).reshape(-1, 2)
    as_set = lambda k: set(map(tuple, np.asarray(k).tolist()))  # noqa: E731
    assert as_set(got) - as_set(ties) == as_set(want) - as_set(ties)
    assert len(as_set(got)) == len(got)


# integrals beyond FP32's range (the screens' bounds are FP32, rounded up):
# (pr|kk) of an orbital k that is empty in the determinant does not matter to
# its single p -> r, and one that is occupied decides it
@pytest.mark.parametrize("k", [1, 3])
@pytest.mark.parametrize("big", [1e38, 1e39, 1e300])
def test_integrals_beyond_fp32(k, big):
    inst = hi.random_tiny(4, 2, 1, 7)
    inst.h, inst.eri = np.zeros((4, 4)), np.zeros((4,) * 4)
    inst.h[0, 2] = inst.h[2, 0] = 0.1
    for p, r in ((0, 2), (2, 0)):
        inst.eri[p, r, k, k] = inst.eri[k, k, p, r] = big
    for c, eps1 in ((1.0, 1e-3), (1e-40, 1e-43), (1e-40, 1e-39), (1.0, 0.2)):
        for keys in (np.array([[0b0011, 0b0001]], np.uint64), np.array([[0b0011, 0b0010]], np.uint64)):
            cv = np.array([c])
            want, _, ties = oracle.select(inst, keys, cv, eps1)
            with _solver(inst) as s:
                got = s.select(eps1, _dev(keys), _dev(cv)).cpu().numpy().view(np.uint64).reshape(-1, 2)
            assert sorted(map(tuple, got.tolist())) == sorted(map(tuple, np.asarray(want).reshape(-1, 2).tolist()))
            assert len(ties) == 0


# the singles sorted by their bounds, at every width and with many equal bounds
# (integrals from a few values): the singles within a threshold are a prefix
@pytest.mark.parametrize("n,na,nb", [(1, 1, 0), (2, 1, 1), (3, 2, 1), (5, 3, 2), (16, 5, 4), (31, 3, 3), (33, 3, 2), (48, 3, 3),
                                     (64, 3, 2)])
def test_singles_of_every_width(n, na, nb):
    inst = hi.random_tiny(n, na, nb, 5)
    g = np.random.default_rng(n)
    h = g.choice([0.0, 0.125, -0.25, 0.5, 3.0], (n, n))
    inst.h = np.triu(h) + np.triu(h, 1).T
    inst.eri = np.zeros((n,) * 4)
    a0, b0 = (1 << na) - 1, (1 << nb) - 1
    k1 = (a0 ^ 1 ^ (1 << (n - 1))) if n > na else a0
    keys = np.array(sorted({(a0, b0), (k1, b0)}), np.uint64)
    c = np.array([1.0, -0.3])[: len(keys)]
    for eps1 in (1e-3, 0.124, 0.2, 0.4, 1.0, 4.0):
        want, _, ties = oracle.select(inst, keys, c, eps1)
        with _solver(inst) as s:
            got = s.select(eps1, _dev(keys), _dev(c)).cpu().numpy().view(np.uint64).reshape(-1, 2)
        assert len(ties) == 0
        assert sorted(map(tuple, got.tolist())) == sorted(map(tuple, np.asarray(want).reshape(-1, 2).tolist()))
