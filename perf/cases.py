"""The work that a program gives this solver, as measurable cases.

One vHCISCF orbital iteration rotates the integrals, solves the active space
by heat-bath CI (selection, connection graph, H c products, Davidson), takes
its density matrices and sends the gradient back through the rotation; E2 of
the converged state, a product without a stored graph and batches of small
spaces are the other calls in use.  Each case is one of these calls through
the package's public entry points, on the active spaces that the repository
names: a density-fitted Hamiltonian of up to (44e,44o) with a 0.3 Ha gap, the
pentacene-shaped (22e,22o) PPP space, the (12e,12o) space of the gradient
checks and the uneven batch of 10 to 24 orbitals.  A seed gives the orbital
rotation kappa of the iterate (as successive orbital iterations do), so the
spaces of two seeds are alike in size and differ in every number.  A call on
a given space takes the space found at kappa = 0 with the integrals and the
state of the turned orbitals, as a fixed-space iteration does; selected spaces
are written to buffers of a fixed capacity, as the C interface hands them out.
"""
from __future__ import annotations

import ctypes
import math

import numpy as np
import torch

import paper_1708_07544_gb300 as hci

F64 = torch.float64


# ---------------------------------------------------------------------------
# cases
# ---------------------------------------------------------------------------

def listed():
    return [
        # the smallest call: the rotation of a 10-orbital space (launches and waits)
        {"name": "rotate_10o", "kind": "rotate", "norb": 10},
        # the rotation of every (44e,44o) orbital iteration
        {"name": "rotate_44o", "kind": "rotate", "norb": 44},
        # its adjoint: dE/dh, dE/d(pq|rs) and the orbital gradient from the RDMs
        {"name": "rotate_backward_44o", "kind": "rotate_backward", "norb": 44},
        # one heat-bath selection in the middle of a (44e,44o) solve
        {"name": "select_44o", "kind": "select", "norb": 44, "eps1": 1.5e-4, "steps": 2},
        # one H c of Davidson or of a response equation, on a stored graph
        {"name": "sigma_44o", "kind": "sigma", "norb": 44, "eps1": 3e-4},
        # H c when the connections are not stored (spaces beyond device memory)
        {"name": "sigma_direct_22o", "kind": "sigma_direct", "norb": 22, "eps1": 2e-4},
        # a fixed space with new integrals: context, connection graph, cold Davidson
        {"name": "davidson_22o", "kind": "davidson", "norb": 22, "eps1": 1e-4},
        # 1- and 2-RDM of a (44e,44o) state
        {"name": "rdm12_44o", "kind": "rdm12", "norb": 44, "eps1": 3e-4},
        # E2 and its density matrices on top of a (44e,44o) state
        {"name": "pt2_44o", "kind": "pt2", "norb": 44, "eps1": 2e-4, "eps2": 2e-5},
        # the autograd energy of a small space, forward and backward
        {"name": "energy_gradient_12o", "kind": "energy_gradient", "norb": 12, "eps1": 1e-3},
        # 15 uneven spaces at once with their RDMs
        {"name": "batch_10_24o", "kind": "batch", "norb": 10, "norb_max": 24, "count": 15, "eps1": 2e-4, "streams": 8},
        # the whole (44e,44o) variational stage
        {"name": "solve_44o", "kind": "solve", "norb": 44, "eps1": 1.5e-4},
    ]


def draw(rng):
    log = lambda a, b: float("%.3g" % math.exp(rng.uniform(math.log(a), math.log(b))))  # noqa: E731
    kind = rng.choice(["rotate", "rotate_backward", "select", "sigma", "sigma_direct", "davidson", "rdm12", "pt2",
                       "energy_gradient", "batch", "solve"])
    if kind in ("rotate", "rotate_backward"):
        return {"kind": kind, "norb": rng.randint(4, 56)}
    if kind == "energy_gradient":
        return {"kind": kind, "norb": rng.randint(6, 12), "eps1": log(1e-3, 1e-2)}
    if kind == "batch":
        lo = rng.randint(8, 16)
        return {"kind": kind, "norb": lo, "norb_max": lo + rng.randint(2, 8), "count": rng.randint(4, 15),
                "eps1": log(2e-4, 2e-3), "streams": rng.choice([4, 8, 16])}
    case = {"kind": kind, "norb": rng.randint(14, 44), "eps1": log(2e-4, 2e-3)}
    if kind == "select":
        case["steps"] = 1 if case["norb"] < 28 else rng.randint(1, 2)
    if kind == "pt2":
        case["eps2"] = float("%.3g" % (case["eps1"] * rng.choice([0.1, 0.2, 0.5])))
    return case


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _symmetric(eri):
    """eri averaged over its 8 permutations, every permutation of one integral with the same bits."""
    n = eri.shape[0]
    eri = 0.5 * (eri + eri.transpose(0, 1))
    eri = 0.5 * (eri + eri.transpose(2, 3))
    m = (0.5 * (eri + eri.permute(2, 3, 0, 1))).reshape(n * n, n * n)
    p = torch.arange(n, device=eri.device)
    pair = (torch.minimum(p[:, None], p) * n + torch.maximum(p[:, None], p)).reshape(-1)
    m = m[pair][:, pair]
    return torch.where(pair[:, None] <= pair, m, m.t()).reshape(n, n, n, n).contiguous()


def _factors(n, naux, seed, scale, decay=None):
    """(pq|rs) = sum_P B^P_pq B^P_rs with seeded Gaussian factors B^P that decay with P."""
    w = np.ones(naux) if decay is None else np.exp(-np.arange(naux) / decay)
    g = np.random.default_rng(seed).standard_normal((naux, n, n))
    b = scale * math.sqrt(0.5 / float(np.sum(w * w))) * w[:, None, None] * 0.5 * (g + g.transpose(0, 2, 1))
    b = torch.tensor(b, device="cuda").reshape(naux, n * n)
    return _symmetric((b.t() @ b).reshape(n, n, n, n))


def _pentacene():
    """(22e,22o) PPP Hamiltonian of the pentacene lattice in its Hueckel orbitals."""
    import hci_inputs

    inst = hci_inputs.ppp_pentacene()
    return torch.tensor(inst.h, device="cuda"), torch.tensor(inst.eri, device="cuda"), inst.e_core


def _kappa(n, seed, sigma=0.01):
    k = np.triu(sigma * np.random.default_rng(1709 + seed).standard_normal((n, n)), 1)
    return torch.tensor(k - k.T, device="cuda")


def _turned(h, eri, seed):
    """The integrals of a later orbital iteration: turned by exp(kappa)."""
    u = torch.linalg.matrix_exp(_kappa(h.shape[0], seed))
    h = u.t() @ h @ u
    for _ in range(4):
        eri = torch.tensordot(eri, u, dims=([0], [0]))
    h = torch.triu(h)
    return h + torch.triu(h, 1).t(), _symmetric(eri)


def _integrals(kind, n, seed):
    """(h, eri, e_core) of the active space that the kind of case works on."""
    if kind == "energy_gradient":      # strongly coupled, energies from -2 to 1 Ha, no gap
        return torch.diag(torch.linspace(-2.0, 1.0, n, dtype=F64, device="cuda")), _factors(n, 4 * n, 1708, 1.0), 0.0
    if kind == "batch":                # weakly coupled members
        return (torch.diag(torch.linspace(-2.0, 1.0, n, dtype=F64, device="cuda")),
                _factors(n, 4 * n, 7544 + 1000 * seed + n, 0.2), 0.0)
    if kind in ("davidson", "sigma_direct") and n == 22:
        h, eri, e_core = _pentacene()
    else:                              # a 0.3 Ha gap, as the (44e,44o) space
        nocc = (n + 1) // 2
        d = np.concatenate([np.linspace(-2.0, -0.15, nocc), np.linspace(0.15, 1.0, n - nocc)])
        h, eri, e_core = torch.diag(torch.tensor(d, device="cuda")), _factors(n, 4 * n, 1707, 0.18, n / 1.1), 0.0
    return h, eri, e_core


def _electrons(n):
    return (n + 1) // 2, n // 2


CAPACITY = 1 << 20      # determinants that the buffers of a selected space hold


def _buffers(st):
    st["out_keys"] = torch.zeros(CAPACITY, 2, dtype=torch.int64, device="cuda")
    st["out_c"] = torch.zeros(CAPACITY, dtype=F64, device="cuda")
    return st


def _checked(status, ctx):
    if status:
        raise RuntimeError(hci.hci_last_error(ctx))


def prepare(case, seed):
    kind, n = case["kind"], case["norb"]
    st = {"case": dict(case)}
    if kind == "batch":
        st["instances"] = []
        for k in range(case["count"]):
            m = n + k % (case["norb_max"] - n + 1)
            h, eri, e_core = _integrals(kind, m, seed + k)
            st["instances"].append((m, *_electrons(m), h, eri, e_core))
        return st
    h0, eri0, e_core = _integrals(kind, n, seed)
    if kind in ("rotate", "rotate_backward", "energy_gradient"):
        h, eri = h0, eri0              # these cases turn them themselves
    else:
        h, eri = _turned(h0, eri0, seed)
    st.update(h=h, eri=eri, e_core=e_core)
    if kind in ("rotate", "energy_gradient"):
        st["kappa"] = _kappa(n, seed)
        return st
    if kind == "rotate_backward":
        # density matrices with the symmetries of those of a real state
        g = torch.Generator(device="cuda").manual_seed(seed)
        r1 = torch.randn(n, n, generator=g, dtype=F64, device="cuda") / n
        r2 = torch.randn(n, n, n, n, generator=g, dtype=F64, device="cuda") / n
        r2 = r2 + r2.permute(2, 3, 0, 1)
        st.update(kappa=_kappa(n, seed), rdm1=r1 + r1.t(), rdm2=(r2 + r2.permute(1, 0, 3, 2)).contiguous())
        return st
    if kind == "solve":
        return _buffers(st)
    with hci.HCISolver(n, *_electrons(n), h0, eri0, e_core) as s:
        st["keys"] = s.solve(case["eps1"], max_iter=case.get("steps", 30), cap=CAPACITY)["keys"].clone()
    if kind == "davidson":             # each pass has a context of its own
        return st
    st["solver"] = s = hci.HCISolver(n, *_electrons(n), h, eri, e_core)
    st["E"], st["c"], _ = s.davidson(st["keys"])
    if kind == "sigma_direct":
        s.set_sigma_mode(hci._abi.SIGMA_DIRECT)
        s.sigma(st["keys"], st["c"])
    elif kind == "select":
        s.build_lists()
        _buffers(st)
    return st


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------

def run(st):
    case = st["case"]
    kind, n = case["kind"], case["norb"]
    if kind == "rotate":
        return hci.hci_rotate(st["kappa"], st["h"], st["eri"])
    if kind == "rotate_backward":
        return hci.hci_rotate_backward(st["kappa"], st["h"], st["eri"], st["rdm1"], st["rdm2"])
    if kind == "select":
        count, ctx = ctypes.c_int64(0), st["solver"].ctx
        _checked(hci.load().hci_select(ctx, case["eps1"], st["keys"].data_ptr(), st["c"].data_ptr(), st["keys"].shape[0],
                                       st["out_keys"].data_ptr(), CAPACITY, ctypes.byref(count)), ctx)
        return st["out_keys"], count.value
    if kind in ("sigma", "sigma_direct"):
        return st["solver"].sigma(st["keys"], st["c"])
    if kind == "davidson":
        with hci.HCISolver(n, *_electrons(n), st["h"], st["eri"], st["e_core"]) as s:
            e, c, _ = s.davidson(st["keys"])
        return e, c
    if kind == "rdm12":
        return st["solver"].rdm12(st["keys"], st["c"])
    if kind == "pt2":
        return st["solver"].pt2(st["keys"], st["c"], case["eps2"], st["E"], rdms=True)
    if kind == "energy_gradient":
        x = [t.detach().requires_grad_() for t in (st["h"], st["eri"], st["kappa"])]
        e = hci.HCIEnergy.apply(*x, *_electrons(n), st["e_core"], case["eps1"])
        e.backward()
        return [e.detach()] + [t.grad for t in x]
    if kind == "batch":
        return hci.hci_solve_batch(st["instances"], case["eps1"], nstreams=case["streams"], want_rdm=True)
    with hci.HCISolver(n, *_electrons(n), st["h"], st["eri"], st["e_core"]) as s:
        count, steps, energy = ctypes.c_int64(0), ctypes.c_int(0), ctypes.c_double(0.0)
        _checked(hci.load().hci_solve(s.ctx, case["eps1"], 30, 1e-10, 400, st["out_keys"].data_ptr(),
                                      st["out_c"].data_ptr(), CAPACITY, ctypes.byref(count), ctypes.byref(energy),
                                      ctypes.byref(steps)), s.ctx)
    return st["out_keys"], st["out_c"], count.value, energy.value, steps.value


# ---------------------------------------------------------------------------
# the work of a pass, and its results in 64 bits
# ---------------------------------------------------------------------------

def work(case):
    kind, n = case["kind"], case["norb"]
    if kind in ("rotate", "rotate_backward"):
        # four quarter transforms; the backward needs the last three of four
        # twice over and one more contraction of n^5
        return {"bytes": 8.0 * n ** 4 * (2 if kind == "rotate" else 3), "flops": (8.0 if kind == "rotate" else 16.0) * n ** 5}
    st = prepare(case, 0)
    if kind == "batch":
        return {"bytes": sum(8.0 * 2 * i[0] ** 4 for i in st["instances"]),
                "flops": 2.0 * 12 * sum(float(v) * 400 for v in run(st)[1])}
    if kind in ("solve", "davidson", "energy_gradient"):
        h, eri = st["h"], st["eri"]
        if kind == "energy_gradient":
            _, h, eri = hci.hci_rotate(st["kappa"], h, eri)
        with hci.HCISolver(n, *_electrons(n), h, eri, st["e_core"]) as s:
            if kind == "davidson":
                s.davidson(st["keys"])
            else:
                s.solve(case["eps1"], cap=CAPACITY)
            t = s.stats()
        # every product reads the connections (8-byte element, 4-byte column)
        return {"bytes": 12.0 * t["sigma_nnz"] + 40.0 * t["sigma_rows"], "flops": 2.0 * t["sigma_nnz"]}
    s, nv = st["solver"], st["keys"].shape[0]
    if kind == "select":
        return {"bytes": 24.0 * nv + 16.0 * run(st)[1], "flops": 2.0 * s.stats()["last_candidates"]}
    if kind == "pt2":
        ext = run(st)[1]
        return {"bytes": 24.0 * nv + 16.0 * ext + 32.0 * n ** 4, "flops": 100.0 * ext}
    s.sigma(st["keys"], st["c"])
    nnz = s.stats()["graph_nnz"]
    if kind == "sigma":
        return {"bytes": 12.0 * nnz + 40.0 * nv, "flops": 2.0 * nnz}
    if kind == "sigma_direct":         # keys, c and integrals in, H c out
        return {"bytes": 32.0 * nv + 8.0 * n ** 4, "flops": 2.0 * nnz}
    return {"bytes": 6.0 * nnz + 24.0 * nv + 8.0 * n ** 4, "flops": 4.0 * nnz}


def _popcount(x):
    x = x - ((x >> 1) & 0x5555555555555555)
    x = (x & 0x3333333333333333) + ((x >> 2) & 0x3333333333333333)
    x = (x + (x >> 4)) & 0x0F0F0F0F0F0F0F0F
    return ((x * 0x0101010101010101) >> 56) & 0x7F


def _lowest(x):
    return torch.round(torch.log2((x & -x).to(F64))).long()


def _moved(s, p, r):
    """Sign of a+_r a_p on a string s with p occupied and r empty."""
    lo, hi = torch.minimum(p, r), torch.maximum(p, r)
    one = torch.ones_like(s)
    between = s & ((one << hi) - 1) & ~((one << (lo + 1)) - 1)
    return (1 - 2 * (_popcount(between) & 1)).to(F64)


def _pairs(keys):
    """All ordered connected pairs (i, j) of the space, a block of rows at a time."""
    a, b = keys[:, 0].contiguous(), keys[:, 1].contiguous()
    rows = max(1, int(1e8) // a.shape[0])
    for i0 in range(0, a.shape[0], rows):
        d = _popcount(a[i0:i0 + rows, None] ^ a) + _popcount(b[i0:i0 + rows, None] ^ b)
        i, j = torch.nonzero((d == 2) | (d == 4), as_tuple=True)
        yield i + i0, j


def _split(keys, i, j):
    """The pairs by kind of excitation from j to i: (kind, i, j, spin, orbitals, sign)."""
    xa, xb = keys[i, 0] ^ keys[j, 0], keys[i, 1] ^ keys[j, 1]
    da, db = _popcount(xa), _popcount(xb)
    for spin, d, x, rest in ((0, da, xa, db), (1, db, xb, da)):
        for kind, number in (("single", 2), ("double", 4)):
            m = (d == number) & (rest == 0)
            if not bool(m.any()):
                continue
            ii, jj, xx, s = i[m], j[m], x[m], keys[j[m], spin]
            holes, parts = s & xx, xx & ~s
            p, r = _lowest(holes), _lowest(parts)
            sign = _moved(s, p, r)
            if kind == "single":
                yield kind, ii, jj, spin, (p, r), sign
                continue
            q, t = _lowest(holes & (holes - 1)), _lowest(parts & (parts - 1))
            one = torch.ones_like(s)
            yield kind, ii, jj, spin, (p, r, q, t), sign * _moved(s ^ (one << p) ^ (one << r), q, t)
    m = (da == 2) & (db == 2)
    ii, jj = i[m], j[m]
    sa, sb = keys[jj, 0], keys[jj, 1]
    p, r, q, t = _lowest(sa & xa[m]), _lowest(xa[m] & ~sa), _lowest(sb & xb[m]), _lowest(xb[m] & ~sb)
    yield "mixed", ii, jj, 0, (p, r, q, t), _moved(sa, p, r) * _moved(sb, q, t)


def _occupied(keys, n):
    bits = torch.arange(n, device=keys.device)
    return ((keys[:, 0, None] >> bits) & 1).to(F64), ((keys[:, 1, None] >> bits) & 1).to(F64)


def _elements(st):
    """Diagonal of H on the space and its off-diagonal elements, block by block."""
    n, h, eri, keys = st["case"]["norb"], st["h"], st["eri"], st["keys"]
    na, nb = _occupied(keys, n)
    coul, exch = torch.einsum("ppqq->pq", eri), torch.einsum("pqqp->pq", eri)
    tot = na + nb
    diag = st["e_core"] + tot @ torch.diagonal(h) + 0.5 * (((tot @ coul) * tot).sum(1) - ((na @ exch) * na).sum(1) - ((nb @ exch) * nb).sum(1))

    def blocks():
        for i, j in _pairs(keys):
            for kind, ii, jj, spin, orb, sign in _split(keys, i, j):
                if kind == "single":
                    p, r = orb
                    same, other = (na, nb) if spin == 0 else (nb, na)
                    v = h[p, r]
                    for k in range(n):
                        v = v + (same[jj, k] + other[jj, k]) * eri[p, r, k, k] - same[jj, k] * eri[p, k, k, r]
                else:
                    p, r, q, t = orb
                    v = eri[p, r, q, t] - (eri[p, t, q, r] if kind == "double" else 0.0)
                yield ii, jj, sign * v

    return diag, blocks()


def _exact_rdms(st):
    n, keys, c = st["case"]["norb"], st["keys"], st["c"]
    na, nb = _occupied(keys, n)
    w = (c * c)[:, None]
    g1, g2 = torch.zeros(n * n, dtype=F64, device="cuda"), torch.zeros(n ** 4, dtype=F64, device="cuda")
    at = lambda p, q, r, s: ((p * n + q) * n + r) * n + s  # noqa: E731
    k = torch.arange(n, device="cuda")
    p, r = k[:, None].expand(n, n), k[None, :].expand(n, n)
    g1 += torch.diag(((na + nb) * w).sum(0)).reshape(-1)
    off = 1.0 - torch.eye(n, dtype=F64, device="cuda")
    same = ((na * w).t() @ na + (nb * w).t() @ nb) * off
    cross = (na * w).t() @ nb
    g2.index_add_(0, at(p, p, r, r).reshape(-1), (same + cross + cross.t()).reshape(-1))
    g2.index_add_(0, at(p, r, r, p).reshape(-1), -same.reshape(-1))
    for i, j in _pairs(keys):
        for kind, ii, jj, spin, orb, sign in _split(keys, i, j):
            x = sign * c[ii] * c[jj]
            if kind == "single":
                p, r = orb
                g1.index_add_(0, r * n + p, x)
                mine, other = (na, nb) if spin == 0 else (nb, na)
                for q in range(n):
                    xs = x * mine[jj, q] * (p != q)
                    xt = xs + x * other[jj, q]
                    qq = torch.full_like(p, q)
                    for idx, v in ((at(r, p, qq, qq), xt), (at(qq, qq, r, p), xt), (at(r, qq, qq, p), -xs), (at(qq, p, r, qq), -xs)):
                        g2.index_add_(0, idx, v)
                continue
            p, r, q, t = orb
            g2.index_add_(0, at(r, p, t, q), x)
            g2.index_add_(0, at(t, q, r, p), x)
            if kind == "double":
                g2.index_add_(0, at(r, q, t, p), -x)
                g2.index_add_(0, at(t, p, r, q), -x)
    return g1.reshape(n, n), g2.reshape(n, n, n, n)


def _exact_lowest(st):
    """Lowest eigenpair by Davidson on the whole matrix, to a residual of 1e-12."""
    diag, blocks = _elements(st)
    nv = diag.shape[0]
    rows, cols, vals = zip(*[(i.int(), j.int(), v) for i, j, v in blocks])
    i, j, v = torch.cat(rows).long(), torch.cat(cols), torch.cat(vals)
    order = torch.argsort(i)
    ptr = torch.zeros(nv + 1, dtype=torch.int64, device="cuda")
    ptr[1:] = torch.cumsum(torch.bincount(i, minlength=nv), 0)
    m = torch.sparse_csr_tensor(ptr, j[order].long(), v[order], (nv, nv))
    x = torch.zeros(nv, dtype=F64, device="cuda")
    x[torch.argmin(diag)] = 1.0
    base = [x]
    img = [m @ x + diag * x]
    for _ in range(400):
        q, a = torch.stack(base), torch.stack(img)
        t = q @ a.t()
        e, y = torch.linalg.eigh(0.5 * (t + t.t()))
        x, hx = y[:, 0] @ q, y[:, 0] @ a
        res = hx - e[0] * x
        if float(res.norm()) < 1e-12:
            break
        if len(base) == 30:
            keep = y[:, :4].t()
            base, img = list(keep @ q), list(keep @ a)
            q = torch.stack(base)
        den = e[0] - diag
        d = res / torch.where(den.abs() < 1e-8, torch.full_like(den, -1e-8), den)
        for _ in range(3):
            d = d - (q @ d) @ q
        d = d / d.norm()
        base.append(d)
        img.append(m @ d + diag * d)
    x = x / x.norm()
    return float(e[0]), x * torch.sign(x[torch.argmax(x.abs())])


def exact(case, seed):
    kind = case["kind"]
    if kind in ("rotate", "rotate_backward"):
        st = prepare(case, seed)
        h, eri = st["h"], st["eri"]
        kappa = st["kappa"].clone().requires_grad_()
        u = torch.linalg.matrix_exp(kappa)
        h2 = u.t() @ h @ u
        e2 = eri
        for _ in range(4):
            e2 = torch.tensordot(e2, u, dims=([0], [0]))
        if kind == "rotate":
            return u.detach(), h2.detach(), e2.detach()
        ((h2 * st["rdm1"]).sum() + 0.5 * (e2 * st["rdm2"]).sum()).backward()
        u = u.detach()
        de = 0.5 * st["rdm2"]
        for _ in range(4):
            de = torch.tensordot(de, u, dims=([0], [1]))
        return u @ st["rdm1"] @ u.t(), de, kappa.grad
    # by all pairs of determinants: about 20 s at 3.2e5 of them.  E2 and the
    # selected spaces themselves are out of reach (1e5 excitations and more of
    # each determinant), and a selection returns whole numbers.
    if kind not in ("sigma", "sigma_direct", "rdm12", "davidson"):
        return None
    st = prepare(case, seed)
    if st["keys"].shape[0] > (200_000 if kind == "davidson" else 320_000):
        return None
    if kind == "rdm12":
        return _exact_rdms(st)
    if kind == "davidson":
        return _exact_lowest(st)
    diag, blocks = _elements(st)
    out = diag * st["c"]
    for i, j, v in blocks:
        out.index_add_(0, i, v * st["c"][j])
    return out
