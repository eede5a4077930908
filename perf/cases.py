"""The cases whose speed is measured: what a user of this package has it do.

Each case is a plain dict; ``kind`` names the entry point and the other values
its sizes.  ``prepare`` draws seeded inputs on the GPU, ``run`` makes one call
of the public entry point, ``exact`` gives the same results in plain FP64 torch
operations, without the package.

The inputs are the synthetic ones of this repository's workloads: molecular-like
random integrals or a periodic Hubbard ring, and a wavefunction grown by a
rank-biased random walk over singles and doubles from the aufbau determinant
with 1/rank coefficients.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2303_05688_gb300 as asci

DEV = "cuda"


# --------------------------------- the cases --------------------------------

def _search(name, norb, na, nb, ndets, C, N, eps=0.0, precision=0, system="random"):
    return dict(name=name, kind="search", system=system, norb=norb, na=na, nb=nb, ndets=ndets,
                C=C, N=N, eps=eps, precision=precision)


def listed():
    return [
        # the smallest search: an embedding-sized Hubbard ring, where latency
        # and launches count
        _search("search_hubbard_8e8o", 8, 4, 4, 100, 100, 1000, system="hubbard"),
        # a small molecular active space, a few hundred thousand pairs
        _search("search_12e12o", 12, 6, 6, 2000, 200, 5000),
        # an ordinary active space, 5.8e7 pairs (and the search of a loop step)
        _search("search_16e16o", 16, 8, 8, 100_000, 10_000, 100_000),
        # an open-shell system of odd sizes with the screen of the paper's runs
        _search("search_13e19o_eps", 19, 7, 6, 30_011, 3_001, 20_011, eps=1e-10),
        # the headline search: Cr2-shaped, 6.7e9 pairs
        _search("search_24e30o", 30, 12, 12, 1_000_000, 100_000, 1_000_000),
        # the same system served in mixed precision with a smaller core
        _search("search_24e30o_fp32", 30, 12, 12, 100_000, 10_000, 100_000, precision=2),
        # the second-order energy of a whole wavefunction (Alg. 1, last step)
        dict(name="pt2_24e30o", kind="pt2", system="random", norb=30, na=12, nb=12, ndets=4000),
        # a batch of small uneven systems, several at a time
        dict(name="many_24", kind="many", count=24, streams=8),
        # the Hamiltonian of a selected space, from the size query to the fill
        dict(name="hamiltonian_16e16o", kind="hamiltonian", norb=16, na=8, nb=8, ndets=100_000),
        # its product with one vector, as an outside eigensolver calls it
        dict(name="spmv_16e16o", kind="spmv", norb=16, na=8, nb=8, ndets=100_000),
        # its ground state from the wavefunction's coefficients
        dict(name="davidson_16e16o", kind="davidson", norb=16, na=8, nb=8, ndets=50_000),
        # the whole method: two steps of search, merge, build, diagonalise
        dict(name="loop_16e16o", kind="loop", norb=16, na=8, nb=8, ndets=20_000, ncdets=2_000,
             ntdets=20_000, steps=2),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["search"] * 6 + ["pt2", "pt2", "many", "hamiltonian", "spmv", "davidson",
                                        "loop"])
    if kind == "many":
        return dict(kind=kind, count=rng.randint(5, 24), streams=rng.choice([2, 4, 8]))
    if kind in ("search", "pt2"):
        system = "hubbard" if kind == "search" and rng.random() < 0.2 else "random"
        norb = rng.randint(8, 14 if system == "hubbard" else 30)
        na = rng.randint(max(2, norb // 4), norb // 2)
        nb = na if rng.random() < 0.6 else max(1, na - rng.randint(1, 2))
        space = math.comb(norb, na) * math.comb(norb, nb) // 4
        nexc = _n_exc(norb, na, nb)
        if kind == "pt2":
            top = max(30, min(space, 20_000, 270_000_000 // nexc))
            return dict(kind=kind, system=system, norb=norb, na=na, nb=nb,
                        ndets=_log(rng, 20, top))
        ndets = _log(rng, 50, max(60, min(space, 1_000_000)))
        C = min(_log(rng, 20, 100_000), ndets, max(20, 2_000_000_000 // nexc))
        N = _log(rng, 100, max(101, min(1_000_000, space, C * nexc // 10)))
        eps = rng.choice([0.0, 0.0, 0.0, 1e-10]) if system == "random" else 0.0
        return dict(kind=kind, system=system, norb=norb, na=na, nb=nb, ndets=ndets, C=C,
                    N=N, eps=eps, precision=rng.choice([0, 0, 0, 1, 2]))
    norb = rng.randint(12, 20)
    na = rng.randint(norb // 3, norb // 2)
    nb = na if rng.random() < 0.6 else na - 1
    space = math.comb(norb, na) * math.comb(norb, nb) // 4
    if kind == "loop":
        ntdets = _log(rng, 500, min(space, 20_000))
        return dict(kind=kind, norb=norb, na=na, nb=nb, ndets=ntdets // 2,
                    ncdets=max(20, ntdets // 10), ntdets=ntdets, steps=2)
    return dict(kind=kind, norb=norb, na=na, nb=nb,
                ndets=_log(rng, 1_000, min(space, 60_000 if kind == "davidson" else 100_000)))


def _n_exc(n, na, nb):
    va, vb = n - na, n - nb
    return (na * va + nb * vb + math.comb(na, 2) * math.comb(va, 2)
            + math.comb(nb, 2) * math.comb(vb, 2) + na * va * nb * vb)


# ---------------------------------- inputs ----------------------------------

def _random_integrals(n, rng):
    """Sorted orbital energies, small hoppings, (pq|rs) decaying with the orbital
    distance, 8-fold symmetric."""
    h1 = np.triu(rng.normal(0.0, 0.05, (n, n)), 1)
    h1 = h1 + h1.T
    h1[np.arange(n), np.arange(n)] = np.sort(rng.uniform(-2.0, 2.0, n))
    p, q = np.meshgrid(np.arange(n), np.arange(n), indexing="ij")
    hi, lo = np.maximum(p, q), np.minimum(p, q)
    pair = (hi * (hi + 1) // 2 + lo).reshape(-1)
    decay = np.exp(-0.3 * np.abs(p - q)).reshape(-1)
    npair = n * (n + 1) // 2
    a, b = np.maximum(pair[:, None], pair[None, :]), np.minimum(pair[:, None], pair[None, :])
    noise = rng.normal(0.0, 0.1, npair * (npair + 1) // 2)[a * (a + 1) // 2 + b]
    eri = 0.5 * decay[:, None] * decay[None, :] * (1.0 + noise)
    return h1, eri.reshape(n, n, n, n)


def _hubbard_integrals(n, U):
    h1 = np.zeros((n, n))
    for p in range(n):
        h1[p, (p + 1) % n] = h1[(p + 1) % n, p] = -1.0
    eri = np.zeros((n,) * 4)
    for p in range(n):
        eri[p, p, p, p] = U
    return h1, eri


def _bits(words, n):
    return ((words[:, None] >> torch.arange(n, device=DEV)[None, :]) & 1).bool()


def _pick2(mask, gen):
    """Two distinct random True columns of each row (or fewer, where it has fewer)."""
    k = torch.rand(mask.shape, generator=gen, device=DEV)
    return torch.topk(torch.where(mask, k, k - 2.0), min(2, mask.shape[1]), dim=1).indices


def _walk(n, na, nb, ndets, gen):
    """Distinct determinants (beta << 32 | alpha) of a rank-biased random walk, rank order."""
    keys = torch.tensor([((1 << nb) - 1) << 32 | ((1 << na) - 1)], dtype=torch.int64, device=DEV)
    one = torch.ones((), dtype=torch.int64, device=DEV)
    kinds = torch.tensor([0.125, 0.25, 0.4375, 0.625], device=DEV)
    counts = ((na, n - na), (nb, n - nb))
    while len(keys) < ndets:
        m = min(max(2 * len(keys), 64), 1 << 19)
        u = torch.rand(m, generator=gen, device=DEV, dtype=torch.float64)
        k = keys[(len(keys) * u ** 3).long().clamp_(max=len(keys) - 1)]
        # alpha single, beta single, alpha-alpha, beta-beta, alpha-beta double
        kind = torch.bucketize(torch.rand(m, generator=gen, device=DEV), kinds, right=True)
        ok = torch.ones(m, dtype=torch.bool, device=DEV)
        for spin, (no, nv) in enumerate(counts):
            occ = _bits((k >> (32 * spin)) & 0xFFFFFFFF, n)
            h, p = _pick2(occ, gen), _pick2(~occ, gen)
            flip = (one << h) ^ (one << p)
            first = (kind == spin) | (kind == 4) | (kind == 2 + spin)
            second = kind == 2 + spin
            ok &= ~(first if min(no, nv) < 1 else second if min(no, nv) < 2 else ~ok)
            k = k ^ torch.where(first, flip[:, 0] << (32 * spin), 0)
            if flip.shape[1] > 1:
                k = k ^ torch.where(second, flip[:, 1] << (32 * spin), 0)
        v, at = torch.sort(k[ok], stable=True)
        first = torch.ones_like(v, dtype=torch.bool)
        first[1:] = v[1:] != v[:-1]
        seen = torch.sort(keys).values
        new = first & (seen[torch.searchsorted(seen, v).clamp_(max=len(seen) - 1)] != v)
        keys = torch.cat([keys, k[ok][torch.sort(at[new]).values]])[:ndets]
    return keys


def _dets(keys):
    return torch.stack([keys & 0xFFFFFFFF, keys >> 32], 1).contiguous()


class _System:
    """Integrals, wavefunction and E0 of one system, from the seed."""

    def __init__(self, system, norb, na, nb, ndets, seed, space=None):
        rng = np.random.default_rng(seed)
        if system == "hubbard":
            h1, eri = _hubbard_integrals(norb, float(rng.uniform(1.0, 8.0)))
        else:
            h1, eri = _random_integrals(norb, rng)
        gen = torch.Generator(device=DEV)
        gen.manual_seed(seed if space is None else space)
        self.n, self.na, self.nb = norb, na, nb
        self.h1, self.eri = torch.tensor(h1, device=DEV), torch.tensor(eri, device=DEV)
        self.keys = _walk(norb, na, nb, ndets, gen)
        if space is not None:  # one space, its neighbouring orbitals swapped by the seed
            gen.manual_seed(seed)
            for p in range(0, norb - 1, 2):
                if float(torch.rand((), generator=gen, device=DEV)) < 0.5:
                    both = (1 << p) | (1 << (p + 32))
                    self.keys = ((self.keys & ~(3 * both)) | ((self.keys & both) << 1)
                                 | ((self.keys >> 1) & both))
        self.dets = _dets(self.keys)
        c = torch.where(torch.rand(ndets, generator=gen, device=DEV) < 0.5, -1.0, 1.0).double()
        c[0] = 1.0
        c /= torch.arange(1, ndets + 1, device=DEV)
        self.c = c / c.norm()
        # an energy below the diagonal of the leading determinants
        self.E0 = float(self.diag(self.keys[:2000]).min()) - 1.0

    def diag(self, keys):
        i = torch.arange(self.n, device=DEV)
        J = self.eri[i[:, None], i[:, None], i[None, :], i[None, :]]
        JK = J - self.eri[i[:, None], i[None, :], i[None, :], i[:, None]]
        out = []
        for k in keys.split(1 << 22):
            a, b = _bits(k & 0xFFFFFFFF, self.n).double(), _bits(k >> 32, self.n).double()
            h = torch.diagonal(self.h1)
            out.append((a + b) @ h + 0.5 * ((a @ JK) * a + (b @ JK) * b).sum(1)
                       + ((a @ J) * b).sum(1))
        return torch.cat(out)


def _many_systems(count, seed):
    """Small uneven systems, Hubbard rings and random integrals in turn, with
    1e3 to 1e4 core determinants and 1e4 to 1e5 selected (at most a quarter of
    the space).  The sizes are the batch's own, the systems the seed's."""
    rng = np.random.default_rng(count)
    out = []
    for k in range(count):
        n = int(rng.choice([8, 10, 12, 14, 16, 18, 20]))
        space = math.comb(n, n // 2) ** 2
        C, N = int(10 ** rng.uniform(3, 4)), min(int(10 ** rng.uniform(4, 5)), space // 4)
        nd = min(2 * C, space // 4)
        s = _System("hubbard" if k % 2 == 0 else "random", n, n // 2, n // 2, nd, seed + 1000 + k)
        out.append(dict(dets=s.dets, coeffs=s.c, E0=s.E0, h1=s.h1, eri=s.eri, ecore=0.0,
                        C=min(C, nd), N=N))
    return out


def _system(case, seed):
    # a Hamiltonian has as many stored elements for one seed as for another
    return _System(case.get("system", "random"), case["norb"], case["na"], case["nb"],
                   case["ndets"], seed, space=17 if case["kind"] == "hamiltonian" else None)


def _selected(case, seed):
    """A system whose wavefunction is in key order, as a search's merge leaves it."""
    s = _system(case, seed)
    s.keys, at = torch.sort(s.keys)
    s.dets, s.c = _dets(s.keys), s.c[at].contiguous()
    return s


def prepare(case, seed):
    kind = case["kind"]
    if kind == "many":
        return case, _many_systems(case["count"], seed), None
    if kind in ("hamiltonian", "spmv", "davidson"):
        s = _selected(case, seed)
        return case, s, None if kind == "hamiltonian" else asci.hamiltonian(s.dets, s.h1, s.eri,
                                                                            0.0)
    return case, _system(case, seed), None


def run(state):
    case, s, H = state
    kind = case["kind"]
    if kind == "search":
        d, sc, st = asci.search(s.dets, s.c, s.E0, s.h1, s.eri, 0.0, case["C"], case["N"],
                                eps=case["eps"], precision=case["precision"], sort_output=True)
        return d, sc, [st.generated, st.surviving, st.unique, st.excluded]
    if kind == "pt2":
        e, st = asci.pt2(s.dets, s.c, s.E0, s.h1, s.eri, 0.0)
        return e, [st.generated, st.unique, st.excluded]
    if kind == "many":
        got = asci.search_many(s, streams=case["streams"], sort_output=True)
        return [x for d, sc, _ in got for x in (d, sc)]
    if kind == "hamiltonian":
        return asci.hamiltonian(s.dets, s.h1, s.eri, 0.0)
    if kind == "spmv":
        return asci.spmv(H, s.c)
    if kind == "davidson":
        e, v, _, _ = asci.davidson(H, s.c, tol=1e-10)
        return e, v
    d, c, e, _ = asci.asci_loop(s.dets, s.c, s.h1, s.eri, 0.0, ncdets=case["ncdets"],
                                ntdets=case["ntdets"], max_steps=case["steps"], etol=0.0,
                                tol=1e-10)
    return d, c, e


# ----------------------------------- work -----------------------------------

def _mean_row(case):
    """Expected stored elements of one row, from the densities measured on such
    spaces at 16 orbitals (about 1 in 270 of 1e5 columns), capped by the row's
    connections."""
    return min(case["ndets"], _n_exc(case["norb"], case["na"], case["nb"]),
               50 + case["ndets"] // 270)


def work(case):
    """Bytes: inputs read once, outputs written once.  Flops: a product and an
    addition for each generated pair or stored element."""
    kind = case["kind"]
    if kind == "many":  # the mean over the drawn sizes
        pairs = np.mean([_n_exc(n, n // 2, n // 2) for n in (8, 10, 12, 14, 16, 18, 20)]) * 3900
        return {"bytes": case["count"] * (7800 * 24 + 3e4 * 24 + 60_000 * 8),
                "flops": case["count"] * 2.0 * float(pairs)}
    n, nd = case["norb"], case["ndets"]
    ints, psi = 8.0 * (n ** 4 + n ** 2), 24.0 * nd
    pairs = _n_exc(n, case["na"], case["nb"])
    if kind == "search":
        return {"bytes": ints + psi + 24.0 * case["N"], "flops": 2.0 * pairs * case["C"]}
    if kind == "pt2":
        return {"bytes": ints + psi + 8.0, "flops": 2.0 * pairs * nd}
    nnz = float(nd) * _mean_row(case)
    if kind == "hamiltonian":
        return {"bytes": ints + 16.0 * nd + 8.0 * nd + 12.0 * nnz, "flops": nnz}
    if kind == "spmv":
        return {"bytes": 12.0 * nnz + 24.0 * nd, "flops": 2.0 * nnz}
    if kind == "davidson":  # the matrix once and both vectors; some 100 products of it
        return {"bytes": 12.0 * nnz + 24.0 * nd, "flops": 200.0 * nnz}
    nt = float(case["ntdets"]) * min(case["ntdets"], 50 + case["ntdets"] // 270)
    return {"bytes": ints + psi + 24.0 * case["ntdets"],
            "flops": case["steps"] * (2.0 * pairs * case["ncdets"] + 200.0 * nt)}


# ---------------------------------- FP64 ------------------------------------

def _between(below, x, y):
    """Occupied orbitals strictly between x (occupied) and y (empty); below: exclusive prefix."""
    bx, by = torch.gather(below, 1, x), torch.gather(below, 1, y)
    return torch.where(y > x, by - bx - 1, bx - by)


def _excitations(s, keys):
    """Every single and double of each key: target keys and H_ij, both (len(keys), n_exc)."""
    n, m = s.n, len(keys)
    i = torch.arange(n, device=DEV)
    kk = s.eri[:, :, i, i]                          # (ia|kk)
    same = kk - s.eri[:, i, i, :].permute(0, 2, 1)  # (ia|kk) - (ik|ka)
    occ = [_bits(keys & 0xFFFFFFFF, n), _bits(keys >> 32, n)]
    one = torch.ones((), dtype=torch.int64, device=DEV)
    targets, values, singles = [], [], []
    for spin, ne in enumerate((s.na, s.nb)):
        o = occ[spin]
        order = torch.sort(o.int(), dim=1, descending=True, stable=True).indices
        oc, vi = order[:, :ne], order[:, ne:]
        below = o.long().cumsum(1) - o.long()
        nv = n - ne
        x = oc[:, :, None].expand(m, ne, nv).reshape(m, -1)
        y = vi[:, None, :].expand(m, ne, nv).reshape(m, -1)
        sign = 1.0 - 2.0 * (_between(below, x, y) & 1).double()
        f = (o.double() @ same.reshape(n * n, n).T + occ[1 - spin].double() @ kk.reshape(n * n, n).T
             + s.h1.reshape(1, -1))
        flip = ((one << x) ^ (one << y)) << (32 * spin)
        targets.append(keys[:, None] ^ flip)
        values.append(sign * torch.gather(f, 1, x * n + y))
        singles.append((x, y, sign, flip))
        if ne > 1 and nv > 1:
            a, b = torch.triu_indices(ne, ne, 1, device=DEV)
            c, d = torch.triu_indices(nv, nv, 1, device=DEV)
            h1, h2 = (oc[:, t][:, :, None].expand(-1, -1, len(c)).reshape(m, -1) for t in (a, b))
            p1, p2 = (vi[:, t][:, None, :].expand(-1, len(a), -1).reshape(m, -1) for t in (c, d))
            lo, hi = torch.minimum(h2, p2), torch.maximum(h2, p2)
            par = (_between(below, h1, p1) + _between(below, h2, p2)
                   + ((h1 > lo) & (h1 < hi)).long() + ((p1 > lo) & (p1 < hi)).long())
            v = (s.eri.reshape(-1)[((h1 * n + p1) * n + h2) * n + p2]
                 - s.eri.reshape(-1)[((h1 * n + p2) * n + h2) * n + p1])
            targets.append(keys[:, None] ^ (((one << h1) ^ (one << p1) ^ (one << h2) ^ (one << p2))
                                            << (32 * spin)))
            values.append((1.0 - 2.0 * (par & 1).double()) * v)
    (xa, ya, sa, fa), (xb, yb, sb, fb) = singles
    at = ((xa * n + ya) * n * n)[:, :, None] + (xb * n + yb)[:, None, :]
    v = s.eri.reshape(-1)[at] * sa[:, :, None] * sb[:, None, :]
    targets.append((keys[:, None, None] ^ fa[:, :, None] ^ fb[:, None, :]).reshape(m, -1))
    values.append(v.reshape(m, -1))
    return torch.cat(targets, 1), torch.cat(values, 1)


def _targets(s, C, eps):
    """Numerators and E0 - H_ii of the unique targets outside the wavefunction, key order."""
    core = torch.argsort(s.c.abs(), descending=True, stable=True)[:C]
    block = max(1, (1 << 24) // _n_exc(s.n, s.na, s.nb))
    keys, vals = [], []
    for part in core.split(block):
        t, v = _excitations(s, s.keys[part])
        t, v = t.reshape(-1), (v * s.c[part][:, None]).reshape(-1)
        if eps > 0.0:
            keep = v.abs() > eps * (s.E0 - s.diag(t)).abs()
            t, v = t[keep], v[keep]
        keys.append(t)
        vals.append(v)
    keys, at = torch.sort(torch.cat(keys))
    vals = torch.cat(vals)[at]
    del at
    keys, inverse = torch.unique_consecutive(keys, return_inverse=True)
    num = torch.zeros(len(keys), dtype=torch.float64, device=DEV).index_add_(0, inverse, vals)
    psi = torch.sort(s.keys).values
    out = psi[torch.searchsorted(psi, keys).clamp_(max=len(psi) - 1)] != keys
    keys, num = keys[out], num[out]
    return keys, num, s.E0 - s.diag(keys)


def _matrix(s):
    """H over s.keys (key order): rows, columns and elements, row by row."""
    n, keys = s.n, s.keys
    occ = torch.cat([_bits(keys & 0xFFFFFFFF, n), _bits(keys >> 32, n)], 1)
    half = occ.half()
    i = torch.arange(n, device=DEV)
    kk = s.eri[:, :, i, i]
    same = kk - s.eri[:, i, i, :].permute(0, 2, 1)
    flat = s.eri.reshape(-1)
    rows, cols, vals = [], [], []
    for r0 in range(0, len(keys), 4096):
        near = half[r0:r0 + 4096] @ half.T >= s.na + s.nb - 2
        r, c = torch.nonzero(near, as_tuple=True)
        r = r + r0
        rows.append(r)
        cols.append(c)
        for rr, cc in zip(r.split(1 << 22), c.split(1 << 22)):
            bra, ket = occ[rr], occ[cc]
            hole, part = ket & ~bra, bra & ~ket
            nh = hole.sum(1)
            ha = hole[:, :n].sum(1)
            big = 2 * n
            pos = torch.arange(2 * n, device=DEV)[None, :]
            h1 = torch.where(hole, pos, big).min(1).values
            h2 = torch.where(hole, pos, -1).max(1).values
            p1 = torch.where(part, pos, big).min(1).values
            p2 = torch.where(part, pos, -1).max(1).values
            # the sign of h1 -> p1, then h2 -> p2, on the string of 2 n spin orbitals
            below = ket.long().cumsum(1) - ket.long()
            v = torch.zeros(len(rr), dtype=torch.float64, device=DEV)
            k0 = nh == 0
            v[k0] = s.diag(keys[rr[k0]])
            k1 = nh == 1
            x, y = h1[k1], p1[k1]
            sg = 1.0 - 2.0 * (_between(below[k1], x[:, None], y[:, None])[:, 0] & 1).double()
            spin = (x >= n).long()
            a, b = ket[k1][:, :n].double(), ket[k1][:, n:].double()
            o, u = torch.where(spin[:, None] == 0, a, b), torch.where(spin[:, None] == 0, b, a)
            x, y = x % n, y % n
            v[k1] = sg * (s.h1[x, y] + (same[x, y] * o).sum(1) + (kk[x, y] * u).sum(1))
            k2 = nh == 2
            a1, a2, b1, b2 = h1[k2], h2[k2], p1[k2], p2[k2]
            lo, hi = torch.minimum(a2, b2), torch.maximum(a2, b2)
            bl = below[k2]
            par = (_between(bl, a1[:, None], b1[:, None])[:, 0]
                   + _between(bl, a2[:, None], b2[:, None])[:, 0]
                   + ((a1 > lo) & (a1 < hi)).long() + ((b1 > lo) & (b1 < hi)).long())
            exch = ha[k2] != 1  # both on one spin
            a1, a2, b1, b2 = a1 % n, a2 % n, b1 % n, b2 % n
            w = flat[((a1 * n + b1) * n + a2) * n + b2]
            w = w - torch.where(exch, flat[((a1 * n + b2) * n + a2) * n + b1], 0.0)
            v[k2] = (1.0 - 2.0 * (par & 1).double()) * w
            vals.append(v)
    return torch.cat(rows), torch.cat(cols), torch.cat(vals)


def _ground(A, v):
    """Lowest eigenpair of the sparse A by Lanczos from v, every vector kept orthogonal."""
    steps = min(A.shape[0], 260)
    V = torch.zeros((steps, A.shape[0]), dtype=torch.float64, device=DEV)
    al, be = [], []
    w = v / v.norm()
    for k in range(steps):
        V[k] = w
        w = A @ w
        al.append(float(w @ V[k]))
        for _ in range(2):
            w = w - V[:k + 1].T @ (V[:k + 1] @ w)
        be.append(float(w.norm()))
        if be[-1] < 1e-13:
            break
        w = w / be[-1]
    m = len(al)
    e, u = np.linalg.eigh(np.diag(al) + np.diag(be[:m - 1], 1) + np.diag(be[:m - 1], -1))
    x = V[:m].T @ torch.tensor(u[:, 0].copy(), device=DEV)
    x = x / x.norm()
    return float(e[0]), x * torch.sign(x[x.abs().argmax()])


def exact(case, seed):
    kind = case["kind"]
    if kind in ("many", "loop") or case.get("system") == "hubbard":
        return None  # several systems; and selections among equal scores
    if kind in ("search", "pt2"):
        C = case.get("C", case["ndets"])
        if C * _n_exc(case["norb"], case["na"], case["nb"]) > 700_000_000:
            return None
        s = _system(case, seed)
        keys, num, den = _targets(s, C, case.get("eps", 0.0))
        if kind == "pt2":
            return float((num * num / den).sum()), None
        score = num / den
        top = torch.argsort(score.abs(), descending=True, stable=True)[:case["N"]]
        return None, score[torch.sort(top).values], None
    s = _selected(case, seed)
    r, c, v = _matrix(s)
    if kind == "hamiltonian":
        return None, None, v
    if kind == "spmv":
        return torch.zeros(len(s.c), dtype=torch.float64, device=DEV).index_add_(0, r, v * s.c[c])
    ptr = torch.zeros(len(s.c) + 1, dtype=torch.int64, device=DEV)
    ptr[1:] = torch.bincount(r, minlength=len(s.c)).cumsum(0)
    return _ground(torch.sparse_csr_tensor(ptr, c, v, size=(len(s.c), len(s.c))), s.c)
