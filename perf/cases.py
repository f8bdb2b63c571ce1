"""The calls that a determinant-CI program makes, as timed cases.

A program that uses the library builds a context for an active space once
(``fci_init``), then spends its time in four calls: sigma vectors (its own
eigensolver or propagator around ``fci_sigma``), whole solves
(``fci_davidson``), densities of the converged vector (``fci_rdm1``,
``fci_rdm2``), and lock-step solves of many small active spaces
(``fci_batch_davidson``).  The active spaces run from a handful of orbitals,
where a call is a few launches, to CAS(16e,16o) with 1.7e8 determinants.

``exact`` is plain torch in FP64: H = sum k_kl E_kl + 1/2 sum (ij|kl) E_ij E_kl
applied through the one-electron operators E_kl, from the same inputs.
"""
import itertools
import math

import numpy as np
import torch

import paper_1707_04346_gb300 as fci


def listed():
    return [
        # a minimal active space inside an outer loop: launches and latency
        {"name": "sigma-f64-cas6", "kind": "sigma", "dtype": "f64", "norb": 6, "na": 3, "nb": 3, "splits": 3},
        # an open-shell space of odd size (462 x 462 strings, ragged tiles)
        {"name": "sigma-f64-11o-6a5b", "kind": "sigma", "dtype": "f64", "norb": 11, "na": 6, "nb": 5, "splits": 3},
        # the size most production CASCI runs use; the benchmark's workload
        {"name": "sigma-f64-cas14", "kind": "sigma", "dtype": "f64", "norb": 14, "na": 7, "nb": 7, "splits": 3},
        # the largest space whose FP64 solve is routine
        {"name": "sigma-f64-cas16", "kind": "sigma", "dtype": "f64", "norb": 16, "na": 8, "nb": 8, "splits": 3},
        # FP32 sigma of a mixed-precision iteration: a small open-shell space, the
        # production size, the largest
        {"name": "sigma-f32-9o-5a4b", "kind": "sigma", "dtype": "f32", "norb": 9, "na": 5, "nb": 4, "splits": 3},
        {"name": "sigma-f32-cas14", "kind": "sigma", "dtype": "f32", "norb": 14, "na": 7, "nb": 7, "splits": 3},
        {"name": "sigma-f32-cas16", "kind": "sigma", "dtype": "f32", "norb": 16, "na": 8, "nb": 8, "splits": 3},
        # whole solves: energies and vectors of a small open-shell space in FP64; the
        # two lowest energies (the singlet-triplet gap) of a larger one in mixed precision
        {"name": "solve-f64-8o-5a4b", "kind": "solve", "norb": 8, "na": 5, "nb": 4, "nroots": 2, "mixed": False},
        {"name": "solve-mixed-cas12", "kind": "solve", "norb": 12, "na": 6, "nb": 6, "nroots": 2, "mixed": True},
        # the density step after a solve
        {"name": "rdm1-cas14", "kind": "rdm1", "dtype": "f64", "norb": 14, "na": 7, "nb": 7},
        {"name": "rdm2-cas12", "kind": "rdm2", "dtype": "f64", "norb": 12, "na": 6, "nb": 6},
        # many small active spaces of mixed size solved together (points of a surface)
        {"name": "batch-mixed-12", "kind": "batch", "ninst": 12, "largest": 10, "nroots": 2, "mixed": True},
    ]


def _space(rng, lo, hi):
    """An active space near half filling: norb in lo..hi, up to one electron off per spin."""
    norb = rng.randint(lo, hi)
    na = min(norb - 1, max(1, (norb + rng.randint(0, 1)) // 2 + rng.choice((0, 0, 0, -1, 1))))
    nb = min(norb - 1, max(1, norb // 2 + rng.choice((0, 0, 0, -1))))
    return norb, na, nb


def draw(rng):
    known = [{k: v for k, v in c.items() if k != "name"} for c in listed()]
    while True:
        case = _one(rng)
        if case not in known:
            return case


def _one(rng):
    kind = rng.choice(("sigma", "sigma", "sigma", "sigma", "solve", "rdm1", "rdm2", "batch"))
    if kind == "sigma":
        # the determinant count grows about fourteenfold per two orbitals, so a
        # uniform norb spreads it over its logarithm
        norb, na, nb = _space(rng, 5, 16)
        return {"kind": kind, "dtype": rng.choice(("f64", "f64", "f32")), "norb": norb, "na": na, "nb": nb,
                "splits": rng.choice((3, 3, 2))}
    if kind == "solve":
        norb, na, nb = _space(rng, 6, 12)
        mixed = rng.random() < 0.5
        if not mixed and na == nb:
            # with n_alpha = n_beta a triplet's largest coefficients come in pairs of
            # opposite sign, so the sign of its vector is open
            na += 1
        return {"kind": kind, "norb": norb, "na": na, "nb": nb, "nroots": rng.randint(2, 3), "mixed": mixed}
    if kind == "batch":
        return {"kind": kind, "ninst": rng.randint(3, 12), "largest": rng.choice((8, 9, 10)), "nroots": 2,
                "mixed": rng.random() < 0.7}
    norb, na, nb = _space(rng, 6, 14 if kind == "rdm1" else 13)
    return {"kind": kind, "dtype": rng.choice(("f64", "f64", "f32")), "norb": norb, "na": na, "nb": nb}


# ---- inputs ---------------------------------------------------------------------


def _integrals(norb, seed):
    """h1 and a positive semidefinite eri with the decay of a localised active space."""
    r = np.random.RandomState((int(seed) * 1000003 + norb) % (1 << 31))
    i = np.arange(norb)
    g = r.standard_normal((norb, norb))
    g = np.triu(g) + np.triu(g, 1).T
    h1 = g * np.exp(-np.abs(i[:, None] - i[None, :]) / 3.0) + np.diag(np.sort(r.uniform(-2.0, 1.0, norb)))
    rank = 40 if norb < 12 else 100
    raw = 0.3 * r.standard_normal((rank, norb, norb)) / (1.0 + np.arange(rank))[:, None, None]
    chol = (np.triu(raw) + np.transpose(np.triu(raw, 1), (0, 2, 1))).reshape(rank, norb * norb)
    eri = (chol.T @ chol).reshape(norb, norb, norb, norb)
    eri = 0.5 * (eri + eri.transpose(2, 3, 0, 1))
    return h1, eri


def _vector(case, seed):
    """A normalised CI vector: coefficients of either sign over several orders of magnitude."""
    n = math.comb(case["norb"], case["na"]) * math.comb(case["norb"], case["nb"])
    gen = torch.Generator(device="cuda").manual_seed(int(seed) + 77)
    c = torch.randn(n, dtype=torch.float64, device="cuda", generator=gen)
    c.mul_(torch.randn(n, dtype=torch.float64, device="cuda", generator=gen).exp_())
    c.div_(torch.linalg.vector_norm(c))
    return c.float() if case["dtype"] == "f32" else c


def _instances(case, seed):
    """Half-filled spaces of 6 orbitals up to the largest, one of that among them."""
    r = np.random.RandomState((int(seed) + 5) % (1 << 31))
    sizes = [case["largest"]] + [6 + (7 * i + 3) % (case["largest"] - 5) for i in range(1, case["ninst"])]
    return [(n, (n + 1) // 2, n // 2) + _integrals(n, r.randint(1 << 20)) for n in sizes]


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        opt = fci.default_options(precision=fci.FCI_PREC_MIXED if case["mixed"] else fci.FCI_PREC_FP64, max_iter=1000)
        return {"kind": kind, "batch": fci.fci_batch_init(_instances(case, seed), opt), "nroots": case["nroots"]}
    norb, na, nb = case["norb"], case["na"], case["nb"]
    h1, eri = _integrals(norb, seed)
    if kind == "solve":
        opt = fci.default_options(precision=fci.FCI_PREC_MIXED if case["mixed"] else fci.FCI_PREC_FP64, max_iter=1000)
        ctx = fci.fci_init(norb, na, nb, h1, eri, opt)
        vecs = None
        if not case["mixed"]:
            vecs = torch.empty((case["nroots"], ctx.ndet), dtype=torch.float64, device="cuda")
        return {"kind": kind, "ctx": ctx, "nroots": case["nroots"], "vecs": vecs}
    ctx = fci.fci_init(norb, na, nb, h1, eri, fci.default_options(f32_splits=case.get("splits", 3)))
    c = _vector(case, seed)
    return {"kind": kind, "ctx": ctx, "c": c, "out": torch.empty_like(c) if kind == "sigma" else None}


def run(state):
    kind = state["kind"]
    if kind == "sigma":
        return fci.fci_sigma(state["ctx"], state["c"], state["out"])
    if kind == "solve":
        e = fci.fci_davidson(state["ctx"], state["nroots"], 1e-10, state["vecs"])
        return {"energies": e} if state["vecs"] is None else {"energies": e, "vectors": state["vecs"]}
    if kind == "rdm1":
        return fci.fci_rdm1(state["ctx"], state["c"])
    if kind == "rdm2":
        return list(fci.fci_rdm2(state["ctx"], state["c"]))
    return fci.fci_batch_davidson(state["batch"], state["nroots"], 1e-10)


# ---- the work of a call -----------------------------------------------------------


def _counts(norb, na, nb):
    """Determinants, and multiply-adds per determinant of the sparse sum over Slater-Condon replacements."""
    def spin(ne):
        single = ne * (norb - ne)
        return ne + single, 1 + single + math.comb(ne, 2) * math.comb(norb - ne, 2)

    n = math.comb(norb, na) * math.comb(norb, nb)
    (sa, ta), (sb, tb) = spin(na), spin(nb)
    return n, sa, sb, ta + tb + sa * sb


def work(case):
    kind = case["kind"]
    if kind == "batch":
        total = {"bytes": 0.0, "flops": 0.0}
        for i in range(case["ninst"]):
            norb = case["largest"] if i == 0 else 6 + (7 * i + 3) % (case["largest"] - 5)
            n, _, _, macs = _counts(norb, (norb + 1) // 2, norb // 2)
            # at least a dozen new directions per root
            total["bytes"] += 12.0 * case["nroots"] * 8 * 4 * n
            total["flops"] += 12.0 * case["nroots"] * 2 * macs * n
        return total
    norb, na, nb = case["norb"], case["na"], case["nb"]
    n, sa, sb, macs = _counts(norb, na, nb)
    size = 4 if case.get("dtype") == "f32" else 8
    if kind == "sigma":
        return {"bytes": 2.0 * size * n + 8.0 * norb ** 4, "flops": 2.0 * macs * n}
    if kind == "solve":
        return {"bytes": 20.0 * case["nroots"] * 8 * 4 * n, "flops": 20.0 * case["nroots"] * 2 * macs * n}
    if kind == "rdm1":
        return {"bytes": 1.0 * size * n + 8.0 * norb ** 2, "flops": 1.0 * (sa + sb) * n}
    pairs = norb * norb
    return {"bytes": 1.0 * size * n + 8.0 * (pairs ** 2 + pairs), "flops": 1.0 * pairs * (pairs + 1) * n}


# ---- the same in plain FP64 --------------------------------------------------------


def _replacements(norb, ne, device):
    """For every (k, l): the string E_kl J (ascending bitmasks) and its sign, 0 where E_kl J = 0."""
    strings = sorted(sum(1 << p for p in occ) for occ in itertools.combinations(range(norb), ne))
    s = np.array(strings, dtype=np.int64)
    idx = np.zeros((norb, norb, len(s)), dtype=np.int64)
    sgn = np.zeros((norb, norb, len(s)))
    for k in range(norb):
        for l in range(norb):
            ok = (s >> l & 1 == 1) & ((s >> k & 1 == 0) | (k == l))
            t = (s & ~(1 << l)) | (1 << k)
            lo, hi = min(k, l), max(k, l)
            between = s & ((1 << hi) - 1) & ~((1 << (lo + 1)) - 1) if hi > lo else np.zeros_like(s)
            odd = np.zeros_like(s)
            for p in range(norb):
                odd ^= between >> p & 1
            idx[k, l] = np.where(ok, np.searchsorted(s, np.where(ok, t, s[0])), 0)
            sgn[k, l] = np.where(ok, 1.0 - 2.0 * odd, 0.0)
    return torch.from_numpy(idx).to(device), torch.from_numpy(sgn).to(device)


class _Plain:
    """H of one space through the operators E_kl, in FP64."""

    def __init__(self, norb, na, nb, h1, eri):
        self.norb, self.dev = norb, "cuda" if torch.cuda.is_available() else "cpu"
        self.ia, self.sa = _replacements(norb, na, self.dev)
        self.ib, self.sb = _replacements(norb, nb, self.dev)
        self.shape = (self.ia.shape[2], self.ib.shape[2])
        self.pairs = [(k, l) for k in range(norb) for l in range(k + 1)]
        w = np.array([[eri[k, l, m, n] for m, n in self.pairs] for k, l in self.pairs])
        self.w = torch.from_numpy(w).to(self.dev)
        k1 = h1 - 0.5 * np.einsum("kjjl->kl", eri)
        self.k1 = [float(k1[k, l]) for k, l in self.pairs]
        self.h1, self.eri = h1, eri
        self.small = max(self.shape) <= 300
        if self.small:  # few strings: the operators of one spin as dense matrices
            k1, eri = torch.from_numpy(k1).to(self.dev), torch.from_numpy(eri).to(self.dev)
            ea, eb = self.dense(self.ia, self.sa), self.dense(self.ib, self.sb)

            def one(e):
                return torch.einsum("kl,klxy->xy", k1, e) + 0.5 * torch.einsum(
                    "pxz,pzy->xy", e.flatten(0, 1), torch.einsum("ijkl,klxy->ijxy", eri, e).flatten(0, 1))

            self.ha, self.hb = one(ea), one(eb)
            self.pa = torch.stack([ea[k, l] + (ea[l, k] if k != l else 0.0) for k, l in self.pairs])
            pb = torch.stack([eb[k, l] + (eb[l, k] if k != l else 0.0) for k, l in self.pairs])
            self.gb = torch.einsum("pq,qxy->pxy", self.w, pb)

    def dense(self, idx, sgn):
        n, ns = self.norb, idx.shape[2]
        e = torch.zeros((n, n, ns, ns), dtype=torch.float64, device=self.dev)
        return e.scatter_add_(2, idx[:, :, None, :], sgn[:, :, None, :].clone())

    def apply(self, k, l, c, rows):
        """(E_kl c) on the given alpha rows."""
        out = c[self.ia[l, k][rows]] * self.sa[l, k][rows][:, None]
        return out.add_(c[rows][:, self.ib[l, k]] * self.sb[l, k][None, :])

    def sigma(self, c):
        c = c.reshape(self.shape)
        if self.small:
            return (self.ha @ c + c @ self.hb.T + (self.pa @ c @ self.gb.transpose(1, 2)).sum(0)).reshape(-1)
        out = torch.zeros_like(c)
        step = max(1, int(4e9 / (8.0 * len(self.pairs) * self.shape[1])))
        for r0 in range(0, self.shape[0], step):
            rows = torch.arange(r0, min(self.shape[0], r0 + step), device=self.dev)
            d = torch.empty((len(self.pairs), len(rows), self.shape[1]), dtype=torch.float64, device=self.dev)
            for p, (k, l) in enumerate(self.pairs):
                d[p] = self.apply(k, l, c, rows)
                if k != l:
                    d[p] += self.apply(l, k, c, rows)
            f = (0.5 * self.w @ d.reshape(len(self.pairs), -1)).reshape(d.shape)
            del d
            for p, (k, l) in enumerate(self.pairs):
                f[p] += self.k1[p] * c[rows]
                for i, j in ((k, l), (l, k)) if k != l else ((k, l),):
                    out.index_add_(0, self.ia[i, j][rows], f[p] * self.sa[i, j][rows][:, None])
                    out[rows] += f[p][:, self.ib[j, i]] * self.sb[j, i][None, :]
            del f
        return out.reshape(-1)

    def diagonal(self):
        n = self.norb
        h = torch.from_numpy(np.diag(self.h1).copy()).to(self.dev)
        jj = torch.from_numpy(np.einsum("iijj->ij", self.eri).copy()).to(self.dev)
        kk = torch.from_numpy(np.einsum("ijji->ij", self.eri).copy()).to(self.dev)
        na = torch.stack([self.sa[p, p] for p in range(n)], 1)
        nb = torch.stack([self.sb[p, p] for p in range(n)], 1)

        def one(x):
            return x @ h + 0.5 * ((x @ (jj - kk)) * x).sum(1)

        return (one(na)[:, None] + one(nb)[None, :] + na @ jj @ nb.T).reshape(-1)

    def lowest(self, nroots):
        """Lowest roots by block Davidson to residuals of 1e-9."""
        diag = self.diagonal()
        n = diag.numel()
        start = torch.argsort(diag)[: nroots + 2]
        b = torch.zeros((len(start), n), dtype=torch.float64, device=self.dev)
        b[torch.arange(len(start), device=self.dev), start] = 1.0
        s = torch.stack([self.sigma(x) for x in b])
        for _ in range(600):
            e, v = torch.linalg.eigh(b @ s.T)
            x, hx = v[:, : nroots + 2].T @ b, v[:, : nroots + 2].T @ s
            r = hx[:nroots] - e[:nroots, None] * x[:nroots]
            if float(torch.linalg.vector_norm(r, dim=1).max()) < 1e-9:
                return e[:nroots], x[:nroots]
            if len(b) > 40:
                b, s = x, hx
            for k in range(nroots):
                t = r[k] / (diag - e[k]).abs().clamp_min(1e-4)
                for _ in range(2):
                    t = t - b.T @ (b @ t)
                norm = torch.linalg.vector_norm(t)
                if float(norm) > 1e-14:
                    t = t / norm
                    t = t - b.T @ (b @ t)
                    t = t / torch.linalg.vector_norm(t)
                    b, s = torch.cat([b, t[None]]), torch.cat([s, self.sigma(t)[None]])
        return None

    def densities(self, c):
        """gamma_pq = <c|E_pq|c> and Gamma_pqrs = <c|E_pq E_rs|c>."""
        n = self.norb
        c = c.reshape(self.shape)
        rows = torch.arange(self.shape[0], device=self.dev)
        g1 = torch.zeros((n, n), dtype=torch.float64, device=self.dev)
        g2 = torch.zeros((n * n, n * n), dtype=torch.float64, device=self.dev)
        step = max(1, int(4e9 / (8.0 * n * n * self.shape[1])))
        for r0 in range(0, self.shape[0], step):
            at = rows[r0: r0 + step]
            d = torch.stack([self.apply(r, s, c, at).reshape(-1) for r in range(n) for s in range(n)])
            g1 += (d @ c[at].reshape(-1)).reshape(n, n)
            g2 += d @ d.T
        # row (q, p) against row (r, s)
        return g1, g2.reshape(n, n, n, n).transpose(0, 1).contiguous()


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        found = []
        for inst in _instances(case, seed):
            got = _Plain(*inst).lowest(case["nroots"])
            if got is None:
                return None
            found.append(got[0].cpu().numpy())
        return np.array(found)
    norb, na, nb = case["norb"], case["na"], case["nb"]
    h1, eri = _integrals(norb, seed)
    plain = _Plain(norb, na, nb, h1, eri)
    if kind == "solve":
        got = plain.lowest(case["nroots"])
        if got is None:
            return None
        e, x = got
        if case["mixed"]:
            return {"energies": e.cpu().numpy()}
        top = x.gather(1, x.abs().argmax(1)[:, None])
        return {"energies": e.cpu().numpy(), "vectors": x * torch.sign(top)}
    c = _vector(case, seed).double()
    if kind == "sigma":
        return plain.sigma(c)
    g1, g2 = plain.densities(c)
    return g1.cpu().numpy() if kind == "rdm1" else [g1.cpu().numpy(), g2.cpu().numpy()]
