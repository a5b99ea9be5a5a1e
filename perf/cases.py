"""The work a user of the exact-diagonalisation library has it do, as timed cases.

Kinds of case:

* ``product``  one Hamiltonian-vector product on a sector whose tables the
  program keeps (``matvec_blocked`` / ``matvec``): the inner operation of
  every Lanczos loop, in both vector layouts and both precisions, with and
  without spin exchange and pair hopping;
* ``phonon``   one product of the coupled electron-phonon sector
  (``eph_matvec``);
* ``ground``   one Lanczos ground state with its vector (``lanczos_ground``);
* ``chain``    one Matsubara Green's function of a known ground state
  (``gf_lanczos``: two 200-step chains and their continued fractions);
* ``solve``    one whole impurity solve from a model (``solve``).

Models follow the paper's protocol: random bath energies in [-2, 2],
hybridisations in [0.2, 0.6], impurity levels at the particle-hole point,
sectors at and next to half filling.  Vectors are uniform in [-1/2, 1/2), the
distribution of the Lanczos start vectors.
"""
import itertools
import math
from types import SimpleNamespace

import numpy as np
import torch

import paper_2105_06806_gb300 as ed

BETA, NMATS, GF_STEPS = 100.0, 512, 200
TOL = 1e-10  # Ritz residual of the ground states
DTYPE = {"fp64": torch.float64, "fp32": torch.float32}


# ------------------------------------------------------------------ the cases

def _product(name, norb, nbath, nup, ndw, precision, layout="blocked", exchange=False):
    return {"name": name, "kind": "product", "norb": norb, "nbath": nbath, "nup": nup, "ndw": ndw,
            "precision": precision, "layout": layout, "exchange": exchange}


def listed():
    return [
        # the smallest sector anyone solves (one orbital, seven bath levels): launch latency
        _product("product_norb1_ns8_fp64", 1, 7, 4, 4, "fp64"),
        # a small three-orbital sector off half filling, odd block widths
        _product("product_norb3_ns12_fp32", 3, 3, 6, 5, "fp32"),
        # one orbital with a long bath: a single wide block per spin
        _product("product_norb1_ns14_fp32", 1, 13, 7, 7, "fp32"),
        # a program that holds its vectors in the paper's sector order
        _product("product_norb2_ns14_sector_fp32", 2, 6, 5, 6, "fp32", layout="sector"),
        # the two-orbital benchmark sector in both precisions
        _product("product_norb2_ns16_fp32", 2, 7, 8, 8, "fp32"),
        _product("product_norb2_ns16_fp64", 2, 7, 8, 8, "fp64"),
        # the three-orbital benchmark sector, the largest that fits one GPU
        _product("product_norb3_ns18_fp32", 3, 5, 9, 9, "fp32"),
        # the rotation-invariant Kanamori interaction (spin exchange, pair hopping)
        _product("product_kanamori_norb3_ns15_fp32", 3, 4, 8, 7, "fp32", exchange=True),
        # the Holstein benchmark: one orbital, a phonon mode cut off at ten quanta
        {"name": "phonon_norb1_ns12_nph10_fp32", "kind": "phonon", "norb": 1, "nbath": 11,
         "nup": 6, "ndw": 6, "precision": "fp32", "nph": 10},
        # a two-orbital ground state with its vector in the default precision
        {"name": "ground_norb2_ns14_fp64", "kind": "ground", "norb": 2, "nbath": 6, "nup": 7,
         "ndw": 7, "precision": "fp64"},
        # the Green's function of one orbital in the default precision
        {"name": "chain_norb2_ns12_fp64", "kind": "chain", "norb": 2, "nbath": 5, "nup": 6,
         "ndw": 5, "precision": "fp64"},
        # a whole small solve with every G, as a DMFT loop or a server repeats it
        {"name": "solve_norb1_ns8_fp64", "kind": "solve", "norb": 1, "nbath": 7, "nup": 4,
         "ndw": 4, "precision": "fp64"},
    ]


def draw(rng):
    kind = rng.choice(["product"] * 6 + ["phonon", "ground", "chain", "solve"])

    def shape(lo, hi, norbs):
        ns, norb = rng.choice([(n, o) for n in range(lo, hi + 1) for o in norbs
                               if n % o == 0 and n // o >= 2])
        return ns, norb

    if kind == "product":
        ns, norb = shape(8, 18, (1, 2, 3, 4, 5))
        if ns == 18 and norb == 1:
            ns, norb = 17, 1
        half = ns // 2
        big = ns > 16
        c = _product("", norb, ns // norb - 1, half + rng.randint(-2, 0 if big else 2),
                     half + rng.randint(-2, 0 if big else 2),
                     "fp32" if big else rng.choice(["fp32", "fp32", "fp64"]),
                     "blocked" if big else rng.choice(["blocked", "blocked", "sector"]),
                     norb > 1 and rng.random() < 0.25)
    elif kind == "phonon":
        ns, norb = shape(8, 12, (1, 2, 3))
        c = {"kind": "phonon", "norb": norb, "nbath": ns // norb - 1,
             "nup": ns // 2 + rng.randint(-2, 1), "ndw": ns // 2 + rng.randint(-2, 1),
             "precision": rng.choice(["fp32", "fp64"]), "nph": rng.randint(1, 10)}
    elif kind == "ground":
        ns, norb = shape(8, 14, (1, 2, 3))
        c = {"kind": "ground", "norb": norb, "nbath": ns // norb - 1, "nup": (ns + 1) // 2,
             "ndw": ns // 2, "precision": "fp64"}
    elif kind == "chain":
        ns, norb = shape(8, 12, (1, 2, 3))
        c = {"kind": "chain", "norb": norb, "nbath": ns // norb - 1,
             "nup": ns // 2 + rng.randint(-1, 1), "ndw": ns // 2, "precision": "fp64"}
    else:
        ns, norb = shape(8, 10, (1, 2, 3))
        c = {"kind": "solve", "norb": norb, "nbath": ns // norb - 1,
             "nup": ns // 2 + rng.randint(-1, 1), "ndw": ns // 2, "precision": "fp64"}
    c["U"] = round(rng.uniform(1.0, 3.0), 3)
    return {k: v for k, v in c.items() if k != "name"}


# ------------------------------------------------------------------ inputs

def _model(case, seed):
    norb, nbath = case["norb"], case["nbath"]
    r = np.random.RandomState((seed * 7919 + 17) % (1 << 31))
    U = case.get("U", 2.0 if norb == 1 else 2.5)
    J = 0.0 if norb == 1 else 0.16 * U
    Ust = U - 2.0 * J
    e_d = -0.5 * (U + (norb - 1) * (2.0 * Ust - J))
    one = np.ones((2, 1, 1))
    x = J if case.get("exchange") else 0.0
    return SimpleNamespace(norb=norb, nbath=nbath, U=U, Ust=Ust, Jh=J, Jx=x, Jp=x,
                           e_imp=np.full((2, norb), e_d),
                           e_bath=one * r.uniform(-2.0, 2.0, (norb, nbath)),
                           v_bath=one * r.uniform(0.2, 0.6, (norb, nbath)))


def _dims(case):
    ns = case["norb"] * (case["nbath"] + 1)
    return math.comb(ns, case["nup"]), math.comb(ns, case["ndw"])


def _vector(n, dtype, seed):
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    return torch.rand(n, dtype=dtype, device="cuda", generator=g) - 0.5


def _phonon(case):
    return 0.5, 0.3, case["nph"]


def prepare(case, seed):
    st = {"case": case, "model": _model(case, seed)}
    kind, p = case["kind"], case["precision"]
    if kind == "solve":
        return st
    s = st["sector"] = ed.Sector(st["model"], case["nup"], case["ndw"])
    if kind == "product":
        v = _vector(s.dim, DTYPE[p], seed)
        if case["layout"] == "blocked":
            vb = torch.empty(s.blocked_dim, dtype=DTYPE[p], device="cuda")
            ed.permute(s, v, vb, True, p)
            v = vb
        st["v"], st["w"] = v, torch.zeros_like(v)
    elif kind == "phonon":
        w0, g, nph = _phonon(case)
        st["ph"] = ed.phonon(w0, [g] * case["norb"], nph)
        st["v"] = _vector(s.dim * (nph + 1), DTYPE[p], seed)
        st["w"] = torch.zeros_like(st["v"])
    elif kind == "ground":
        st["psi"] = torch.zeros(s.dim, dtype=DTYPE[p], device="cuda")
    elif kind == "chain":
        st["psi"] = torch.zeros(s.dim, dtype=DTYPE[p], device="cuda")
        st["e0"] = ed.lanczos_ground(s, p, psi=st["psi"], tol=TOL)["e0"]
    return st


def run(st):
    case = st["case"]
    kind, p = case["kind"], case["precision"]
    if kind == "product":
        f = ed.matvec_blocked if case["layout"] == "blocked" else ed.matvec
        f(st["sector"], st["v"], st["w"], p)
        return st["w"]
    if kind == "phonon":
        ed.eph_matvec(st["sector"], st["ph"], st["v"], st["w"], p)
        return st["w"]
    if kind == "ground":
        r = ed.lanczos_ground(st["sector"], p, psi=st["psi"], tol=TOL)
        return {"e0": r["e0"], "psi": st["psi"]}
    if kind == "chain":
        G, info = ed.gf_lanczos(st["sector"], st["psi"], st["e0"], 0, 0, p, GF_STEPS, BETA, NMATS)
        return {"G": G, "weights": [info["weight_particle"], info["weight_hole"]]}
    r, G = ed.solve(st["model"], case["nup"], case["ndw"], precision=p, nmats=NMATS, beta=BETA,
                    gf_steps=GF_STEPS, tol=TOL)
    return {"e0": r["e0"], "G": G}


# ------------------------------------------------------------------ work

#: Steps a ground state takes at these sizes (each reads one vector and writes one).
GROUND_STEPS = 90


def work(case):
    """One product reads v and writes w; per element it multiplies by the
    diagonal and by the elements of H of its row (a hop per bath level of
    which exactly one end is occupied: about half of them per spin)."""
    du, dd = _dims(case)
    size = 8 if case["precision"] == "fp64" else 4
    nb = case["norb"] * case["nbath"]
    ns = nb + case["norb"]
    hops = sum(nb * 2 * n * (ns - n) / (ns * (ns - 1)) for n in (case["nup"], case["ndw"]))
    dim, flops = du * dd, 3.0 + 2.0 * hops
    kind = case["kind"]
    if kind == "product":
        if case["exchange"]:
            flops += 2.0 * case["norb"] * (case["norb"] - 1) / 4.0
        return {"bytes": 2 * size * dim, "flops": flops * dim}
    if kind == "phonon":
        n = dim * (case["nph"] + 1)
        return {"bytes": 2 * size * n, "flops": (flops + 7.0) * n}
    if kind == "ground":
        k = GROUND_STEPS
        return {"bytes": k * 2 * size * dim, "flops": k * (flops + 8.0) * dim}
    # chains: every step one product and the recurrence on a sector next to this one
    chains = 2 if kind == "chain" else 2 * case["norb"] * (1 if case["nup"] == case["ndw"] else 2)
    steps = GF_STEPS * chains + (0 if kind == "chain" else GROUND_STEPS)
    return {"bytes": steps * 2 * size * dim, "flops": steps * (flops + 8.0) * dim}


# ------------------------------------------------------------------ 64-bit values

class _Spin:
    """Basis of one spin (ascending strings), its hops as partial maps and the
    block-major order of the library's padded layout, from the definitions."""

    def __init__(self, m, spin, n):
        norb, nbath = m.norb, m.nbath
        ns = norb * (nbath + 1)
        st = np.sort(np.fromiter((sum(1 << b for b in c)
                                  for c in itertools.combinations(range(ns), n)), dtype=np.int64,
                                 count=math.comb(ns, n)))
        self.dim, self.strings = len(st), st
        occ = (st[:, None] >> np.arange(ns)) & 1
        eps = np.concatenate([m.e_imp[spin], m.e_bath[spin].reshape(-1)])
        imp = occ[:, :norb].sum(1)
        self.occ = occ[:, :norb]
        self.e = occ @ eps + (m.Ust - m.Jh) * (imp * (imp - 1) // 2)
        self.hops = []  # (target, source, value) of every bath level
        for a in range(norb):
            for nu in range(nbath):
                b = norb + a * nbath + nu
                src = np.nonzero(occ[:, a] != occ[:, b])[0]
                dst = np.searchsorted(st, st[src] ^ (1 << a) ^ (1 << b))
                sg = 1 - 2 * (occ[src, a + 1:b].sum(1) & 1)
                self.hops.append((dst, src, sg * m.v_bath[spin, a, nu]))
        # c+ / c and the moves between impurity orbitals
        self.moves = {}
        for a in range(norb):
            for b in range(norb):
                if a != b:
                    src = np.nonzero(occ[:, b] & ~occ[:, a] & 1)[0]
                    dst = np.searchsorted(st, st[src] ^ (1 << a) ^ (1 << b))
                    lo, hi = min(a, b), max(a, b)
                    self.moves[a, b] = (dst, src, 1.0 - 2 * (occ[src, lo + 1:hi].sum(1) & 1))
        # block-major order: by the group occupations, then by the group strings
        groups = [((st >> a) & 1) | (((st >> (norb + a * nbath)) & ((1 << nbath) - 1)) << 1)
                  for a in range(norb)]
        pops = [occ[:, [a] + list(range(norb + a * nbath, norb + (a + 1) * nbath))].sum(1)
                for a in range(norb)]
        self.order = np.lexsort(groups[::-1] + pops[::-1])
        key = np.stack(pops, 1)[self.order]
        new = np.concatenate([[True], np.any(key[1:] != key[:-1], axis=1)])
        sizes = np.diff(np.concatenate([np.nonzero(new)[0], [self.dim]]))
        padded = (sizes + 3) // 4 * 4
        first = np.concatenate([[0], np.cumsum(padded)])
        self.stride = int(first[-1])
        block = np.cumsum(new) - 1
        self.column = first[block] + np.arange(self.dim) - np.concatenate([[0], np.cumsum(sizes)])[block]


def _t(x):
    return torch.as_tensor(x, device="cuda")


class _Exact:
    """H v of one sector in 64 bits with plain torch, v as [D_dw, D_up]."""

    def __init__(self, m, nup, ndw):
        self.m, self.nup, self.ndw = m, nup, ndw
        self.up, self.dw = _Spin(m, 0, nup), _Spin(m, 1, ndw)
        self.dim = self.up.dim * self.dw.dim
        no = m.norb
        self.wmat = np.full((no, no), m.Ust) + (m.U - m.Ust) * np.eye(no)

    def apply(self, v):
        up, dw, m = self.up, self.dw, self.m
        v = v.reshape(dw.dim, up.dim)
        w = torch.empty_like(v)
        oc, mid = _t(up.occ.astype(float)), _t(self.wmat)
        eu, e_d, od = _t(up.e), _t(dw.e), _t(dw.occ.astype(float))
        hops = [tuple(map(_t, h)) for h in up.hops]
        step = max(1, (1 << 27) // up.dim)
        for r in range(0, dw.dim, step):
            x = v[r:r + step]
            y = (eu[None, :] + e_d[r:r + step, None] + od[r:r + step] @ mid @ oc.T) * x
            for dst, src, val in hops:
                y.index_add_(1, dst, x.index_select(1, src) * val)
            w[r:r + step] = y
        cstep = max(1, (1 << 27) // dw.dim)
        for dst, src, val in [tuple(map(_t, h)) for h in dw.hops]:
            for c in range(0, up.dim, cstep):
                w[:, c:c + cstep].index_add_(0, dst, v[:, c:c + cstep].index_select(0, src)
                                             * val[:, None])
        for a, b in itertools.permutations(range(m.norb), 2):
            ud, us, uv = map(_t, up.moves[a, b])
            for k, j in (((b, a), m.Jx), ((a, b), m.Jp)):
                if j and len(us):
                    dd, ds, dv = map(_t, dw.moves[k])
                    part = v.index_select(0, ds).index_select(1, us) * (j * dv[:, None] * uv)
                    full = torch.zeros((len(ds), up.dim), dtype=v.dtype, device=v.device)
                    full.index_add_(1, ud, part)
                    w.index_add_(0, dd, full)
                    del part, full
        return w

    def blocked(self, w):
        out = torch.zeros((self.dw.dim, self.up.stride), dtype=w.dtype, device=w.device)
        col, order = _t(self.up.column), _t(self.up.order)
        rows = _t(self.dw.order)
        step = max(1, (1 << 27) // self.up.dim)
        for r in range(0, self.dw.dim, step):
            out[r:r + step, col] = w.index_select(0, rows[r:r + step]).index_select(1, order)
        return out.reshape(-1)

    def lanczos(self, v0, steps):
        """alpha, beta and the vectors of a fully re-orthogonalised chain."""
        n = min(steps, self.dim)
        Q = torch.zeros((n, self.dim), dtype=torch.float64, device="cuda")
        q = v0 / v0.norm()
        al, be = [], []
        for j in range(n):
            Q[j] = q
            w = self.apply(q).reshape(-1)
            al.append(float(w @ q))
            for _ in range(2):
                w = w - Q[:j + 1].T @ (Q[:j + 1] @ w)
            b = float(w.norm())
            if b < 1e-10 or j + 1 == n:
                break
            be.append(b)
            q = w / b
        return np.array(al), np.array(be[:len(al) - 1]), Q[:len(al)]

    def ground(self):
        g = torch.Generator(device="cuda").manual_seed(1)
        v = torch.rand(self.dim, dtype=torch.float64, device="cuda", generator=g) - 0.5
        for _ in range(2):
            al, be, Q = self.lanczos(v, 160)
            e, y = np.linalg.eigh(np.diag(al) + np.diag(be, 1) + np.diag(be, -1))
            v = Q.T @ _t(y[:, 0])
        return float(e[0]), (v / v.norm()).reshape(self.dw.dim, self.up.dim)

    def green(self, e0, psi, orb, spin):
        """G_{orb,spin}(i w_n) and the two weights from chains on the N+1 and N-1 sectors."""
        wn = (2 * np.arange(NMATS) + 1) * np.pi / BETA
        G, weights = np.zeros(NMATS, complex), []
        for sgn in (1, -1):
            n = [self.nup + (sgn if spin == 0 else 0), self.ndw + (sgn if spin == 1 else 0)]
            if min(n) < 0 or max(n) > self.m.norb * (self.m.nbath + 1):
                weights.append(0.0)
                continue
            t = _Exact(self.m, *n)
            here, there = ((self.up, t.up) if spin == 0 else (self.dw, t.dw))
            st = there.strings
            hit = np.nonzero(((st >> orb) & 1) == (sgn > 0))[0]
            src = np.searchsorted(here.strings, st[hit] ^ (1 << orb))
            par = sum((st[hit] >> k) & 1 for k in range(orb)) + np.zeros(len(hit), int)
            val = _t(1.0 - 2 * ((par + (self.nup if spin else 0)) & 1))
            phi = torch.zeros((t.dw.dim, t.up.dim), dtype=torch.float64, device="cuda")
            if spin == 0:
                phi[:, _t(hit)] = psi[:, _t(src)] * val
            else:
                phi[_t(hit)] = psi[_t(src)] * val[:, None]
            weight = float((phi * phi).sum())
            weights.append(weight)
            if weight == 0.0:
                continue
            al, be, _ = t.lanczos(phi.reshape(-1), GF_STEPS)
            z = e0 + sgn * 1j * wn
            f = z - al[-1]
            for a, b in zip(al[-2::-1], be[::-1]):
                f = z - a - b * b / f
            G += sgn * weight / f
        return G, weights


def exact(case, seed):
    m, kind = _model(case, seed), case["kind"]
    du, dd = _dims(case)
    if kind in ("chain", "solve", "ground") and du * dd > 2_000_000:
        return None  # a re-orthogonalised chain of this size takes too long
    x = _Exact(m, case["nup"], case["ndw"])
    if kind == "product":
        w = x.apply(_vector(du * dd, DTYPE[case["precision"]], seed).double())
        return x.blocked(w) if case["layout"] == "blocked" else w.reshape(-1)
    if kind == "phonon":
        w0, g, nph = _phonon(case)
        v = _vector(du * dd * (nph + 1), DTYPE[case["precision"]], seed).double()
        v = v.reshape(nph + 1, dd, du)
        w = torch.stack([x.apply(v[p]) for p in range(nph + 1)])
        ng = g * (_t(x.up.occ.sum(1).astype(float))[None, :]
                  + _t(x.dw.occ.sum(1).astype(float))[:, None])
        for p in range(nph + 1):
            w[p] += w0 * p * v[p]
            if p > 0:
                w[p] += ng * math.sqrt(p) * v[p - 1]
            if p < nph:
                w[p] += ng * math.sqrt(p + 1) * v[p + 1]
        return w.reshape(-1)
    e0, psi = x.ground()
    if kind == "ground":
        return {"e0": e0, "psi": None}  # the sign of the vector is the library's own
    if kind == "chain":
        G, weights = x.green(e0, psi, 0, 0)
        return {"G": G, "weights": weights}
    G = np.zeros((2, m.norb, NMATS), complex)
    for s in range(2):
        for o in range(m.norb):
            # the bath does not depend on the spin: with N_up = N_dw neither does G
            G[s, o] = G[0, o] if s and case["nup"] == case["ndw"] else x.green(e0, psi, o, s)[0]
    return {"e0": e0, "G": G}
