"""The work that users of this framework have it do, as cases that can be timed.

A user's program hands an active space (h, Cholesky factors, electrons, 2 S_z)
to `Context.solve` or `Context.solve_batched`, or holds a matrix-product state
and asks for parts of the pass: H_eff applied to a vector, one Davidson solve,
the environments and the energy of an installed state, its reduced density
matrices and orbital entropies.  The sizes are those of this repository's
workloads: CAS(6,6) M=64 up to CAS(20,20) M=1024, batches of 8 to 14 orbitals,
odd orbital and electron numbers and 2 S_z != 0 as in its tests.

Inputs come from the seed alone: integrals of the distribution that every
workload here uses, and, where a state is installed, canonical blocks whose
sectors crowd around the mean occupation and whose sites are weakly mixing
isometries, as in a converged sweep.  `exact` recomputes a result in 64 bits
from the determinants of the sector, where these are few enough.
"""
from __future__ import annotations

import math

import numpy as np

from paper_2609_09990_gb300 import gbdmrg

QN = ((0, 0), (1, 0), (0, 1), (1, 1))   # electrons (alpha, beta) of the local states 0, a, b, ab
PRECISION = {"fp64": 0, "tf32": 1, "bf16": 2}


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # the smallest whole calculation (400 determinants, full bond, with
        # RDMs): what a user runs first, bound by launches and host work
        dict(name="solve cas6 fp64", kind="solve", n=6, ne=6, sz=0, M=64, sweeps=4, prec="fp64", refine=2,
             tol=1e-9, rdms=True),
        # an ordinary whole calculation in the mixed tiers from the seeded start
        dict(name="solve cas10 bf16", kind="solve", n=10, ne=10, sz=0, M=128, sweeps=2, prec="bf16", refine=0,
             tol=1e-6, rdms=False),
        # several small active spaces in one call (the batched workload's sizes)
        dict(name="batch 8 spaces bf16", kind="batch", n=8, spread=3, count=8, M=96, sweeps=1, prec="bf16",
             refine=0, tol=1e-6),
        # one H_eff product and its diagonal, FP64, small and odd: an open shell
        dict(name="heff cas9 sz1 fp64", kind="heff", n=9, ne=9, sz=1, M=72),
        # the same in the middle of the largest FP64 workload
        dict(name="heff cas16 fp64", kind="heff", n=16, ne=16, sz=0, M=512),
        # one two-site Davidson solve, FP64, at the centre of CAS(12,12)
        dict(name="davidson cas12 fp64", kind="davidson", n=12, ne=12, sz=0, M=256, prec="fp64", refine=0, tol=1e-5),
        # and in the mixed tiers, at the centre of the headline CAS(16,16)
        # and of the largest CAS(20,20) workload
        dict(name="davidson cas16 bf16", kind="davidson", n=16, ne=16, sz=0, M=512, prec="bf16", refine=0, tol=1e-5),
        dict(name="davidson cas20 bf16", kind="davidson", n=20, ne=20, sz=0, M=1024, prec="bf16", refine=0, tol=1e-4),
        # a stored state taken up again: every environment is built, then <H>
        dict(name="energy cas14 fp64", kind="energy", n=14, ne=14, sz=0, M=384),
        # what a converged state is wanted for: 1-/2-RDMs at full size,
        # orbital entropies for an ordering, the 3-RDM of a small space
        dict(name="rdms cas16", kind="rdms", n=16, ne=16, sz=0, M=512),
        dict(name="entropies cas13", kind="entropies", n=13, ne=11, sz=1, M=200),
        dict(name="rdm3 cas9", kind="rdm3", n=9, ne=9, sz=1, M=96),
    ]


def draw(rng):
    """One more case: the kinds above at sizes between the smallest and the largest of each."""
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["solve", "solve", "batch", "heff", "heff", "davidson", "davidson", "energy", "rdms",
                       "entropies", "rdm3"])
    if kind == "batch":
        return dict(kind=kind, n=rng.randint(7, 9), spread=rng.randint(1, 3), count=rng.randint(4, 10),
                    M=log(32, 128), sweeps=1, prec=rng.choice(["fp64", "bf16", "tf32"]), refine=0, tol=1e-6)
    if kind == "rdm3":
        n = rng.randint(5, 9)
        return dict(kind=kind, n=n, **_electrons(rng, n), M=log(24, 96))
    n = rng.randint(6, 10) if kind == "solve" else rng.randint(7, 16)
    c = dict(kind=kind, n=n, **_electrons(rng, n))
    c["M"] = log(32, 128) if kind == "solve" else log(40, {16: 512, 15: 448, 14: 384, 13: 320}.get(n, 256))
    if kind == "solve":
        # an FP64 solve at full bond also returns its RDMs
        c.update(sweeps=rng.randint(1, 2), prec=rng.choice(["fp64", "bf16", "tf32"]), refine=0, tol=1e-6, rdms=False)
    if kind == "davidson":
        c.update(prec=rng.choice(["fp64", "bf16", "tf32"]) if n <= 12 else "bf16", refine=0, tol=1e-5)
    return c


def _electrons(rng, n):
    """Near half filling, closed and open shells."""
    sz = rng.choice([0, 0, 1, -1, 2])
    ne = n + rng.choice([0, 0, -1, 1, -2])
    return dict(ne=ne + (ne + sz) % 2, sz=sz)


# ------------------------------------------------------------------ inputs
def _integrals(n, rng):
    """h: diagonal U[-2,0], off-diagonal N(0,0.05); 3 n Cholesky vectors N(0,0.1) exp(-|p-q|/3)."""
    h = np.triu(rng.normal(0.0, 0.05, (n, n)), 1)
    h = h + h.T + np.diag(rng.uniform(-2.0, 0.0, n))
    p = np.arange(n)
    L = np.triu(rng.normal(0.0, 0.1, (3 * n, n, n)) * np.exp(-np.abs(p[:, None] - p[None, :]) / 3.0))
    return h, L + np.transpose(np.triu(L, 1), (0, 2, 1))


def _bonds(n, na, nb, M):
    """Sector dimensions of every bond, {(N_alpha, N_beta): dim}: at most M states, crowded around the
    mean occupation as a decimation leaves them, each no larger than both neighbours support."""
    dims = []
    for k in range(n + 1):
        ex, wt = {}, {}
        for a in range(max(0, na - (n - k)), min(k, na) + 1):
            for b in range(max(0, nb - (n - k)), min(k, nb) + 1):
                m = min(math.comb(k, a) * math.comb(k, b), math.comb(n - k, na - a) * math.comb(n - k, nb - b))
                ex[a, b] = m
                r2 = (a - na * k / n) ** 2 + (b - nb * k / n) ** 2
                wt[a, b] = math.sqrt(m) * math.exp(-r2 / 2.6)
        d, left = {}, M
        if sum(ex.values()) <= M:
            d = dict(ex)
        else:   # proportional shares, capped by the multiplicity, what a cap frees handed on
            open_ = dict(wt)
            while left > 0 and open_:
                tot = sum(open_.values())
                add = {q: min(int(left * w / tot), ex[q] - d.get(q, 0)) for q, w in open_.items()}
                if not any(add.values()):
                    q = max(open_, key=open_.get)
                    add = {q: 1}
                for q, m in add.items():
                    d[q] = d.get(q, 0) + m
                left = M - sum(d.values())
                open_ = {q: w for q, w in open_.items() if d.get(q, 0) < ex[q]}
        dims.append({q: m for q, m in d.items() if m > 0})
    changed = True
    while changed:
        changed = False
        for k in list(range(1, n + 1)) + list(range(n - 1, -1, -1)):
            for q in list(dims[k]):
                for j, sg in ((k - 1, -1), (k + 1, 1)):
                    if not 0 <= j <= n:
                        continue
                    sup = sum(dims[j].get((q[0] + sg * s[0], q[1] + sg * s[1]), 0) for s in QN)
                    if dims[k].get(q, 0) > sup:
                        changed = True
                        dims[k][q] = sup
                if not dims[k].get(q, 1):
                    del dims[k][q]
    return [dict(sorted(d.items())) for d in dims]


def _isometry(rng, rows, cols):
    """rows x cols with orthonormal columns: each column mostly one row, weakly mixed with the others."""
    g = rng.normal(0.0, 0.25 / math.sqrt(rows), (rows, cols))
    g[rng.permutation(rows)[:cols], np.arange(cols)] += 1.0
    return np.linalg.qr(g)[0]


def _mps(n, na, nb, M, center, rng):
    """Blocks {(q_l, s): array} of every site: left-orthonormal before `center`, right-orthonormal after it,
    the normalised centre in between with weights that fall with the rank."""
    bonds = _bonds(n, na, nb, M)
    sites = []
    for i in range(n):
        bl, br, site = bonds[i], bonds[i + 1], {}
        if i < center:
            for r in br:
                parts = [(q, s) for s in range(4) for q in [(r[0] - QN[s][0], r[1] - QN[s][1])] if q in bl]
                u, at = _isometry(rng, sum(bl[q] for q, _ in parts), br[r]), 0
                for q, s in parts:
                    site[q, s] = u[at:at + bl[q]]
                    at += bl[q]
        else:
            for q in bl:
                parts = [(r, s) for s in range(4) for r in [(q[0] + QN[s][0], q[1] + QN[s][1])] if r in br]
                if i == center:
                    for r, s in parts:
                        fall = np.exp(-4.0 * (np.arange(bl[q])[:, None] / bl[q] + np.arange(br[r])[None, :] / br[r]))
                        site[q, s] = rng.normal(0.0, 1.0, fall.shape) * fall
                else:
                    v, at = _isometry(rng, sum(br[r] for r, _ in parts), bl[q]).T, 0
                    for r, s in parts:
                        site[q, s] = v[:, at:at + br[r]]
                        at += br[r]
        if i == center:
            norm = math.sqrt(sum(float((b * b).sum()) for b in site.values()))
            site = {key: b / norm for key, b in site.items()}
        sites.append(site)
    return bonds, sites


def _packed(bonds, sites):
    """The exchange format of `Context.set_mps`: counts, sector triples and blocks, back to back."""
    tri = [x for d in bonds for q, m in d.items() for x in (q[0], q[1], m)]
    blocks = [sites[i][q, s].ravel() for i in range(len(sites)) for q in bonds[i] for s in range(4)
              if (q, s) in sites[i]]
    return np.array([len(d) for d in bonds], np.int32), np.array(tri, np.int32), np.concatenate(blocks)


def _center(c):
    return 0 if c["kind"] == "energy" else c["n"] // 2 - 1


def _inputs(case, seed):
    """What the seed alone decides: integrals, the installed state, the vector."""
    rng = np.random.default_rng([seed, 20 * case["n"] + case["M"]])
    if case["kind"] == "batch":
        probs = []
        for i in range(case["count"]):
            n = case["n"] + i % (case["spread"] + 1)
            h, chol = _integrals(n, rng)
            probs.append((h, chol, n - n % 2, 0))
        return dict(problems=probs)
    n = case["n"]
    h, chol = _integrals(n, rng)
    out = dict(h=h, chol=chol, start=int(rng.integers(1, 1 << 30)))
    if case["kind"] == "solve":
        return out
    na, nb = (case["ne"] + case["sz"]) // 2, (case["ne"] - case["sz"]) // 2
    k = _center(case)
    bonds, sites = _mps(n, na, nb, case["M"], k, rng)
    out.update(bonds=bonds, sites=sites, packed=_packed(bonds, sites))
    if case["kind"] == "heff":
        out["x"] = rng.normal(0.0, 1.0, _two_site(bonds, k)[0])
        out["x"] /= np.linalg.norm(out["x"])
    return out


def _two_site(bonds, k):
    """Length of the two-site vector of (k, k+1), and its middle sectors' (rows, columns)."""
    mid = {}
    for q, m in bonds[k].items():
        for s in QN:
            Q = (q[0] + s[0], q[1] + s[1])
            mid.setdefault(Q, [0, 0])[0] += m
    for Q in mid:
        mid[Q][1] = sum(bonds[k + 2].get((Q[0] + s[0], Q[1] + s[1]), 0) for s in QN)
    pairs = [(a, b) for a, b in mid.values() if b]
    return sum(a * b for a, b in pairs), pairs


# ------------------------------------------------------------------ one pass
def prepare(case, seed):
    d = _inputs(case, seed)
    state = dict(case=case, ctx=gbdmrg.Context(0))
    if case["kind"] == "batch":
        M, S = case["M"], case["sweeps"]
        state["problems"] = [(h, chol, ne, sz, [M] * S, [case["tol"]] * S,
                              dict(seed=1, precision=PRECISION[case["prec"]], fp64_refine=case["refine"]))
                             for h, chol, ne, sz in d["problems"]]
        return state
    state.update(h=d["h"], chol=d["chol"], start=d["start"])
    if case["kind"] == "solve":
        return state
    state["packed"] = d["packed"]
    state["ctx"].setup(d["h"], d["chol"], case["ne"], case["sz"], [case["M"]], [case.get("tol", 1e-8)],
                       seed=d["start"], precision=PRECISION[case.get("prec", "fp64")])
    if case["kind"] != "energy":
        state["ctx"].set_mps(*d["packed"], _center(case))
    if case["kind"] == "heff":
        state["x"] = d["x"]
    return state


def run(state):
    c, ctx = state["case"], state["ctx"]
    kind = c["kind"]
    if kind == "solve":
        r = ctx.solve(state["h"], state["chol"], c["ne"], c["sz"], [c["M"]] * c["sweeps"], [c["tol"]] * c["sweeps"],
                      rdms=c["rdms"], seed=state["start"], precision=PRECISION[c["prec"]], fp64_refine=c["refine"])
        out = dict(energy=r["energy"], sweep_energies=r["sweep_energies"])
        if c["rdms"]:
            out.update(rdm1=r["rdm1"], rdm2=r["rdm2"])
        return out
    if kind == "batch":
        _, rs = ctx.solve_batched(state["problems"])
        return dict(energy=np.array([r["energy"] for r in rs]),
                    sweep_energies=np.concatenate([r["sweep_energies"] for r in rs]))
    if kind == "heff":
        y, diag = ctx.apply_heff(_center(c), state["x"], want_diag=True)
        return dict(y=y, diag=diag)
    if kind == "davidson":
        # (Ritz value of the last tier, <x|H|x> in FP64, |r|): |r| and, in the
        # reduced tiers, the Ritz value only say where the iteration stopped
        ritz, energy, _ = ctx.probe_step(_center(c), PRECISION[c["prec"]], c["refine"], c["tol"])
        return dict(energy=energy, ritz=ritz) if c["prec"] == "fp64" else dict(energy=energy)
    if kind == "energy":
        ctx.set_mps(*state["packed"], _center(c))
        return dict(energy=ctx.final_energy())
    if kind == "rdms":
        g1, g2 = ctx.rdms(c["n"])
        return dict(rdm1=g1, rdm2=g2)
    if kind == "entropies":
        s1, mi = ctx.orbital_entropies(c["n"])
        return dict(s1=s1, mi=mi)
    return dict(rdm3=ctx.rdm3(c["n"]))


def work(case):
    """Bytes in and out, and the floating-point operations of the block products (estimated from the sector
    dimensions and the channels 2 + 4 n + 8 m^2 - 2 m of a bond whose smaller side has m sites)."""
    n, kind = case["n"], case["kind"]
    if kind == "batch":
        one = [work(dict(kind="solve", n=case["n"] + i % (case["spread"] + 1), ne=case["n"] + i % (case["spread"] + 1),
                         sz=(case["n"] + i % (case["spread"] + 1)) % 2, M=case["M"], sweeps=case["sweeps"]))
               for i in range(case["count"])]
        return {k: sum(w[k] for w in one) for k in ("bytes", "flops")}
    na, nb = (case["ne"] + case["sz"]) // 2, (case["ne"] - case["sz"]) // 2
    bonds = _bonds(n, na, nb, case["M"])

    def channels(k):
        m = min(k, n - k)
        return 2 + 4 * n + 8 * m * m - 2 * m

    def sigma(k):   # about a quarter of the 16 local elements of a channel are set
        return 0.5 * channels(k + 1) * sum(a * b * (a + b) for a, b in _two_site(bonds, k)[1])

    def sectors(k):
        return sum(m * m for m in bonds[k].values())

    def update(k):   # environments of bond k+1 from those of bond k, one of each conjugate pair
        return 0.5 * channels(k + 1) * sum(8.0 * m ** 3 for m in bonds[k + 1].values())

    mps = 8.0 * sum(m * sum(bonds[i + 1].get((q[0] + s[0], q[1] + s[1]), 0) for s in QN)
                    for i in range(n) for q, m in bonds[i].items())
    ints = 8.0 * (n * n + 3 * n ** 3)
    k = _center(case) if kind != "solve" else 0
    envs = 8.0 * (channels(k) * sectors(k) + channels(k + 2) * sectors(k + 2))
    if kind == "solve":   # about ten H_eff products a step
        steps = [j for j in range(n - 1)] * (2 * case["sweeps"])
        return dict(bytes=ints + mps, flops=sum(10 * sigma(j) + update(j) for j in steps))
    if kind == "heff":
        return dict(bytes=envs + 24.0 * _two_site(bonds, k)[0], flops=sigma(k))
    if kind == "davidson":   # about thirty products from an unconverged state
        return dict(bytes=envs + mps, flops=30 * sigma(k))
    if kind == "energy":
        return dict(bytes=mps + ints, flops=sum(update(j) for j in range(n - 1)))
    if kind == "rdm3":
        dets = math.comb(n, na) * math.comb(n, nb)
        return dict(bytes=mps + 8.0 * n ** 6, flops=2.0 * n ** 6 * dets / 6)
    strings = 8.0 * n * n if kind == "rdms" else 30.0 * n   # operator strings open at a bond
    return dict(bytes=mps + 8.0 * n ** 4, flops=sum(strings * 8.0 * m ** 3 for j in range(n) for m in bonds[j].values()))


# ------------------------------------------------------------------ 64-bit results from the determinants
class _Space:
    """Determinants of a sector as 2 n-bit integers (orbital p, spin s at bit 2 p + s; creators in bit order),
    and E_pq = sum_s a+_ps a_qs on vectors over them."""

    def __init__(self, n, na, nb):
        self.n = n
        d = np.arange(1 << (2 * n), dtype=np.int64)
        alpha = int("01" * n, 2)
        d = d[(np.bitwise_count(d & alpha) == na) & (np.bitwise_count(d & (alpha << 1)) == nb)]
        self.det = d
        self.pos = np.full(1 << (2 * n), -1, np.int64)
        self.pos[d] = np.arange(d.size)
        self.ops = [[self._op(2 * p + s, 2 * q + s) for s in (0, 1)] for p in range(n) for q in range(n)]

    def _op(self, p, q):
        d = self.det
        src = np.nonzero((d >> q & 1) & ((d >> p & 1) == 0) if p != q else d >> q & 1)[0]
        lo, hi = min(p, q), max(p, q)
        between = ((1 << hi) - 1) & ~((1 << (lo + 1)) - 1) if hi > lo else 0
        sign = 1.0 - 2.0 * (np.bitwise_count(d[src] & between) & 1)
        return src, self.pos[d[src] ^ (1 << p) ^ (1 << q)] if p != q else src, sign

    def apply(self, pq, v, out):
        for src, dst, sign in self.ops[pq]:
            out[..., dst] += sign * v[..., src]

    def all(self, v):
        D = np.zeros((self.n * self.n, v.size))
        for pq in range(self.n * self.n):
            self.apply(pq, v, D[pq])
        return D

    def hamiltonian(self, h, chol):
        n = self.n
        eri = np.einsum("Qpq,Qrs->pqrs", chol, chol)
        h1 = (h - 0.5 * np.einsum("prrq->pq", eri)).reshape(-1)
        eri = eri.reshape(n * n, n * n)

        def H(v):
            D = self.all(v)
            y = h1 @ D
            G = 0.5 * (eri @ D)
            for pq in range(n * n):
                self.apply(pq, G[pq], y)
            return y
        return H


class _State:
    """The installed state and the two-site basis of its centre, in determinants."""

    def __init__(self, case, d):
        n, k = case["n"], _center(case)
        self.bonds, self.k, self.n = d["bonds"], k, n
        self.space = _Space(n, (case["ne"] + case["sz"]) // 2, (case["ne"] - case["sz"]) // 2)
        left = {(0, 0): (np.zeros(1, np.int64), np.ones((1, 1)))}
        for i in range(k):
            new = {}
            for (q, s), b in d["sites"][i].items():
                new.setdefault((q[0] + QN[s][0], q[1] + QN[s][1]), []).append((left[q][0] | s << 2 * i, left[q][1] @ b))
            left = {r: (np.concatenate([x for x, _ in v]), np.concatenate([x for _, x in v])) for r, v in new.items()}
        right = {q: (np.zeros(1, np.int64), np.ones((1, 1))) for q in self.bonds[n]}
        for i in range(n - 1, k + 1, -1):
            new = {}
            for (q, s), b in d["sites"][i].items():
                r = (q[0] + QN[s][0], q[1] + QN[s][1])
                new.setdefault(q, []).append((right[r][0] | s << 2 * i, b @ right[r][1].T))
            right = {q: (np.concatenate([x for x, _ in v]), np.concatenate([x for _, x in v], axis=1).T)
                     for q, v in new.items()}
        self.blocks, at = [], 0
        for q in self.bonds[k]:
            for s1 in range(4):
                for s2 in range(4):
                    r = (q[0] + QN[s1][0] + QN[s2][0], q[1] + QN[s1][1] + QN[s2][1])
                    if r not in self.bonds[k + 2]:
                        continue
                    m, p = self.bonds[k][q], self.bonds[k + 2][r]
                    det = (left[q][0][:, None] | s1 << 2 * k | s2 << 2 * (k + 1)) | right[r][0][None, :]
                    self.blocks.append((at, m, p, self.space.pos[det], left[q][1], right[r][1]))
                    at += m * p
        self.size = at
        a, b = d["sites"][k], d["sites"][k + 1]
        x = np.zeros(self.size)
        at = 0
        for q in self.bonds[k]:
            for s1 in range(4):
                mid = (q[0] + QN[s1][0], q[1] + QN[s1][1])
                for s2 in range(4):
                    r = (mid[0] + QN[s2][0], mid[1] + QN[s2][1])
                    if r not in self.bonds[k + 2]:
                        continue
                    m, p = self.bonds[k][q], self.bonds[k + 2][r]
                    if (q, s1) in a and (mid, s2) in b:
                        x[at:at + m * p] = (a[q, s1] @ b[mid, s2]).ravel()
                    at += m * p
        self.x = x

    def to_det(self, x):
        v = np.zeros(self.space.det.size)
        for at, m, p, pos, L, R in self.blocks:
            v[pos] = L @ x[at:at + m * p].reshape(m, p) @ R.T
        return v

    def from_det(self, v):
        x = np.empty(self.size)
        for at, m, p, pos, L, R in self.blocks:
            x[at:at + m * p] = (L.T @ v[pos] @ R).ravel()
        return x


def _lowest(op, x, steps=220):
    """Lowest eigenvalue by Lanczos with full orthogonalisation, from x."""
    V, a, b = [x / np.linalg.norm(x)], [], []
    for j in range(min(steps, x.size)):
        w = op(V[j])
        a.append(float(w @ V[j]))
        for _ in range(2):
            B = np.array(V)
            w = w - B.T @ (B @ w)
        t, z = np.linalg.eigh(np.diag(a) + np.diag(b, 1) + np.diag(b, -1))
        beta = float(np.linalg.norm(w))
        if beta * abs(z[-1, 0]) < 1e-9 or beta < 1e-12:
            break
        b.append(beta)
        V.append(w / beta)
    return float(t[0])


def _densities(S, v):
    n, D = S.n, S.all(v)
    g1 = (D @ v).reshape(n, n)
    flip = np.arange(n * n).reshape(n, n).T.ravel()
    ee = (D[flip] @ D.T).reshape(n, n, n, n)   # <E_pq E_rs>
    g2 = ee.copy()
    for q in range(n):
        g2[:, q, q, :] -= g1
    return g1, g2, ee, D, flip


def _entropies(S, v):
    n = S.n
    occ = [(S.det >> 2 * i) & 3 for i in range(n)]
    s1 = np.zeros(n)
    for i in range(n):
        p = np.array([np.sum(v[occ[i] == s] ** 2) for s in range(4)])
        s1[i] = -np.sum(p[p > 1e-14] * np.log(p[p > 1e-14]))
    mi = np.zeros((n, n))
    for i in range(n):
        for j in range(i + 1, n):
            ni, nj = np.bitwise_count(occ[i]), np.bitwise_count(occ[j])
            before_i = np.bitwise_count(S.det & ((1 << 2 * i) - 1))
            before_j = np.bitwise_count(S.det & ((1 << 2 * j) - 1)) - ni
            sign = 1.0 - 2.0 * ((before_i * ni + before_j * nj) & 1)
            rest = S.det & ~((3 << 2 * i) | (3 << 2 * j))
            _, col = np.unique(rest, return_inverse=True)
            A = np.zeros((16, int(col.max()) + 1))
            A[occ[i] + 4 * occ[j], col] = sign * v
            w = np.linalg.eigvalsh(A @ A.T)
            w = w[w > 1e-14]
            mi[i, j] = mi[j, i] = max(s1[i] + s1[j] + np.sum(w * np.log(w)), 0.0)
    return s1, mi


def exact(case, seed):
    kind, n = case["kind"], case["n"]
    limit = {"solve": 7, "heff": 10, "davidson": 9, "energy": 10, "rdms": 10, "entropies": 10, "rdm3": 9}
    if n > limit.get(kind, 0):
        return None
    d = _inputs(case, seed)
    if kind == "solve":
        na, nb = (case["ne"] + case["sz"]) // 2, (case["ne"] - case["sz"]) // 2
        if case["prec"] != "fp64" or case["sweeps"] < 3 or _full(n, na, nb) > case["M"]:
            return None   # a truncated or unconverged state has no value of its own
        S = _Space(n, na, nb)
        H = S.hamiltonian(d["h"], d["chol"])
        m = np.array([H(e) for e in np.eye(S.det.size)])
        w, z = np.linalg.eigh(0.5 * (m + m.T))
        out = dict(energy=float(w[0]), sweep_energies=None)
        if case["rdms"]:
            g1, g2 = _densities(S, z[:, 0])[:2]
            out.update(rdm1=g1, rdm2=g2)
        return out
    T = _State(case, d)
    S = T.space
    H = S.hamiltonian(d["h"], d["chol"])
    if kind == "heff":
        diag = None
        if S.det.size * T.size <= 4e6:
            diag = np.empty(T.size)
            for i in range(T.size):
                e = np.zeros(T.size)
                e[i] = 1.0
                e = T.to_det(e)
                diag[i] = e @ H(e)
        return dict(y=T.from_det(H(T.to_det(d["x"]))), diag=diag)
    if kind == "davidson":
        low = _lowest(lambda x: T.from_det(H(T.to_det(x))), T.x)
        return dict(energy=low, ritz=low) if case["prec"] == "fp64" else dict(energy=low)
    v = T.to_det(T.x)
    v /= np.linalg.norm(v)
    if kind == "energy":
        return dict(energy=float(v @ H(v)))
    if kind == "entropies":
        s1, mi = _entropies(S, v)
        return dict(s1=s1, mi=mi)
    g1, g2, ee, D, flip = _densities(S, v)
    if kind == "rdms":
        return dict(rdm1=g1, rdm2=g2)
    g3 = np.empty((n, n, n, n, n, n))
    for rs in range(n * n):   # <E_pq E_rs E_tu>
        F = np.zeros_like(D)
        S.apply(rs, D, F)
        g3[:, :, rs // n, rs % n] = (D[flip] @ F.T).reshape(n, n, n, n)
    for i in range(n):
        g3[:, :, :, i, i, :] -= ee
        g3[:, i, i, :, :, :] -= g2
        g3[:, i, :, :, i, :] -= np.transpose(g2, (2, 0, 1, 3))
    return dict(rdm3=g3)


def _full(n, na, nb):
    """Largest bond dimension of the untruncated state."""
    return max(sum(min(math.comb(k, a) * math.comb(k, b), math.comb(n - k, na - a) * math.comb(n - k, nb - b))
                   for a in range(max(0, na - n + k), min(k, na) + 1) for b in range(max(0, nb - n + k), min(k, nb) + 1))
               for k in range(n + 1))
