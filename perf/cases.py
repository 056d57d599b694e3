"""Performance cases of the state-vector ADAPT-VQE path.

Each case is one call (or one short sequence of calls) that a user's program
makes through the package's public classes: H psi in both precisions, the
pool-gradient screen, energy + gradient evaluations of an ansatz on the dense
and on the sparse path, a whole ADAPT job, a batch of molecules, H psi over
the stored Hamiltonian, and the ranker's proposal pass.

Systems are the package's synthetic hydrogen-chain stand-ins: n orbitals at or
near half filling (12 to 32 qubits), integrals from `synth.integrals`.

listed()/draw(rng) give cases, prepare(case, seed) what a program holds before
the call, run(state) one pass, work(case) the bytes and operations no
implementation can do without, exact(case, seed) the result in 64 bits from
plain torch and numpy.
"""
from __future__ import annotations

import itertools
from math import comb

import numpy as np
import torch

import synth
import paper_2604_01176_gb300 as hy

DTYPES = {"f64": torch.float64, "f32": torch.float32}
SIZES = {"f64": 8, "f32": 4}


# ---------------------------------------------------------------------------
# cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # the smallest system of the tests and the smoke run: one H psi, all
        # launch latency
        dict(name="hpsi_f64_12q", kind="hpsi", n=6, na=3, nb=3, dtype="f64"),
        # ordinary double-precision H psi: every dense FP64 evaluation
        dict(name="hpsi_f64_24q", kind="hpsi", n=12, na=6, nb=6, dtype="f64"),
        # float bulk of the mixed-precision mode, open shell: both string
        # counts ragged (1,716 x 1,287 rows and columns)
        dict(name="hpsi_f32_26q_open", kind="hpsi", n=13, na=7, nb=5, dtype="f32"),
        # the largest: the 32-qubit headline system's float H psi
        dict(name="hpsi_f32_32q", kind="hpsi", n=16, na=8, nb=8, dtype="f32"),
        # the ADAPT screen of the whole spin-adapted pool, double precision
        dict(name="screen_f64_24q", kind="screen", n=12, na=6, nb=6, dtype="f64", pool="sd"),
        # the screen of the qubit-excitation pool on a float state at 28 qubits
        dict(name="screen_f32_28q", kind="screen", n=14, na=7, nb=7, dtype="f32", pool="qeb"),
        # two ansatz lengths of a small dense ADAPT run, as its optimiser
        # evaluates them (energy and gradient at two points each)
        dict(name="evaluate_f64_20q", kind="evaluate", n=10, na=5, nb=5, dtype="f64",
             sparse=False, length=12),
        # the same on the sparse path at 28 qubits, a longer ansatz (supports of
        # thousands of determinants and up)
        dict(name="evaluate_sparse_28q", kind="evaluate", n=14, na=7, nb=7, dtype="f64",
             sparse=True, length=12),
        # a whole ADAPT job: 32 qubits, 10 iterations from Hartree-Fock
        dict(name="adapt_job_32q", kind="job", n=16, na=8, nb=8, iters=10),
        # many molecules of 8 to 12 orbitals at once: sigma, energies, screens
        dict(name="batch_f64_20mol", kind="batch", count=20, lo=8, hi=12, dtype="f64"),
        # H psi streamed from the explicitly stored Hamiltonian
        dict(name="explicit_f32_24q", kind="explicit", n=12, na=6, nb=6, dtype="f32"),
        # the learned ranker's pass over the pool: features, then the network
        dict(name="ranker_f64_24q", kind="ranker", n=12, na=6, nb=6, dtype="f64"),
    ]


def _filling(rng, n):
    """Electron counts at or near half filling (open and closed shells)."""
    na = min(n - 1, max(1, (n + 1) // 2 + rng.choice([-1, 0, 0, 1])))
    nb = min(n - 1, max(1, n // 2 + rng.choice([-1, 0, 0, 1])))
    return na, nb


def draw(rng):
    kind = rng.choice(["hpsi", "hpsi", "screen", "screen", "evaluate", "evaluate", "job", "batch",
                       "explicit", "ranker"])
    dtype = rng.choice(["f64", "f32"])
    if kind == "hpsi":
        n = rng.randint(6, 14 if dtype == "f64" else 15)
    elif kind == "screen":
        n = rng.randint(6, 14)
    elif kind == "explicit":
        n = rng.randint(8, 12)
    elif kind == "ranker":
        n = rng.randint(6, 13)
    elif kind == "job":
        n = rng.randint(10, 15)
    else:
        n = rng.randint(8, 14)
    na, nb = _filling(rng, n)
    if kind == "screen":
        return dict(kind=kind, n=n, na=na, nb=nb, dtype=dtype, pool=rng.choice(["sd", "qeb"]))
    if kind == "evaluate":
        sparse = n >= 11 or rng.random() < 0.5
        return dict(kind=kind, n=n, na=na, nb=nb, dtype=dtype, sparse=sparse,
                    length=rng.randint(4, 12 if sparse else 14))
    if kind == "job":
        return dict(kind=kind, n=n, na=na, nb=nb, iters=rng.randint(4, 9))
    if kind == "batch":
        lo = rng.randint(6, 10)
        return dict(kind=kind, count=rng.randint(3, 20), lo=lo, hi=rng.randint(lo, 12), dtype=dtype)
    return dict(kind=kind, n=n, na=na, nb=nb, dtype=dtype)


# ---------------------------------------------------------------------------
# what a program holds before the call
# ---------------------------------------------------------------------------
def _system(c, seed):
    h1, h2, ec = synth.integrals(c["n"], 1000 + seed)
    return h1, h2, ec


def _vector(n_det, dtype, seed):
    """A normalised dense state of seeded normal amplitudes."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    v = torch.randn(n_det, dtype=DTYPES[dtype], device="cuda", generator=g)
    return v / torch.linalg.vector_norm(v)


def _n_det(c):
    return comb(c["n"], c["na"]) * comb(c["n"], c["nb"])


def _pair(c, seed):
    """psi and a stand-in for H psi: a multiple of psi plus another vector."""
    psi = _vector(_n_det(c), c["dtype"], 3 * seed + 1)
    sigma = _vector(_n_det(c), c["dtype"], 3 * seed + 2)
    return psi, (sigma - 2.0 * psi)


def _ansatz(c, seed, size):
    """Seeded distinct pool operators and angles of an optimised ansatz's size,
    at two points a line search apart."""
    rng = np.random.default_rng(seed)
    ops = rng.choice(size, size=min(c["length"], size), replace=False).astype(np.int64)
    th = 0.15 * rng.standard_normal(len(ops))
    return ops, np.stack([th, th + 0.01 * rng.standard_normal(len(ops))])


def _molecules(c, seed):
    """The batch's systems, sizes lo..hi in turn, at half filling."""
    out = []
    for i in range(c["count"]):
        n = c["lo"] + i % (c["hi"] - c["lo"] + 1)
        na, nb = synth.half_filling(n)
        out.append((n, na, nb, 2000 + 100 * seed + i))
    return out


def prepare(case, seed):
    c = dict(case)
    kind = c["kind"]
    if kind == "batch":
        mols = _molecules(c, seed)
        hams = [hy.Hamiltonian(*synth.integrals(n, s), n, na, nb) for n, na, nb, s in mols]
        pools = [hy.Pool(h) for h in hams]
        batch = hy.Batch(hams)
        batch.set_pools(pools)
        psi = batch.pack([_vector(h.n_det, c["dtype"], 7 * seed + i) for i, h in enumerate(hams)],
                         DTYPES[c["dtype"]])
        return dict(kind=kind, hams=hams, pools=pools, batch=batch, psi=psi,
                    sigma=batch.empty(DTYPES[c["dtype"]]),
                    energies=torch.zeros(len(hams), dtype=torch.float64, device="cuda"),
                    g=torch.zeros(int(batch.pool_offsets[-1]), dtype=torch.float64, device="cuda"))
    h1, h2, ec = _system(c, seed)
    ham = hy.Hamiltonian(h1, h2, ec, c["n"], c["na"], c["nb"])
    s = dict(kind=kind, ham=ham)
    if kind == "hpsi":
        s["psi"] = _vector(ham.n_det, c["dtype"], 3 * seed + 1)
        s["out"] = torch.empty_like(s["psi"])
    elif kind == "explicit":
        s["psi"] = _vector(ham.n_det, c["dtype"], 3 * seed + 1)
        s["out"] = torch.empty_like(s["psi"])
        s["matrix"] = hy.ExplicitH(ham, DTYPES[c["dtype"]])
    elif kind == "screen":
        s["pool"] = hy.Pool(ham, c["pool"])
        s["psi"], s["sigma"] = _pair(c, seed)
        s["g"] = torch.empty(len(s["pool"]), dtype=torch.float64, device="cuda")
    elif kind == "ranker":
        s["pool"] = hy.Pool(ham)
        s["ranker"] = hy.Ranker(hidden=256, seed=7)
        s["psi"], s["sigma"] = _pair(c, seed)
    elif kind == "evaluate":
        pool = hy.Pool(ham)
        s.update(pool=pool, dtype=DTYPES[c["dtype"]])
        s["adapt"] = hy.Adapt(ham, pool, "f64" if c["dtype"] == "f64" else "mixed",
                              max_iter=c["length"], sparse=c["sparse"])
        s["ops"], s["thetas"] = _ansatz(c, seed, len(pool))
    elif kind == "job":
        pool = hy.Pool(ham)
        s.update(pool=pool, iters=c["iters"])
        s["adapt"] = hy.Adapt(ham, pool, "f64", max_iter=c["iters"], sparse=True)
    else:
        raise ValueError(f"unknown kind {kind}")
    return s


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def run(s):
    kind = s["kind"]
    if kind == "hpsi":
        return s["ham"].apply_h(s["psi"], out=s["out"])
    if kind == "explicit":
        return s["matrix"].apply(s["psi"], out=s["out"])
    if kind == "screen":
        return s["pool"].gradients(s["psi"], s["sigma"], out=s["g"])
    if kind == "ranker":
        feat = hy.ranker_features(s["ham"], s["pool"], s["psi"], sigma=s["sigma"])
        return {"features": feat, "scores": s["ranker"].predict(feat)}
    if kind == "batch":
        b = s["batch"]
        b.apply_h(s["psi"], s["sigma"], s["energies"])
        b.gradients(s["psi"], s["sigma"], out=s["g"])
        return {"sigma": s["sigma"], "energies": s["energies"], "gradients": s["g"]}
    if kind == "evaluate":
        ad, out = s["adapt"], []
        for length in (len(s["ops"]) - 1, len(s["ops"])):
            ad.set_ansatz(s["ops"][:length], s["thetas"][0, :length])
            for th in s["thetas"]:
                e, g = ad.evaluate(th[:length], s["dtype"])
                out.append({"energy": e, "gradient": g})
        return out
    ad = s["adapt"]
    ad.set_ansatz([], [])
    recs = ad.run(s["iters"])
    ops, th = ad.ansatz()
    return {"energies": np.array([r["energy"] for r in recs]), "ops": ops, "thetas": th}


# ---------------------------------------------------------------------------
# what one pass cannot do without
# ---------------------------------------------------------------------------
def _couplings(n, na, nb):
    """Nonzero elements of H per determinant row."""
    sa, sb = na * (n - na), nb * (n - nb)
    return 1 + sa + sb + comb(na, 2) * comb(n - na, 2) + comb(nb, 2) * comb(n - nb, 2) + sa * sb


def _screen_pairs(n, na, nb):
    """Connected determinant pairs over every constituent of the pool (the
    same set of excitations in both pools)."""
    Na, Nb = comb(n, na), comb(n, nb)
    va, vb = n - na, n - nb

    def pairs(k, r):
        return comb(n - 2 * r, k - r) if k >= r and n >= 2 * r else 0

    p = na * va * pairs(na, 1) * Nb + nb * vb * pairs(nb, 1) * Na
    p += comb(na, 2) * comb(va, 2) * pairs(na, 2) * Nb + comb(nb, 2) * comb(vb, 2) * pairs(nb, 2) * Na
    p += na * va * nb * vb * pairs(na, 1) * pairs(nb, 1)
    return p


def work(case):
    c, kind = case, case["kind"]
    if kind == "batch":
        b = f = 0.0
        for n, na, nb, _ in _molecules(c, 0):
            N = comb(n, na) * comb(n, nb)
            b += 4 * N * SIZES[c["dtype"]]            # psi, sigma of each of the two calls
            f += 2 * _couplings(n, na, nb) * N + 4 * _screen_pairs(n, na, nb)
        return {"bytes": b, "flops": f}
    n, na, nb = c["n"], c["na"], c["nb"]
    N, w = _n_det(c), _couplings(n, na, nb)
    if kind == "hpsi":
        return {"bytes": 2 * N * SIZES[c["dtype"]], "flops": 2 * w * N}
    if kind == "explicit":      # a 16-bit column and a value per stored entry
        return {"bytes": N * w * (2 + SIZES[c["dtype"]]) + 2 * N * SIZES[c["dtype"]],
                "flops": 2 * w * N}
    if kind == "screen":
        return {"bytes": 2 * N * SIZES[c["dtype"]], "flops": 4 * _screen_pairs(n, na, nb)}
    if kind == "ranker":        # both vectors' weights over pairs of orbitals of each spin
        return {"bytes": 2 * N * SIZES[c["dtype"]], "flops": 4.0 * N * (na + nb)}
    if kind == "evaluate":      # two points of two lengths: H psi and three rotated vectors each
        support = min(N, 2 ** c["length"]) if c["sparse"] else N
        rows = min(w, support)
        return {"bytes": 4 * 8 * support * SIZES[c["dtype"]], "flops": 8.0 * support * rows}
    support = [min(N, 2 ** i) for i in range(c["iters"])]
    return {"bytes": float(sum(16 * s * min(w, N) for s in support)),
            "flops": float(sum(2 * s * w for s in support))}


# ---------------------------------------------------------------------------
# the results in 64 bits, from plain torch and numpy
# ---------------------------------------------------------------------------
class _Strings:
    """Occupation strings of k electrons in n orbitals in ascending order and
    the action of a+_p a_q on them."""

    def __init__(self, n, k):
        self.n, self.k = n, k
        self.s = np.array(sorted(sum(1 << i for i in t) for t in itertools.combinations(range(n), k)),
                          dtype=np.int64)
        self.rank = {int(v): i for i, v in enumerate(self.s)}
        self.cache = {}

    def single(self, p, q, sign=True):
        """(domain, image, sign) of a+_p a_q (without the sign: +1)."""
        key = (p, q, sign)
        if key not in self.cache:
            s = self.s
            ok = (s >> q & 1) == 1
            if p != q:
                ok &= (s >> p & 1) == 0
            dom = np.flatnonzero(ok)
            t = s[dom]
            img = dom if p == q else np.searchsorted(s, t ^ (1 << p) ^ (1 << q))
            lo, hi = min(p, q), max(p, q)
            between = t >> (lo + 1) & ((1 << max(hi - lo - 1, 0)) - 1)
            par = np.zeros(len(t), dtype=np.int64)
            for i in range(self.n):
                par ^= between >> i & 1
            sg = 1.0 - 2.0 * par if sign else np.ones(len(t))
            self.cache[key] = tuple(torch.from_numpy(np.ascontiguousarray(x)).cuda()
                                    for x in (dom, img, sg))
        return self.cache[key]

    def double(self, a, i, b, j, sign=True):
        """(domain, image, sign) of (a+_a a_i)(a+_b a_j), four distinct orbitals."""
        d1, m1, s1 = self.single(b, j, sign)
        d2, m2, s2 = self.single(a, i, sign)
        at = torch.full((len(self.s),), -1, dtype=torch.int64, device="cuda")
        at[d2] = torch.arange(len(d2), device="cuda")
        k = at[m1]
        ok = k >= 0
        return d1[ok], m2[k[ok]], s1[ok] * s2[k[ok]]


class _Space:
    def __init__(self, n, na, nb):
        self.n, self.na, self.nb = n, na, nb
        self.a, self.b = _Strings(n, na), _Strings(n, nb)
        self.Na, self.Nb = len(self.a.s), len(self.b.s)

    def hpsi(self, h1, h2, ec, psi):
        """H psi from spin-summed single excitations: H = sum h'_pq E_pq +
        1/2 sum (pq|rs) E_pq E_rs, h'_ps = h_ps - 1/2 sum_r (pr|rs)."""
        n, nn = self.n, self.n ** 2
        x = psi.view(self.Na, self.Nb)
        D = torch.zeros((nn, self.Na, self.Nb), dtype=torch.float64, device="cuda")
        for p, q in itertools.product(range(n), repeat=2):
            self._add_single(D[p * n + q], x, p, q)
        hp = torch.from_numpy(h1 - 0.5 * np.einsum("prrs->ps", h2)).cuda().reshape(1, nn)
        V = torch.from_numpy(0.5 * h2.reshape(nn, nn)).cuda()
        D = D.view(nn, -1)
        out = ec * psi.clone()
        for c0 in range(0, D.shape[1], 1 << 20):
            blk = D[:, c0:c0 + (1 << 20)]
            out[c0:c0 + (1 << 20)] += (hp @ blk)[0]
            blk.copy_(V @ blk)
        D = D.view(nn, self.Na, self.Nb)
        o2 = out.view(self.Na, self.Nb)
        for p, q in itertools.product(range(n), repeat=2):
            self._add_single(o2, D[p * n + q], p, q)
        return out

    def _add_single(self, out, x, p, q):
        d, m, s = self.a.single(p, q)
        out.index_add_(0, m, x.index_select(0, d) * s[:, None])
        d, m, s = self.b.single(p, q)
        out.index_add_(1, m, x.index_select(1, d) * s[None, :])

    # -- pool: constituents as (alpha part, beta part), a part = list of (a, i) moves
    def pool(self, kind):
        n = self.n
        occ = (range(self.na), range(self.nb))
        ops = []

        def ok(sp, *moves):
            return all(i in occ[sp] and a >= len(occ[sp]) for a, i in moves)

        def same(sp, *moves):
            return (list(moves), []) if sp == 0 else ([], list(moves))

        if kind == "qeb":
            vir = (range(self.na, n), range(self.nb, n))
            for sp in (0, 1):
                ops += [[same(sp, (a, i))] for i in occ[sp] for a in vir[sp]]
            for sp in (0, 1):
                ops += [[same(sp, (a, i), (b, j))] for i, j in itertools.combinations(occ[sp], 2)
                        for a, b in itertools.combinations(vir[sp], 2)]
            ops += [[([(a, i)], [(b, j)])] for i in occ[0] for j in occ[1] for a in vir[0]
                    for b in vir[1]]
            return ops

        def push(cons):
            if cons:
                ops.append(cons)

        def opposite(a, i, b, j):
            return [([(a, i)], [(b, j)])] if ok(0, (a, i)) and ok(1, (b, j)) else []

        for i in range(n):
            for a in range(i + 1, n):
                push([same(sp, (a, i)) for sp in (0, 1) if ok(sp, (a, i))])
        for i, j in itertools.combinations(range(n), 2):
            for a, b in itertools.combinations(range(n), 2):
                push([same(sp, (a, i), (b, j)) for sp in (0, 1) if ok(sp, (a, i), (b, j))])
        for i, j in itertools.combinations_with_replacement(range(n), 2):
            for a, b in itertools.combinations_with_replacement(range(n), 2):
                c1, c2 = opposite(a, i, b, j), opposite(b, j, a, i)
                if i < j and a < b:
                    push(c1 + c2)
                    push(opposite(a, j, b, i) + opposite(b, i, a, j))
                elif i == j and a == b:
                    push(c1)
                else:
                    push(c1)
                    push(c2)
        return ops

    def _part(self, strings, moves, sign):
        if not moves:
            r = torch.arange(len(strings.s), device="cuda")
            return r, r, torch.ones(len(strings.s), dtype=torch.float64, device="cuda")
        if len(moves) == 1:
            return strings.single(*moves[0], sign)
        return strings.double(*moves[0], *moves[1], sign)

    def cons(self, con, sign):
        return self._part(self.a, con[0], sign), self._part(self.b, con[1], sign)

    def gradient(self, op, psi, sigma, sign=True):
        """2 <sigma|A psi>."""
        x, y = psi.view(self.Na, self.Nb), sigma.view(self.Na, self.Nb)
        g = torch.zeros((), dtype=torch.float64, device="cuda")
        for con in op:
            (da, ma, sa), (db, mb, sb) = self.cons(con, sign)

            def at(v, r, c):
                w = v.index_select(0, r) if con[0] else v
                return w.index_select(1, c) if con[1] else w

            t = at(y, ma, mb) * at(x, da, db) - at(y, da, db) * at(x, ma, mb)
            g += torch.einsum("ab,a,b->", t, sa, sb)
        return 2.0 * g

    def rotate(self, op, theta, psi, sign=True):
        """exp(theta A) psi in place, one constituent after another."""
        x = psi.view(self.Na, self.Nb)
        cs, sn = float(np.cos(theta)), float(np.sin(theta))
        for con in op:
            (da, ma, sa), (db, mb, sb) = self.cons(con, sign)
            sg = sn * sa[:, None] * sb[None, :]
            u, v = x[da[:, None], db[None, :]], x[ma[:, None], mb[None, :]]
            x[da[:, None], db[None, :]] = cs * u - sg * v
            x[ma[:, None], mb[None, :]] = cs * v + sg * u
        return psi


def _exact_evaluate(c, seed):
    sp = _Space(c["n"], c["na"], c["nb"])
    h1, h2, ec = _system(c, seed)
    pool = sp.pool("sd")
    ops, thetas = _ansatz(c, seed, len(pool))
    out = []
    for length in (len(ops) - 1, len(ops)):
        for th in thetas:
            psi = torch.zeros(_n_det(c), dtype=torch.float64, device="cuda")
            psi[0] = 1.0
            for k, t in zip(ops[:length], th):
                sp.rotate(pool[k], t, psi)
            lam = sp.hpsi(h1, h2, ec, psi)
            e = float(psi @ lam)
            g = np.zeros(length)
            for l in range(length - 1, -1, -1):
                g[l] = float(sp.gradient(pool[ops[l]], psi, lam))
                sp.rotate(pool[ops[l]], -th[l], psi)
                sp.rotate(pool[ops[l]], -th[l], lam)
            out.append({"energy": e, "gradient": g})
    return out


def exact(case, seed):
    c, kind = dict(case), case["kind"]
    if kind in ("job", "ranker") or c.get("n", 0) > 14:
        return None
    if kind == "evaluate":
        return _exact_evaluate(c, seed)
    if kind == "batch":
        parts, energies, grads = [], [], []
        for i, (n, na, nb, s) in enumerate(_molecules(c, seed)):
            sp = _Space(n, na, nb)
            psi = _vector(sp.Na * sp.Nb, c["dtype"], 7 * seed + i).double()
            sigma = sp.hpsi(*synth.integrals(n, s), psi)
            energies.append(float(psi @ sigma))
            grads += [sp.gradient(op, psi, sigma) for op in sp.pool("sd")]
            parts += [sigma, torch.zeros(-len(sigma) % 32, dtype=torch.float64, device="cuda")]
        return {"sigma": torch.cat(parts), "energies": np.array(energies),
                "gradients": torch.stack(grads)}
    sp = _Space(c["n"], c["na"], c["nb"])
    if kind in ("hpsi", "explicit"):
        psi = _vector(_n_det(c), c["dtype"], 3 * seed + 1).double()
        return sp.hpsi(*_system(c, seed), psi)
    psi, sigma = (v.double() for v in _pair(c, seed))
    return torch.stack([sp.gradient(op, psi, sigma, c["pool"] == "sd") for op in sp.pool(c["pool"])])
