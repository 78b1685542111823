"""The calls whose time counts: what a user of the MBE(3)-OSV-MP2 library has it do.

listed() names the cases, draw() gives more of the same ranges, prepare() makes what a program
holds before the call (inputs on the GPU and a Context), run() makes one pass through the public
entry points, work() counts what a pass cannot do without and exact() gives the outputs from plain
torch in 64 bits, without the library.

Systems are synthetic boxes (constant density, 20 orbitals per (10 A)^3) or chains (1.5 A) of
localized orbitals, with B[i,a,P] = 0.1 exp(-|r_i - r_a| / lam) z; z is a normal draw (B stored by
the caller) or the library's counter-based draw (B regenerated on the device from a seed).  The
geometry belongs to the case (so its clusters are always the same ones), the energies, z and mixing
rotations to the seed.
"""
import math

import numpy as np
import torch

import paper_2603_16575_gb300 as pkg

DEV = "cuda:0" if torch.cuda.is_available() else "cpu"
F64 = torch.float64


# ---------------------------------------------------------------- the cases
def _case(kind, n_occ, n_vir=0, n_aux=0, prec="fp64", lam=1.0, r2=8.0, r3=6.0, l_osv=1e-4, stored=False,
          chain=False, method="exact"):
    return dict(kind=kind, n_occ=n_occ, n_vir=n_vir, n_aux=n_aux, prec=prec, lam=lam, r2=r2, r3=r3, l_osv=l_osv,
                stored=stored, chain=chain, method=method)


def listed():
    return [
        # a few orbitals, the size of a first try or of a unit test: latency and launches
        dict(_case("energy", 6, 40, 96, lam=1.5, r2=3.5, r3=3.0), name="energy_n6_fp64"),
        # a small molecule from RI integrals that the caller stores, reference precision
        dict(_case("energy", 32, 160, 600, stored=True), name="energy_n32_fp64"),
        # the same size in the fast form: one step of a scan or of dynamics
        dict(_case("energy", 32, 160, 600, prec="mixed"), name="energy_n32_mixed"),
        # a middle-sized molecule in reference precision, B regenerated; odd numbers of virtuals
        dict(_case("energy", 48, 243, 901), name="energy_n48_fp64"),
        # production size in the fast form: thousands of uneven fragments
        dict(_case("energy", 128, 640, 2400, prec="mixed"), name="energy_n128_mixed"),
        # clusters chosen by OSV overlap instead of by distance, with the weak pairs
        dict(_case("screened", 64, 320, 1200, prec="mixed"), name="screened_n64_mixed"),
        # a peptide-shaped chain with randomized OSVs
        dict(_case("energy", 100, 750, 2000, prec="mixed", chain=True, method="randomized"), name="chain_n100_rosv"),
        # energy and gradient through autograd, from a stored B
        dict(_case("grad", 64, 320, 1200, stored=True), name="grad_n64_fp64"),
        # the gradient with the OSVs relaxed
        dict(_case("relaxed", 24, 120, 450), name="relaxed_n24_fp64"),
        # every pair of one subsystem coupled, OSVs untruncated (the closed-form check of a set-up)
        dict(_case("solve", 10, 50, 200, lam=3.0, l_osv=0.0), name="solve_n10_untruncated"),
        # orbital localization ahead of all this
        dict(_case("localize", 128), name="localize_n128"),
        # OSVs of a large virtual space and the pair classes, as a first look at a system's cost
        dict(_case("osv", 24, 760, 3001), name="osv_v760_fp64"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["energy", "energy", "energy", "energy_mixed", "energy_mixed", "energy_mixed", "chain",
                       "screened", "grad", "relaxed", "solve", "localize", "osv"])
    per = rng.uniform(4.0, 7.0)        # virtuals per orbital
    aux = rng.uniform(3.2, 4.2)        # auxiliaries per virtual
    if kind in ("energy", "energy_mixed"):
        mixed = kind == "energy_mixed"
        n = _log(rng, 6, 120 if mixed else 48)
        v = max(24, int(n * per))
        return _case("energy", n, v, int(v * aux), prec="mixed" if mixed else "fp64", stored=rng.random() < 0.4)
    if kind == "chain":
        n = _log(rng, 24, 110)
        v = int(n * rng.uniform(7.4, 7.6))
        return _case("energy", n, v, int(v * 2.7), prec="mixed", chain=True, method="randomized")
    if kind == "screened":
        n = _log(rng, 16, 64)
        v = int(n * 5.0)
        return _case("screened", n, v, int(v * aux), prec=rng.choice(["mixed", "mixed", "fp64"]) if n < 32 else "mixed")
    if kind in ("grad", "relaxed"):
        n = _log(rng, 6, 50 if kind == "grad" else 28)
        v = max(24, int(n * 5.0))
        return _case(kind, n, v, int(v * aux), stored=rng.random() < 0.5)
    if kind == "solve":
        n = rng.randint(3, 10)
        v = rng.randint(20, 50)
        return _case("solve", n, v, int(v * aux), lam=3.0, l_osv=rng.choice([0.0, 0.0, 1e-4]))
    if kind == "localize":
        return _case("localize", _log(rng, 12, 140))
    return _case("osv", rng.randint(8, 24), rng.randint(200, 740), rng.randint(800, 3000))


# ---------------------------------------------------------------- inputs
def _geometry(case):
    n, v = case["n_occ"], case["n_vir"]
    g = np.random.default_rng(1000 * n + v)
    if case["chain"]:
        r = np.zeros((n, 3))
        r[:, 0] = 1.5 * np.arange(n)
        rv = r[np.arange(v) % n] + 0.7 * g.standard_normal((v, 3))
    else:
        edge = 10.0 * (n / 20.0) ** (1.0 / 3.0)
        r = edge * g.random((n, 3))
        rv = edge * g.random((v, 3))
    return r, rv


def _dist(a, b):
    d = a[:, None, :] - b[None, :, :]
    return np.sqrt(np.sum(d * d, axis=-1))


def _inputs(case, seed):
    r, rv = _geometry(case)
    n, v = case["n_occ"], case["n_vir"]
    g = np.random.default_rng(seed)
    f = 1e-2 * np.exp(-_dist(r, r) / 2.0)
    np.fill_diagonal(f, -1.5 + 1.2 * g.random(n))
    e = 0.1 + 4.9 * g.random(v)
    env = 0.1 * np.exp(-_dist(r, rv) / case["lam"])
    s = {"r": r, "f": torch.tensor(f, device=DEV), "e": torch.tensor(e, device=DEV),
         "env": torch.tensor(env, device=DEV), "seed": int(seed)}
    if case["stored"]:
        gen = torch.Generator(device=DEV).manual_seed(int(seed))
        s["B"] = torch.randn((n, v, case["n_aux"]), dtype=F64, device=DEV, generator=gen) * s["env"][:, :, None]
    return s


def _orbitals(case, seed):
    """Delocalized orthonormal orbitals: one localized orbital per atom (4 AOs each, tails on its
    neighbours), mixed by a random rotation."""
    n = case["n_occ"]
    r, _ = _geometry(case)
    g = np.random.default_rng(seed)
    at = np.repeat(np.arange(n), 4)
    w = 0.3 * np.exp(-_dist(r, r)[at] / 1.5)
    w[at[:, None] == np.arange(n)[None, :]] = 1.0
    loc, _ = np.linalg.qr(g.standard_normal((4 * n, n)) * w)
    rot, _ = np.linalg.qr(g.standard_normal((n, n)))
    return np.ascontiguousarray(loc @ rot), np.arange(0, 4 * n + 1, 4, dtype=np.int32)


def prepare(case, seed):
    if case["kind"] == "localize":
        C, ao = _orbitals(case, seed)
        return {"case": case, "ctx": pkg.Context(0), "C": torch.tensor(C, device=DEV), "ao": ao}
    s = _inputs(case, seed)
    s["case"] = case
    s["ctx"] = pkg.Context(0, osv_prec=case["prec"], osv_method=case["method"])
    if case["kind"] == "grad":
        s["fn"] = pkg.osvmp2.mbe3_energy_function()
        if "B" not in s:
            s["B"] = pkg.osvmp2.generate_B(case["n_occ"], case["n_vir"], case["n_aux"], s["seed"], s["env"])
        for k in ("B", "f", "e"):
            s[k].requires_grad_(True)
    return s


# ---------------------------------------------------------------- one pass
def _build(s):
    c = s["case"]
    if "B" in s:
        return s["ctx"].build_osv(s["f"], s["e"], c["l_osv"], B=s["B"], r_occ=s["r"])
    return s["ctx"].build_osv(s["f"], s["e"], c["l_osv"], env=s["env"], seed=s["seed"], r_occ=s["r"], n_aux=c["n_aux"])


def run(state):
    s, c, ctx = state, state["case"], state["ctx"]
    kind = c["kind"]
    if kind == "localize":
        U, L, sweeps = ctx.localize_pm(s["C"], s["ao"])
        return {"U": U, "L": L, "sweeps": sweeps}
    if kind == "grad":
        E = s["fn"].apply(ctx, s["B"], s["f"], s["e"], s["r"], c["r2"], c["r3"], c["prec"], c["l_osv"])
        dB, df, de = torch.autograd.grad(E, (s["B"], s["f"], s["e"]))
        return {"E": E, "dB": dB, "df": df, "de": de}
    n_osv = _build(s)
    if kind == "osv":
        s2b, cls, counts = ctx.pair_screening()
        return {"n_osv": n_osv, "s2b": s2b, "cls": cls, "counts": list(counts)}
    if kind == "solve":
        E, pe, _ = ctx.solve(range(c["n_occ"]), c["prec"])
        return {"n_osv": n_osv, "E": E, "pairs": pe}
    if kind == "relaxed":
        E, dB, df, de, _, gap = ctx.energy_grad_relaxed(c["r2"], c["r3"])
        return {"n_osv": n_osv, "E": E, "dB": dB, "df": df, "de": de, "gap": gap}
    out = {"n_osv": n_osv}
    if kind == "screened":
        out["E"], out["E_weak"], _ = ctx.mbe3_energy_screened(c["prec"])
        out["pair_e"] = _pair_table(c["n_occ"], *ctx.fragment_results(), *ctx.weak_results())
    else:
        out["E"], _ = ctx.mbe3_energy(c["r2"], c["r3"], c["prec"])
        out["orbs"], out["weights"], out["frag_e"] = ctx.fragment_results()
    return out


def _pair_table(n, orbs, weights, e, weak, weak_e):
    """Energies by orbital pair, as a program tabulates them: one-orbital clusters on the diagonal,
    pair clusters above it, weak pairs below it, and the triples' number and weighted sum last."""
    t = np.zeros((n + 1, n))
    one, two = orbs[:, 1] < 0, (orbs[:, 1] >= 0) & (orbs[:, 2] < 0)
    t[orbs[one, 0], orbs[one, 0]] = e[one]
    t[orbs[two, 0], orbs[two, 1]] = e[two]
    t[weak[:, 1], weak[:, 0]] = weak_e
    t[n, 0], t[n, 1] = np.sum(~one & ~two), np.sum((weights * e)[~one & ~two])
    return t


# ---------------------------------------------------------------- what a pass cannot do without
def work(case):
    n, v, x = case["n_occ"], case["n_vir"], case["n_aux"]
    if case["kind"] == "localize":   # ~4 sweeps of n^2 / 2 rotations over n atoms
        return {"bytes": 8.0 * (4 * n * n + n * n), "flops": 4 * 0.5 * n * n * (10.0 * n * n + 4 * n)}
    r, rv = _geometry(case)
    # an OSV count per orbital: the virtuals within the reach of the envelope at the 1e-4 cut
    near = (_dist(r, rv) < 4.6 * case["lam"]).sum(axis=1).clip(4) if case["l_osv"] > 0 else np.full(n, v)
    k = np.minimum(near, v).astype(float)
    byt = 8.0 * ((n * v * x if case["stored"] else n * v) + n * n + v + 3 * n)
    fl = n * (1.0 * v * v * x + (4.0 / 3.0) * v ** 3)
    if case["kind"] == "osv":
        return {"bytes": byt + 12.0 * n * n, "flops": fl + sum(2.0 * v * k[i] * k[j] for i in range(n) for j in range(i))}
    d = _dist(r, r)
    if case["kind"] == "solve":
        pairs, frags = [(i, j) for i in range(n) for j in range(i, n)], [tuple(range(n))]
    else:
        c2, c3 = (5.5, 4.0) if case["kind"] == "screened" else (case["r2"], case["r3"])
        pairs = [(i, i) for i in range(n)] + [(i, j) for i in range(n) for j in range(i + 1, n) if d[i, j] <= c2]
        frags = _triples(d, min(c2, c3)) + [p for p in pairs]
    m = {p: min(k[p[0]] + (k[p[1]] if p[0] != p[1] else 0.0), v) for p in pairs}
    for i, j in pairs:
        fl += 2.0 * x * v * m[i, j] + 2.0 * x * m[i, j] ** 2 + 4.0 * v * k[i] * k[j] + 12.0 * m[i, j] ** 3
    for fr in frags:                  # ten sweeps of the couplings
        o = sorted(set(fr))
        pm = np.mean([m.get((a, b), 2 * k.mean()) for a in o for b in o if a <= b])
        fl += 10.0 * 0.5 * len(o) * (len(o) + 1) * 2 * (len(o) - 1) * 4.0 * pm ** 3
    if case["kind"] in ("grad", "relaxed"):
        byt += 8.0 * (n * v * x + n * n + v)
        fl += sum(4.0 * x * v * m[p] for p in pairs)
    if case["kind"] == "relaxed":
        fl += n * 8.0 * v ** 3 + 2.0 * n * v * v * x
    return {"bytes": byt + 40.0 * len(frags), "flops": fl}


def _triples(d, cut):
    n = d.shape[0]
    return [(i, j, k) for i in range(n) for j in range(i + 1, n) if d[i, j] <= cut
            for k in range(j + 1, n) if d[i, k] <= cut and d[j, k] <= cut]


# ---------------------------------------------------------------- the same in 64 bits, in plain torch
_M = (1 << 64) - 1


def _s64(x):
    return x - (1 << 64) if x >> 63 else x


def _mix(z):
    for sh, mul in ((30, 0xBF58476D1CE4E5B9), (27, 0x94D049BB133111EB), (31, None)):
        z = z ^ ((z >> sh) & ((1 << (64 - sh)) - 1))
        if mul is not None:
            z = z * _s64(mul)
    return z


def _mix_int(z):
    z &= _M
    z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & _M
    z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & _M
    return z ^ (z >> 31)


def _B(s, case, i):
    """B[i]; without a stored B the counter-based draw: the sum of twelve 16-bit fields of three
    consecutive SplitMix64 outputs, centred."""
    if "B" in s:
        return s["B"][i]
    v, x = case["n_vir"], case["n_aux"]
    key = _mix_int(s["seed"] ^ ((5 * 0xD1B54A32D192ED03) & _M))
    ctr = torch.arange(i * v * x, (i + 1) * v * x, device=DEV)
    tot = torch.zeros_like(ctr)
    for t in range(3):
        h = _mix((ctr * 3 + (t + 1)) * _s64(0x9E3779B97F4A7C15) + _s64(key))
        for sh in (0, 16, 32, 48):
            tot += (h >> sh) & 0xFFFF
    return s["env"][i][:, None] * ((tot - 393210).to(F64) * 2.0 ** -16).reshape(v, x)


def _clusters(n, pairs, triples):
    tp, cnt = {}, np.zeros(n, dtype=np.int64)
    w = np.ones(n, dtype=np.int64)
    for i, j in pairs:
        w[i] -= 1
        w[j] -= 1
    for t in triples:
        for p in ((t[0], t[1]), (t[0], t[2]), (t[1], t[2])):
            tp[p] = tp.get(p, 0) + 1
        for q in t:
            cnt[q] += 1
    return ([((i,), int(w[i] + cnt[i])) for i in range(n)] + [(p, 1 - tp.get(p, 0)) for p in pairs]
            + [(t, 1) for t in triples])


class _Exact:
    """OSVs, orthonormal pair bases U (span of [Q_i Q_j], F diagonal in them) and Jacobi sweeps of
    every fragment, all zero-padded to the largest pair order and batched."""

    def __init__(self, case, s):
        self.case, self.s = case, s
        n = case["n_occ"]
        self.f, self.e = s["f"].detach(), s["e"].detach()
        self.fh = self.f.cpu().numpy()
        self.B = [_B(s, case, i).detach() for i in range(n)]
        self.w, self.V, self.T = [], [], []
        for i in range(n):
            T = (self.B[i] @ self.B[i].T) / (self.e[:, None] + self.e[None, :] - 2.0 * self.f[i, i])
            w, V = torch.linalg.eigh(T)
            self.w.append(w.flip(0))
            self.V.append(V.flip(1))
            self.T.append(T)
        l = case["l_osv"]
        self.k = [int((w >= l).sum()) if l > 0 else case["n_vir"] for w in self.w]
        self.Q = [V[:, :k] for V, k in zip(self.V, self.k)]

    def bases(self, frags):
        need = sorted({(a, b) for o, _ in frags for a in o for b in o if a <= b})
        self.id = {p: t for t, p in enumerate(need)}
        U, et = [], []
        for i, j in need:
            P = self.Q[i] if i == j else torch.cat([self.Q[i], self.Q[j]], 1)
            q, sv, _ = torch.linalg.svd(P, full_matrices=False)
            q = q[:, sv * sv >= 1e-10 * sv[0] * sv[0]]
            ew, W = torch.linalg.eigh(q.T @ (self.e[:, None] * q))
            U.append(q @ W)
            et.append(ew)
        R = max(u.shape[1] for u in U)
        self.U = torch.zeros((len(need), self.case["n_vir"], R), dtype=F64, device=DEV)
        self.et = torch.zeros((len(need), R), dtype=F64, device=DEV)
        self.on = torch.zeros((len(need), R), dtype=F64, device=DEV)
        self.K = torch.zeros((len(need), R, R), dtype=F64, device=DEV)
        for t, (i, j) in enumerate(need):
            r = U[t].shape[1]
            self.U[t, :, :r], self.et[t, :r], self.on[t, :r] = U[t], et[t], 1.0
            self.K[t, :r, :r] = (U[t].T @ self.B[i]) @ (U[t].T @ self.B[j]).T

    def solve(self, frags, each):
        """Energies of the fragments; each(orbital lists, weights, pair ids, Y) sees every batch."""
        en = torch.zeros(len(frags), dtype=F64, device=DEV)
        R = self.K.shape[1]
        step = max(1, int(3e8 / (R * R * 40)))
        for nc in (1, 2, 3):
            at = [t for t, (o, _) in enumerate(frags) if len(o) == nc]
            for lo in range(0, len(at), step):
                ids = at[lo:lo + step]
                orb = [frags[t][0] for t in ids]
                pr = [(a, b) for a in range(nc) for b in range(a, nc)]
                pid = {p: torch.tensor([self.id[o[p[0]], o[p[1]]] for o in orb], device=DEV) for p in pr}
                fo = {(a, b): torch.tensor([self.fh[o[a], o[b]] for o in orb], dtype=F64, device=DEV)[:, None, None]
                      for a in range(nc) for b in range(nc)}
                D, K, sig = {}, {}, {}
                for p in pr:
                    t = self.et[pid[p]]
                    m = self.on[pid[p]]
                    m = m[:, :, None] * m[:, None, :]
                    D[p] = (t[:, :, None] + t[:, None, :] - fo[p[0], p[0]] - fo[p[1], p[1]]) * m + (1.0 - m)
                    K[p] = self.K[pid[p]]
                    for q in pr:
                        if p != q and set(p) & set(q):
                            sig[p, q] = self.U[pid[p]].transpose(1, 2) @ self.U[pid[q]]
                Y = {p: -K[p] / D[p] for p in pr}
                for _ in range(100):
                    new = {}
                    for a, b in pr:
                        C = torch.zeros_like(K[a, b])
                        for k in range(nc):
                            for u, w, fk, skip in ((k, b, fo[a, k], k == a), (a, k, fo[k, b], k == b)):
                                if not skip:
                                    q = (min(u, w), max(u, w))
                                    y = Y[q] if u <= w else Y[q].transpose(1, 2)
                                    sg = sig[(a, b), q]
                                    C += fk * (sg @ y @ sg.transpose(1, 2))
                        new[a, b] = (C - K[a, b]) / D[a, b]
                    off = max(float((new[p] - Y[p]).abs().max()) for p in pr)
                    Y = new
                    if off < 1e-15:
                        break
                for p in pr:
                    en[torch.tensor(ids, device=DEV)] += (2.0 if p[0] < p[1] else 1.0) * (
                        K[p] * (2.0 * Y[p] - Y[p].transpose(1, 2))).sum((1, 2))
                if each is not None:
                    each(orb, [frags[t][1] for t in ids], pid, Y)
        return en

    def gradient(self, frags, relaxed):
        """dE/dB, dE/df (symmetrised), dE/de of the Hylleraas functional; relaxed: with the
        response of the kept OSVs to T_ii."""
        n, v, x = self.case["n_occ"], self.case["n_vir"], self.case["n_aux"]
        G = torch.zeros((n, n, v, v), dtype=F64, device=DEV)     # sum of weighted T~_ij
        df = torch.zeros((n, n), dtype=F64, device=DEV)
        de = torch.zeros(v, dtype=F64, device=DEV)
        dQ = [torch.zeros_like(q) for q in self.Q]
        if relaxed:
            X = {p: torch.linalg.pinv(self.U[t].T @ (self.Q[p[0]] if p[0] == p[1] else
                 torch.cat([self.Q[p[0]], self.Q[p[1]]], 1))) for p, t in self.id.items()}
            BB = {p: self.B[p[0]] @ self.B[p[1]].T for p in self.id}

        def each(orb, wt, pid, Y):
            for q, (o, c) in enumerate(zip(orb, wt)):
                nc = len(o)
                T = {}
                for (a, b), ids in pid.items():
                    U = self.U[ids[q]]
                    T[a, b] = U @ Y[a, b][q] @ U.T
                    T[b, a] = T[a, b].T
                Tt = {p: 2.0 * t - t.T for p, t in T.items()}
                for (a, b), t in Tt.items():
                    G[o[a], o[b]] += c * t
                    de.add_(2.0 * c * (t * T[a, b]).sum(1))
                for a in range(nc):
                    for b in range(nc):
                        g = sum((Tt[a, j] * T[b, j]).sum() + (Tt[j, b] * T[j, a]).sum() for j in range(nc))
                        df[o[a], o[b]] -= c * g
                if not relaxed:
                    continue
                for (a, b), ids in pid.items():
                    p = (o[a], o[b])
                    res = BB[p] + self.e[:, None] * T[a, b] + T[a, b] * self.e[None, :]
                    for k in range(nc):
                        res = res - self.f[p[0], o[k]] * T[k, b] - self.f[o[k], p[1]] * T[a, k]
                    rt = 2.0 * res - res.T
                    U, y, xm = self.U[ids[q]], Y[a, b][q], X[p]
                    dP = (4.0 if a < b else 2.0) * c * (rt @ U @ y.T + rt.T @ U @ y) @ xm.T
                    dQ[p[0]].add_(dP[:, :self.k[p[0]]])
                    if a < b:
                        dQ[p[1]].add_(dP[:, self.k[p[0]]:])

        en = self.solve(frags, each)
        dB = torch.stack([4.0 * sum(G[i, j] @ self.B[j] for j in range(n)) for i in range(n)])
        gap = math.inf
        if relaxed:
            for i in range(n):
                w, V, k = self.w[i], self.V[i], self.k[i]
                if k == 0 or k == v:
                    continue
                y = (V[:, k:].T @ dQ[i]) / (w[None, :k] - w[k:, None])
                gap = min(gap, float(w[k - 1] - w[k]))
                Z = V[:, k:] @ y @ V[:, :k].T
                Z = 0.5 * (Z + Z.T)
                D = self.e[:, None] + self.e[None, :] - 2.0 * self.f[i, i]
                dB[i] += 2.0 * (Z / D) @ self.B[i]
                t = Z * self.T[i] / D
                de -= 2.0 * t.sum(1)
                df[i, i] += 2.0 * t.sum()
        return en, dB, 0.5 * (df + df.T), de, gap


def exact(case, seed):
    kind, n = case["kind"], case["n_occ"]
    if kind == "localize":
        return _exact_localize(case, seed)
    if case["method"] == "randomized" or n * case["n_vir"] ** 2 > 1.2e8 or n * case["n_occ"] > 9000:
        return None        # the draws decide the randomized OSVs; the rest would take too long
    s = prepare(case, seed) if kind == "grad" and not case["stored"] else _inputs(case, seed)
    if kind == "solve" and case["l_osv"] == 0.0:
        return _exact_untruncated(case, s)
    if kind == "solve":
        return None
    x = _Exact(case, s)
    out = {"n_osv": np.array(x.k, dtype=np.int32)}
    r = s["r"]
    if kind in ("osv", "screened"):
        s2b = np.ones((n, n))
        for i in range(n):
            for j in range(i + 1, n):
                S = x.Q[i].T @ x.Q[j]
                s2b[i, j] = s2b[j, i] = float((S * S).sum()) / math.sqrt(x.k[i] * x.k[j])
        cls = np.where(s2b >= 1e-2, 2, np.where(s2b >= 1e-7, 1, 0)).astype(np.int32)
        if kind == "osv":
            np.fill_diagonal(cls, 2)
            up = cls[np.triu_indices(n, 1)]
            out.update(s2b=s2b, cls=cls, counts=[int((up == t).sum()) for t in (2, 1, 0)])
            return out
        pairs = [(i, j) for i in range(n) for j in range(i + 1, n) if cls[i, j] == 2]
        triples = [(i, j, k) for i, j in pairs for k in range(j + 1, n) if cls[i, k] == 2 and cls[j, k] == 2
                   and (s2b[i, j] + s2b[i, k] + s2b[j, k]) / 3.0 >= 0.2]
    else:
        d2 = ((r[:, None, :] - r[None, :, :]) ** 2).sum(-1)
        pairs = [(i, j) for i in range(n) for j in range(i + 1, n) if d2[i, j] <= case["r2"] ** 2]
        triples = _triples(np.sqrt(d2), min(case["r2"], case["r3"]))
    frags = _clusters(n, pairs, triples)
    x.bases(frags)
    wts = np.array([c for _, c in frags], dtype=np.int32)
    orbs = np.array([list(o) + [-1] * (3 - len(o)) for o, _ in frags], dtype=np.int32)
    if kind in ("grad", "relaxed"):
        en, dB, df, de, gap = x.gradient(frags, kind == "relaxed")
        E = float((en.cpu() * torch.tensor(wts, dtype=F64)).sum())
        out = {"E": torch.tensor(E, dtype=F64) if kind == "grad" else E, "dB": dB, "df": df, "de": de}
        return out if kind == "grad" else {"n_osv": np.array(x.k, dtype=np.int32), **out, "gap": gap}
    diag = [0.0] * n

    def each(orb, wt, pid, Y):
        for (a, b), ids in pid.items():
            if a == b:
                A = [x.Q[o[a]].T @ x.U[t] for o, t in zip(orb, ids)]
                for q, o in enumerate(orb):
                    diag[o[a]] = diag[o[a]] + wt[q] * (A[q] @ Y[a, b][q] @ A[q].T)

    en = x.solve(frags, each if kind == "screened" else None).cpu().numpy()
    out["E"] = float((en * wts).sum())
    if kind == "screened":
        weak = [(i, j) for i in range(n) for j in range(i + 1, n) if cls[i, j] == 1]
        we = np.zeros(len(weak))
        eig = [torch.linalg.eigh(q.T @ (x.e[:, None] * q)) for q in x.Q]
        Bt = [q.T @ b for q, b in zip(x.Q, x.B)]
        for t, (i, j) in enumerate(weak):
            K, S = Bt[i] @ Bt[j].T, x.Q[i].T @ x.Q[j]
            rhs = K - x.fh[i, j] * (diag[i] @ S + S @ diag[j])
            (ei, Wi), (ej, Wj) = eig[i], eig[j]
            T = -(Wi.T @ rhs @ Wj) / (ei[:, None] + ej[None, :] - x.fh[i, i] - x.fh[j, j])
            we[t] = 4.0 * float(((Wi.T @ K @ Wj) * T).sum())
        out["E_weak"] = float(we.sum())
        out["E"] += out["E_weak"]
        out["pair_e"] = _pair_table(n, orbs, wts, en, np.array(weak, dtype=np.int32).reshape(-1, 2), we)
        return out
    out["orbs"], out["weights"], out["frag_e"] = orbs, wts, en
    return out


def _exact_untruncated(case, s):
    """The closed form: amplitudes in the canonical orbitals, energies rotated back to the given ones."""
    n = case["n_occ"]
    B = torch.stack([_B(s, case, i) for i in range(n)])
    eo, V = torch.linalg.eigh(s["f"])
    Bc = torch.einsum("iaP,ik->kaP", B, V)
    K = torch.einsum("iaP,jbP->ijab", B, B)
    Kc = torch.einsum("iaP,jbP->ijab", Bc, Bc)
    e = s["e"]
    T = Kc / (eo[:, None, None, None] + eo[None, :, None, None] - e[None, None, :, None] - e[None, None, None, :])
    T = torch.einsum("klab,ik,jl->ijab", T, V, V)
    pe = (K * (2.0 * T - T.transpose(2, 3))).sum((2, 3))
    out = [float(pe[i, j]) * (2.0 if i < j else 1.0) for i in range(n) for j in range(i, n)]
    return {"n_osv": np.full(n, case["n_vir"], dtype=np.int32), "E": float(sum(out)), "pairs": np.array(out)}


def _exact_localize(case, seed):
    C, ao = _orbitals(case, seed)
    n = case["n_occ"]
    P = np.stack([C[a:b].T @ C[a:b] for a, b in zip(ao[:-1], ao[1:])], axis=2)
    P = np.ascontiguousarray(P)
    U = np.eye(n)
    sweeps, gain = 0, math.inf
    while gain > 1e-3 and sweeps < 100:
        sweeps, gain = sweeps + 1, 0.0
        for i in range(n):
            for j in range(i + 1, n):
                d = P[i, i] - P[j, j]
                a, b = P[i, j] @ P[i, j] - 0.25 * (d @ d), P[i, j] @ d
                th = 0.25 * math.atan2(b, -a)
                sn, cs = math.sin(th), math.cos(th)
                if abs(sn) < 1e-10:
                    continue
                gain += math.hypot(a, b) * (1.0 - math.cos(4.0 * th))
                U[:, i], U[:, j] = cs * U[:, i] + sn * U[:, j], cs * U[:, j] - sn * U[:, i]
                P[i], P[j] = cs * P[i] + sn * P[j], cs * P[j] - sn * P[i]
                P[:, i], P[:, j] = cs * P[:, i] + sn * P[:, j], cs * P[:, j] - sn * P[:, i]
    return {"U": U, "L": float(sum((P[i, i] ** 2).sum() for i in range(n))), "sweeps": sweeps}
