"""Performance cases of the Fock-build framework.

Each case is work that a user's program has the library do through the Python binding
(``paper_1708_00033_gb300.hf``): Fock builds of one molecule from the smallest to the evaluation size,
in FP64 and mixed precision, with host and device matrices and with both synthetic bases; difference builds
of an incremental SCF; batched builds of many small molecules; the set-up of a geometry; whole SCF runs
from the learned guess; a training step of that guess; and the eigensolver.

``exact`` restates what the library computes in plain torch, FP64: McMurchie-Davidson integrals over
Hermite Gaussians, the closed-shell J and K, the SCF cycle and the small network with its gradients.
"""
import functools
import math

import numpy as np
import torch

from paper_1708_00033_gb300 import guess, hf, inputs

TAU = inputs.BENCH_SCHWARZ_TAU       # 1e-10, the Schwarz threshold of the benchmarked workloads
PRIM_TAU = inputs.BENCH_PRIM_TAU     # 1e-14
FP32_CUTOFF = 1e-4                   # mixed precision: quartets with a bound below it run in FP32
DEV = "cuda:0"


def listed():
    return [
        # One water molecule: the smallest build, where launches and the longest single quartet count
        # (geometry scans, the first molecule a user tries).
        {"name": "fock_1w", "kind": "fock", "waters": 1, "tau": TAU},
        # The parity workload of the tests: 4 waters, 100 functions, no screening at all.
        {"name": "fock_4w_unscreened", "kind": "fock", "waters": 4, "tau": 0.0},
        # A mid-size cluster of an odd size through host (numpy) matrices, with J and K returned as well.
        {"name": "fock_13w_host", "kind": "fock", "waters": 13, "tau": TAU, "host": True, "jk": True},
        # The size of the held-out SCF evaluation clusters: 800 functions, all FP64.
        {"name": "fock_32w", "kind": "fock", "waters": 32, "tau": TAU},
        # The benchmarked 1,600-function cluster in mixed FP32/FP64 precision: the bulk of a mixed SCF.
        {"name": "mixed_64w", "kind": "fock", "waters": 64, "tau": TAU, "fp32": FP32_CUTOFF},
        # Split-valence basis with sp shells, contractions of one and of three primitives.
        {"name": "fock_10w_sp", "kind": "fock", "waters": 10, "tau": TAU, "sp": True},
        # J and K of a density change with density-weighted screening: a step of an incremental SCF.
        {"name": "delta_24w", "kind": "delta", "waters": 24, "tau": TAU, "fp32": FP32_CUTOFF},
        # Many independent small molecules in one call (U{1..8} waters each).
        {"name": "batch_16", "kind": "batch", "molecules": 16, "most": 8},
        # A new geometry: normalisation, one-electron matrices, pair data, bounds and quartet lists.
        {"name": "setup_20w", "kind": "setup", "waters": 20, "tau": TAU},
        # A whole SCF from the shipped learned guess: inference, builds, DIIS, diagonalisations.
        {"name": "scf_4w", "kind": "scf", "waters": 4, "tau": TAU},
        # One training step of the learned guess (forward, backward, Adam) on a default minibatch.
        {"name": "train_2048", "kind": "train", "batch": 2048},
        # Eigenpairs of a Fock-sized symmetric matrix (15 waters, odd order).
        {"name": "eigh_375", "kind": "eigh", "n": 375},
    ]


def _spread(rng, lo, hi):
    """A whole number in [lo, hi], spread evenly over its logarithm."""
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo - 0.49), math.log(hi + 0.49)))))))


def draw(rng):
    kind = rng.choice(["fock", "fock", "mixed", "sp", "delta", "batch", "setup", "scf", "train", "eigh"])
    if kind == "fock":
        n = _spread(rng, 1, 32)
        return {"kind": "fock", "waters": n, "tau": 0.0 if n <= 4 and rng.random() < 0.5 else TAU,
                "host": rng.random() < 0.3, "jk": rng.random() < 0.3}
    if kind == "mixed":
        return {"kind": "fock", "waters": _spread(rng, 2, 60), "tau": TAU, "fp32": FP32_CUTOFF,
                "jk": rng.random() < 0.3}
    if kind == "sp":
        return {"kind": "fock", "waters": _spread(rng, 1, 40), "tau": TAU, "sp": True, "host": rng.random() < 0.3}
    if kind == "delta":
        c = {"kind": "delta", "waters": _spread(rng, 2, 30), "tau": TAU}
        return {**c, "fp32": FP32_CUTOFF} if rng.random() < 0.5 else c
    if kind == "batch":
        return {"kind": "batch", "molecules": _spread(rng, 2, 40), "most": rng.randint(2, 8)}
    if kind == "setup":
        return {"kind": "setup", "waters": _spread(rng, 1, 40), "tau": TAU, "sp": rng.random() < 0.3}
    if kind == "scf":
        return {"kind": "scf", "waters": _spread(rng, 1, 8), "tau": TAU}
    if kind == "train":
        return {"kind": "train", "batch": _spread(rng, 64, 4096)}
    return {"kind": "eigh", "n": _spread(rng, 8, 600)}


# ------------------------------------------------------------------ inputs --


@functools.lru_cache(maxsize=1)
def _context():
    """The library context a program creates once, on torch's current stream."""
    return hf.Context(0)


def _molecule(waters, seed, sp=False):
    geom = inputs.water_cluster(waters, inputs.CONFIG_GUESS_EVAL, int(seed))
    return geom, (inputs.synthetic_sp_basis if sp else inputs.synthetic_basis)(geom)


def _normal(shape, seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return torch.randn(shape, dtype=torch.float64, device=DEV, generator=g)


def _density(S, n_occ, G):
    """P = 2 C C^T with the random orbitals C = G L^-T, L L^T = G^T S G: tr(PS) = 2 n_occ."""
    L = torch.linalg.cholesky(G.T @ S @ G)
    C = torch.linalg.solve_triangular(L, G.T, upper=False).T
    P = 2.0 * C @ C.T
    return (0.5 * (P + P.T)).contiguous()


def _densities(case, seed, ref):
    """The density of a build, or the change between two successive ones."""
    n_occ = inputs.n_electrons(ref.geom) // 2
    S = ref.overlap()
    G = _normal((ref.n_bf, n_occ), seed)
    P = _density(S, n_occ, G)
    if case["kind"] == "delta":
        P = (_density(S, n_occ, G + 1e-4 * _normal(G.shape, seed + 1000)) - P).contiguous()
    return P


def _train_data(case, seed):
    """A minibatch as the training set holds it: pair features of a cluster, targets and masks of its head."""
    n = case["batch"]
    rng = np.random.default_rng([int(seed), 7])
    d = rng.normal(size=(n, 3)) * 4.0
    head = rng.choice(3, size=n, p=[0.14, 0.44, 0.42])  # O-O, O-H, H-H shares of a water cluster
    R = np.linalg.norm(d, axis=1, keepdims=True)
    u = d / R
    X = np.concatenate([R, u, (u[:, :, None] * u[:, None, :]).reshape(n, 9), np.eye(3)[head]], axis=1)
    lo, hi = np.array([0, 225, 300])[head], np.array([225, 300, 325])[head]
    col = np.arange(325)[None, :]
    mask = (col >= lo[:, None]) & (col < hi[:, None])
    T = np.where(mask, 0.3 * rng.normal(size=(n, 325)) * np.exp(-0.3 * R), 0.0)
    return X.astype(np.float32), T.astype(np.float32), mask.astype(np.float32)


def _symmetric(n, seed):
    """A symmetric matrix with a Fock-like spectrum: a few deep levels, then a band, coupled throughout."""
    A = _normal((n, n), seed)
    A = 0.5 * (A + A.T) / math.sqrt(n)
    d = torch.linspace(-1.0, 4.0, n, dtype=torch.float64, device=DEV)
    d[: max(1, n // 25)] -= 19.0
    return (A + torch.diag(d)).cpu().numpy()


def _batch_sizes(case):
    """Waters of each molecule: part of the workload, so the same for every seed (the geometries are not)."""
    rng = np.random.default_rng([case["molecules"], case["most"]])
    return [int(x) for x in rng.integers(1, case["most"] + 1, size=case["molecules"])]


def prepare(case, seed):
    kind = case["kind"]
    ctx = _context()
    th = {"schwarz_tau": case.get("tau", TAU), "prim_tau": PRIM_TAU if case.get("tau", TAU) > 0 else 0.0}
    state = {"kind": kind, "case": case, "ctx": ctx, "th": th}
    if kind in ("fock", "delta", "scf", "setup"):
        geom, basis = _molecule(case["waters"], seed, case.get("sp", False))
        state.update(geom=geom, basis=basis)
        if kind != "setup":
            state["system"] = hf.System(ctx, geom, basis, fp32_cutoff=case.get("fp32", 0.0), **th)
        if kind in ("fock", "delta"):
            P = _densities(case, seed, Reference(geom, basis))
            state["P"] = P.cpu().numpy() if case.get("host") else P
        if kind == "scf":
            state["model"] = hf.Model(ctx, guess.load_weights()[0])
    elif kind == "batch":
        geoms, bases, P = [], [], []
        for m, n in enumerate(_batch_sizes(case)):
            geom, basis = _molecule(n, seed + 100 * m)
            geoms.append(geom)
            bases.append(basis)
            P.append(_densities(case, seed + 100 * m, Reference(geom, basis)).reshape(-1))
        state["batch"] = hf.Batch(ctx, geoms, bases, **th)
        state["P"] = torch.cat(P)
        state["F"] = torch.empty_like(state["P"])
    elif kind == "train":
        state["model"] = hf.Model(ctx, inputs.guess_init_weights(int(seed)))
        state["data"] = [torch.from_numpy(a).to(DEV) for a in _train_data(case, seed)]
    else:
        state["A"] = _symmetric(case["n"], seed)
    return state


def run(state):
    kind, case = state["kind"], state["case"]
    if kind == "fock":
        r = state["system"].fock_build(state["P"], want_J=case.get("jk", False), want_K=case.get("jk", False))
        return {k: r[k] for k in ("F", "J", "K", "E_elec") if r[k] is not None}
    if kind == "delta":
        J, K = hf.fock_build_partial(state["system"], state["P"], density_screen=True)
        return {"J": J, "K": K}
    if kind == "batch":
        _, E = state["batch"].fock_build(state["P"], state["F"], energies=True)
        return {"F": state["F"], "E": E}
    if kind == "setup":
        system = hf.System(state["ctx"], state["geom"], state["basis"], **state["th"])
        S, H = system.one_electron(device=True)
        return {"S": S, "H": H}
    if kind == "scf":
        r = hf.scf(state["system"], P_guess=hf.guess_predict(state["model"], state["system"]))
        return {"E": r["energy"], "P": r["P"], "eps": r["eps"]}
    if kind == "train":
        loss = state["model"].train_step(*state["data"], lr=1e-3)
        return {"loss": loss, "gradients": state["model"].weights(gradients=True)}
    w, V = hf.eigh(state["ctx"], state["A"])
    return {"w": w, "V": V}


# -------------------------------------------------------------------- work --

# Floating-point operations of one primitive quartet by total angular momentum (vertical recurrence with
# its set-up and Boys functions), and how many of a contracted quartet's primitive quartets reach 1e-14.
_PRIM_FLOPS = (40, 60, 130, 300, 700, 1500, 3000, 6500, 15000)
_PRIM_SHARE = 0.33


def _quartets(geom, basis, tau):
    """Operations estimate over the unique shell quartets whose Schwarz-like overlap bound passes tau."""
    l, at, off = [], [], basis.prim_offsets()
    a, npr = [], []
    for s in range(basis.n_shells):
        for x in ((0, 1) if basis.l[s] < 0 else (int(basis.l[s]),)):
            l.append(x)
            at.append(int(basis.atom[s]))
            a.append(float(basis.exps[off[s]:off[s + 1]].min()))
            npr.append(int(basis.nprim[s]))
    l, at, a, npr = np.array(l), np.array(at), np.array(a), np.array(npr)
    i, j = np.tril_indices(len(l))
    R2 = ((geom.xyz[at[i]] - geom.xyz[at[j]]) ** 2).sum(1)
    Q = np.exp(-a[i] * a[j] / (a[i] + a[j]) * R2)
    L, pp = l[i] + l[j], npr[i] * npr[j]
    flops = 0.0
    for L1 in range(5):
        q1 = np.sort(Q[L == L1])
        for L2 in range(L1 + 1):
            q2 = np.sort(Q[L == L2])
            if not len(q1) or not len(q2):
                continue
            n = float((len(q2) - np.searchsorted(q2, tau / np.maximum(q1, 1e-200))).sum()) * (0.5 if L1 == L2 else 1.0)
            prims = pp[L == L1].mean() * pp[L == L2].mean() * (_PRIM_SHARE if tau > 0 else 1.0)
            flops += n * prims * _PRIM_FLOPS[L1 + L2]
    return float(flops)


def _n_bf(basis):
    return int(sum(4 if x < 0 else inputs.NCART[int(x)] for x in basis.l))


def work(case):
    kind = case["kind"]
    if kind in ("fock", "delta"):
        geom, basis = _molecule(case["waters"], 0, case.get("sp", False))
        flops = _quartets(geom, basis, case["tau"] if kind == "fock" else case["tau"] * 1e4)
        outs = 2 if kind == "delta" else 3 if case.get("jk") else 1
        return {"bytes": 8.0 * _n_bf(basis) ** 2 * (1 + outs), "flops": flops}
    if kind == "batch":
        ms = [_molecule(n, m) for m, n in enumerate(_batch_sizes(case))]
        return {"bytes": 16.0 * sum(_n_bf(b) ** 2 for _, b in ms), "flops": sum(_quartets(g, b, TAU) for g, b in ms)}
    if kind == "setup":
        geom, basis = _molecule(case["waters"], 0, case.get("sp", False))
        N, pairs = _n_bf(basis), basis.n_shells * (basis.n_shells + 1) / 2
        # one bound per pair from its (ab|ab) quartet, one nuclear-attraction sum per pair
        return {"bytes": 16.0 * N * N, "flops": pairs * 81 * 1000 + 4.0 * N * N * geom.n_atoms * 9 * 10}
    if kind == "scf":
        geom, basis = _molecule(case["waters"], 0)
        N = _n_bf(basis)
        return {"bytes": 16.0 * N * N, "flops": 12 * (_quartets(geom, basis, TAU) + 20.0 * N ** 3)}
    if kind == "train":
        n, w = case["batch"], 256 * 16 + 256 * 256 + 325 * 256
        return {"bytes": 4.0 * n * (16 + 2 * 325) + 28.0 * w, "flops": 2.0 * n * (3 * w - 256 * 16)}
    return {"bytes": 16.0 * case["n"] ** 2 + 8.0 * case["n"], "flops": 9.0 * case["n"] ** 3}


# ------------------------------------------------------------------- exact --


def _hermites(L):
    return [(t, u, n - t - u) for n in range(L + 1) for t in range(n, -1, -1) for u in range(n - t, -1, -1)]


def _cart(l):
    return [(x, y, l - x - y) for x in range(l, -1, -1) for y in range(l - x, -1, -1)]


def _boys(L, T):
    """[F_0(T), ..., F_L(T)]: the ascending series for the top order below 40, erf and the upward recursion above."""
    Ts = T.clamp(max=40.0)
    term = torch.full_like(Ts, 1.0 / (2 * L + 1))
    top = term.clone()
    for i in range(1, 160):
        term = term * (2.0 * Ts / (2 * L + 2 * i + 1))
        top += term
    e = torch.exp(-Ts)
    low = [None] * (L + 1)
    low[L] = e * top
    for m in range(L - 1, -1, -1):
        low[m] = (2.0 * Ts * low[m + 1] + e) / (2 * m + 1)
    Tb = T.clamp(min=40.0)
    eb = torch.exp(-Tb)
    F = 0.5 * torch.sqrt(math.pi / Tb) * torch.erf(torch.sqrt(Tb))
    out = []
    for m in range(L + 1):
        out.append(torch.where(T < 40.0, low[m], F))
        F = ((2 * m + 1) * F - eb) / (2.0 * Tb)
    return out


def _hermite_coulomb(L, alpha, X, Y, Z):
    """{(t, u, v): R_tuv} for t + u + v <= L."""
    F = _boys(L, alpha * (X * X + Y * Y + Z * Z))
    cur = {(0, 0, 0): [(-2.0 * alpha) ** m * F[m] for m in range(L + 1)]}
    for h in _hermites(L)[1:]:
        i = next(k for k in range(3) if h[k])
        one = tuple(h[k] - (k == i) for k in range(3))
        D = (X, Y, Z)[i]
        low = cur[one]
        r = [D * low[m + 1] for m in range(len(low) - 1)]
        if h[i] >= 2:
            two = cur[tuple(h[k] - 2 * (k == i) for k in range(3))]
            r = [x + (h[i] - 1) * two[m + 1] for m, x in enumerate(r)]
        cur[h] = r
    return {h: v[0] for h, v in cur.items()}


class Reference:
    """One molecule in plain torch FP64."""

    def __init__(self, geom, basis):
        self.geom = geom
        self.xyz = torch.tensor(geom.xyz, dtype=torch.float64, device=DEV)
        groups, off, bf = {}, basis.prim_offsets(), 0
        for s in range(basis.n_shells):
            ex = tuple(basis.exps[off[s]:off[s + 1]])
            parts = [(0, basis.coefs), (1, basis.coefs_p)] if basis.l[s] < 0 else [(int(basis.l[s]), basis.coefs)]
            for l, co in parts:
                g = groups.setdefault((l, len(ex)), {"atom": [], "bf": [], "ex": [], "co": []})
                g["atom"].append(int(basis.atom[s]))
                g["bf"].append(bf)
                g["ex"].append(ex)
                # coefficients multiply normalised primitives: N ~ a^((2 l + 3) / 4); the rest is common
                g["co"].append([c * a ** (0.5 * l + 0.75) for c, a in zip(co[off[s]:off[s + 1]], ex)])
                bf += len(_cart(l))
        self.n_bf = bf
        self.groups = []
        for (l, n), g in sorted(groups.items(), reverse=True):
            self.groups.append({"l": l, "A": self.xyz[torch.tensor(g["atom"], device=DEV)],
                                "bf": torch.tensor(g["bf"], device=DEV),
                                "ex": torch.tensor(g["ex"], dtype=torch.float64, device=DEV),
                                "co": torch.tensor(g["co"], dtype=torch.float64, device=DEV)})
        self.pairs = [self._pair(self.groups[i], self.groups[j], i == j)
                      for i in range(len(self.groups)) for j in range(i, len(self.groups))]
        d = torch.empty(bf, dtype=torch.float64, device=DEV)
        for q in self.pairs:  # unit self-overlap of every function
            same = (q["mu"] == q["nu"])
            d[q["mu"][same]] = (q["E"][..., 0] * ((math.pi / q["p"]) ** 1.5)[:, None, :]).sum(-1)[same]
        norm = d.rsqrt()
        for q in self.pairs:
            q["E"] *= (norm[q["mu"]] * norm[q["nu"]])[..., None, None]
        self.norm = norm

    def _pair(self, g, h, same):
        n, m = g["ex"].shape[0], h["ex"].shape[0]
        if same:
            i, j = torch.tril_indices(n, n, device=DEV)
        else:
            i, j = (x.reshape(-1) for x in torch.meshgrid(torch.arange(n, device=DEV), torch.arange(m, device=DEV),
                                                          indexing="ij"))
        k = i.shape[0]
        a = g["ex"][i][:, :, None].expand(-1, -1, h["ex"].shape[1]).reshape(k, -1)
        b = h["ex"][j][:, None, :].expand(-1, g["ex"].shape[1], -1).reshape(k, -1)
        c = (g["co"][i][:, :, None] * h["co"][j][:, None, :]).reshape(k, -1)
        A, B = g["A"][i], h["A"][j]
        p = a + b
        P = (a[..., None] * A[:, None] + b[..., None] * B[:, None]) / p[..., None]
        la, lb = g["l"], h["l"]
        E1 = [self._hermite_1d(la, lb + 2, a, b, A[:, d], B[:, d], P[:, :, d]) for d in range(3)]
        ca, cb, hs = _cart(la), _cart(lb), _hermites(la + lb)
        E = torch.stack([torch.stack([c * E1[0][x[0]][y[0]][t[0]] * E1[1][x[1]][y[1]][t[1]] * E1[2][x[2]][y[2]][t[2]]
                                      if all(t[d] <= x[d] + y[d] for d in range(3)) else torch.zeros_like(c)
                                      for t in hs], -1) for x in ca for y in cb], 1)
        mu = g["bf"][i][:, None] + torch.arange(len(ca), device=DEV).repeat_interleave(len(cb))[None]
        nu = h["bf"][j][:, None] + torch.arange(len(cb), device=DEV).repeat(len(ca))[None]
        return {"la": la, "lb": lb, "L": la + lb, "p": p, "P": P, "E": E, "mu": mu, "nu": nu, "b": b, "c": c, "E1": E1}

    @staticmethod
    def _hermite_1d(la, lb, a, b, A, B, P):
        """E[i][j][t] of one direction, E_0^00 carrying exp(-ab/p (A - B)^2)."""
        p = a + b
        PA, PB, h = P - A[:, None], P - B[:, None], 0.5 / p
        E = [[None] * (lb + 1) for _ in range(la + 1)]
        E[0][0] = [torch.exp(-a * b / p * ((A - B) ** 2)[:, None])]

        def up(e, X):
            n = len(e)
            z = torch.zeros_like(p)
            return [h * (e[t - 1] if t >= 1 else z) + X * (e[t] if t < n else z)
                    + (t + 1) * (e[t + 1] if t + 1 < n else z) for t in range(n + 1)]

        for i in range(la + 1):
            if i:
                E[i][0] = up(E[i - 1][0], PA)
            for j in range(1, lb + 1):
                E[i][j] = up(E[i][j - 1], PB)
        return E

    def _full(self, blocks):
        M = torch.empty((self.n_bf, self.n_bf), dtype=torch.float64, device=DEV)
        for q, v in zip(self.pairs, blocks):
            M[q["mu"], q["nu"]] = v
            M[q["nu"], q["mu"]] = v
        return M

    def overlap(self):
        return self._full([(q["E"][..., 0] * ((math.pi / q["p"]) ** 1.5)[:, None, :]).sum(-1) for q in self.pairs])

    def core(self):
        """T + V."""
        Z = torch.tensor(self.geom.Z, dtype=torch.float64, device=DEV)
        out = []
        for q in self.pairs:
            E1, b, w = q["E1"], q["b"], q["c"] * (math.pi / q["p"]) ** 1.5
            T = []
            for x in _cart(q["la"]):
                for y in _cart(q["lb"]):
                    s = [E1[d][x[d]][y[d]][0] for d in range(3)]
                    k = []
                    for d in range(3):
                        j = y[d]
                        v = -2.0 * b * b * E1[d][x[d]][j + 2][0] + b * (2 * j + 1) * s[d]
                        k.append(v - 0.5 * j * (j - 1) * E1[d][x[d]][j - 2][0] if j >= 2 else v)
                    T.append((w * (k[0] * s[1] * s[2] + s[0] * k[1] * s[2] + s[0] * s[1] * k[2])).sum(-1))
            T = torch.stack(T, 1) * self.norm[q["mu"]] * self.norm[q["nu"]]
            hs, V = _hermites(q["L"]), torch.zeros_like(T)
            step = max(1, int(2e6 // (q["p"].shape[0] * q["p"].shape[1])))
            for c0 in range(0, Z.shape[0], step):
                D = q["P"][:, :, None, :] - self.xyz[c0:c0 + step]
                R = _hermite_coulomb(q["L"], q["p"][:, :, None], D[..., 0], D[..., 1], D[..., 2])
                R = torch.stack([(R[h] * Z[c0:c0 + step]).sum(-1) * (2 * math.pi / q["p"]) for h in hs], -1)
                V -= torch.einsum("kcph,kph->kc", q["E"], R)
            out.append(T + V)
        return self._full(out)

    def nuclear(self):
        Z = torch.tensor(self.geom.Z, dtype=torch.float64, device=DEV)
        i, j = torch.triu_indices(len(Z), len(Z), 1, device=DEV)
        return float((Z[i] * Z[j] / (self.xyz[i] - self.xyz[j]).norm(dim=1)).sum())

    def eri(self):
        """(mu nu|la si) over all N^4 indices."""
        N = self.n_bf
        G = torch.empty((N, N, N, N), dtype=torch.float64, device=DEV)
        for x, A in enumerate(self.pairs):
            for B in self.pairs[: x + 1]:
                self._eri_block(A, B, G)
        return G

    @staticmethod
    def _eri_block(A, B, G):
        hA, hB = _hermites(A["L"]), _hermites(B["L"])
        L = A["L"] + B["L"]
        nB, pB = B["p"].shape
        step = max(1, int(4e6 // (A["p"].shape[1] * nB * pB * (1 + L))))
        for k0 in range(0, A["p"].shape[0], step):
            p, P, E = (A[s][k0:k0 + step] for s in ("p", "P", "E"))
            pp, qq = p[:, :, None, None], B["p"][None, None]
            D = P[:, :, None, None, :] - B["P"][None, None]
            R = _hermite_coulomb(L, pp * qq / (pp + qq), D[..., 0], D[..., 1], D[..., 2])
            pref = 2.0 * math.pi ** 2.5 / (pp * qq * torch.sqrt(pp + qq))
            out = 0.0
            for i, h in enumerate(hA):
                S = torch.stack([R[tuple(h[d] + g[d] for d in range(3))] * (pref * (-1.0) ** sum(g)) for g in hB], -1)
                out = out + torch.einsum("apbc,axp->axbc", torch.einsum("apbqh,bcqh->apbc", S, B["E"]), E[..., i])
            m, n = A["mu"][k0:k0 + step, :, None, None], A["nu"][k0:k0 + step, :, None, None]
            r, s = B["mu"][None, None], B["nu"][None, None]
            for i, j in ((m, n), (n, m)):
                for k, l in ((r, s), (s, r)):
                    G[i, j, k, l] = out
                    G[k, l, i, j] = out


def _jk(G, P):
    N = P.shape[0]
    J = (G.reshape(N * N, N * N) @ P.reshape(-1)).reshape(N, N)
    K = torch.empty_like(J)
    for m in range(N):  # K_mn = sum_ls (ml|ns) P_ls
        K[m] = (G[m][:, :, :] * P[:, None, :]).sum((0, 2))
    return J, K


def _cost(waters, sp=False):
    """Roughly the seconds that the N^4 integrals of a cluster take here."""
    return waters ** 4 * (0.001 if sp else 0.03)


def _exact_scf(ref, n_occ):
    """Converged closed-shell SCF (core guess, DIIS), the converged density and its orbital energies."""
    S, H, G = ref.overlap(), ref.core(), ref.eri()
    s, U = torch.linalg.eigh(S)
    X = U @ torch.diag(s.rsqrt()) @ U.T
    fs, es, F = [], [], H
    for it in range(200):
        if it:
            J, K = _jk(G, P)
            F = H + J - 0.5 * K
            E = 0.5 * float((P * (H + F)).sum())
            e = X.T @ (F @ P @ S - S @ P @ F) @ X
            if float(e.abs().max()) < 1e-11:
                break
            fs, es = (fs + [F])[-8:], (es + [e])[-8:]
            if len(fs) > 1:
                m = len(fs)
                Bm = torch.zeros((m + 1, m + 1), dtype=torch.float64)
                Bm[:m, :m] = torch.tensor([[float((x * y).sum()) for y in es] for x in es])
                Bm[:m, :m] /= Bm[:m, :m].abs().max()
                Bm[m, :m] = Bm[:m, m] = -1.0
                rhs = torch.zeros(m + 1, dtype=torch.float64)
                rhs[m] = -1.0
                c = torch.linalg.lstsq(Bm, rhs[:, None], driver="gelsd").solution[:m, 0].tolist()
                F = sum(ck * fk for ck, fk in zip(c, fs))
        eps, V = torch.linalg.eigh(X.T @ F @ X)
        C = X @ V[:, :n_occ]
        P = 2.0 * C @ C.T
    return {"E": E + ref.nuclear(), "P": P.cpu().numpy(), "eps": torch.linalg.eigvalsh(X.T @ F @ X).cpu().numpy()}


def _exact_train(case, seed):
    """Loss and gradients of the masked squared error; the products use the weights' bfloat16 values."""
    X, T, M = (torch.from_numpy(a).to(DEV).double() for a in _train_data(case, seed))
    w = torch.from_numpy(inputs.guess_init_weights(int(seed))).to(DEV)
    shapes, parts, o = [(256, 16), (256,), (256, 256), (256,), (325, 256), (325,)], [], 0
    for s in shapes:
        k = math.prod(s)
        v = w[o:o + k].reshape(s)
        parts.append((v.bfloat16().double() if len(s) == 2 else v.double()).requires_grad_())
        o += k
    W1, b1, W2, b2, W3, b3 = parts
    act = torch.nn.functional.silu
    Y = act(act(X @ W1.T + b1) @ W2.T + b2) @ W3.T + b3
    loss = (M * (Y - T) ** 2).sum() / X.shape[0]
    loss.backward()
    return {"loss": float(loss.detach()), "gradients": torch.cat([p.grad.reshape(-1) for p in parts]).cpu().numpy()}


def exact(case, seed):
    kind = case["kind"]
    if kind == "train":
        return _exact_train(case, seed)
    if kind == "eigh":  # eigenvectors have no sign of their own
        return {"w": np.linalg.eigvalsh(_symmetric(case["n"], seed)), "V": None}
    if kind == "batch":
        sizes = _batch_sizes(case)
        if sum(_cost(n) for n in sizes) > 15:
            return None
        F, E = [], []
        for m, n in enumerate(sizes):
            ref = Reference(*_molecule(n, seed + 100 * m))
            P, H = _densities(case, seed + 100 * m, ref), ref.core()
            J, K = _jk(ref.eri(), P)
            F.append(H + J - 0.5 * K)
            E.append(0.5 * float((P * (H + F[-1])).sum()))
        return {"F": torch.cat([f.reshape(-1) for f in F]).cpu().numpy(), "E": np.array(E)}
    ref = Reference(*_molecule(case["waters"], seed, case.get("sp", False)))
    if kind == "setup":
        return {"S": ref.overlap().cpu().numpy(), "H": ref.core().cpu().numpy()}
    if _cost(case["waters"], case.get("sp", False)) > 15:
        return None
    if kind == "scf":
        return _exact_scf(ref, inputs.n_electrons(ref.geom) // 2)
    P = _densities(case, seed, ref)
    J, K = _jk(ref.eri(), P)
    if kind == "delta":
        return {"J": J.cpu().numpy(), "K": K.cpu().numpy()}
    H = ref.core()
    F = H + J - 0.5 * K
    out = {"F": F.cpu().numpy(), "E_elec": 0.5 * float((P * (H + F)).sum())}
    if case.get("jk"):
        out.update(J=J.cpu().numpy(), K=K.cpu().numpy())
    return out
