"""Generator of the FP64 class kernels with Hermite accumulators.

McMurchie-Davidson integrals with the geometry of the shell pairs taken out of the primitive loop.  For a
pair of primitives (exponents a, b, p = a + b) the product of the Cartesian functions [e0| is a sum over
Hermite Gaussians of order t with coefficients E_t that follow, per direction, from
    E_t^{e+1} = w E_{t-1}^e + PA E_t^e + (t+1) E_{t+1}^e,   w = 1/(2p),  PA = -(b/p) AB,
so every coefficient is a sum of (monomial of AB) x r^k w^s, r = b/p, and AB is the same for all primitives
of the shell pair.  The primitive loop therefore only accumulates, per bra scaling (k, s) and ket scaling
(k', s'),
    H[(k,s),(k',s')][N] += pref r^k w^s r'^k' w'^s' R_N(P - Q),
R_N the Hermite Coulomb integral (one recurrence over N = (t, u, v), no matter how many components the class
has), and the contracted quartet applies the AB and CD monomials once:
    X[0; k,s; N] = H,  X[e+1_i; k,s; N] = X[e; k,s+1; N+1_i] - AB_i X[e; k+1,s; N] + N_i X[e; k,s; N-1_i],
[e0|f0] = X[e; 0,0; 0] on both sides (N-raising and -lowering terms change sign on the ket), followed by the
same horizontal recurrence and digestion as the other kernels.  FP64 instructions per primitive quartet fall
by 1.3 (low classes) to 2.3 times ((dd|dd): 8,681 to 3,764) against the Obara-Saika vertical recurrence.

With u = 2b, v = 2p, and W = l_a + l_b, r^k w^s = w^W u^k v^(W-k-s): w^W is part of the stored prefactor, and
one scaling per side is 1.

Two kernels per class share this:
  thread: one quartet per thread (or lane group), accumulators in registers;
  warp:   one quartet per warp.  Phase 1, one primitive quartet per lane: R_N and the scalings go to shared
          memory.  Phase 2, accumulators spread over the lanes (slot s of lane l is accumulator 32 s + l):
          every lane adds S[pair] R[N] of each primitive quartet.  The contracted steps give each lane one
          column of the intermediate.
"""
from __future__ import annotations

CART = {L: [(x, y, L - x - y) for x in range(L, -1, -1) for y in range(L - x, -1, -1)] for L in range(9)}
AX = "xyz"
Z3 = (0, 0, 0)


def add(t, i, k=1):
    l = list(t)
    l[i] += k
    return tuple(l)


def plus(a, b):
    return tuple(x + y for x, y in zip(a, b))


def scalings(la, lb):
    """{(k, s): set of Hermite orders} of a pair, in a fixed order."""
    out = {}
    for deg in range(la, la + lb + 1):
        for h in range(deg + 1):
            for j in range((deg - h) // 2 + 1):
                out.setdefault((deg - h - 2 * j, h + j), set()).add(h)
    return dict(sorted(out.items(), key=lambda kv: (-kv[0][1], -kv[0][0])))


def items(la, lb):
    return [(k, s, t) for (k, s), hs in scalings(la, lb).items() for h in sorted(hs) for t in CART[h]]


def accumulators(la, lb, lc, ld):
    """[(bra scaling index, ket scaling index, N)], grouped by scaling pair."""
    B, K = scalings(la, lb), scalings(lc, ld)
    out = []
    for i, hb in enumerate(B.values()):
        for j, hk in enumerate(K.values()):
            for n in sorted({x + y for x in hb for y in hk}):
                out += [(i, j, t) for t in CART[n]]
    return out


def hermites(L):
    return [t for n in range(L + 1) for t in CART[n]]


def tname(t):
    return "%d%d%d" % t


class Ops:
    """FP64 operations counted as the other generators do: every add and multiply is one."""

    def __init__(self):
        self.n = 0


def scale_lines(la, lb, rec, pre, ops, start=None):
    """Lines computing start u^k v^(W-k-s) of every scaling, each from another by one multiplication (start: a
    factor, or None for 1); returns (lines, [name or None for 1])."""
    W = la + lb
    have = {(0, 0): start}
    if start is None:
        have.update({(1, 0): f"{rec}.u", (0, 1): f"{rec}.v"})
    lines = []

    def need(k, m):
        if (k, m) in have:
            return have[(k, m)]
        k1, m1 = (k - 1, m) if k > m or m == 0 else (k, m - 1)
        base = need(k1, m1)
        nm = f"{pre}_{k}_{m}"
        lines.append(f"const double {nm} = {base} * {rec}.{'u' if k1 < k else 'v'};")
        ops.n += 1
        have[(k, m)] = nm
        return nm

    return lines, [need(k, W - k - s) for (k, s) in scalings(la, lb)]


def r_lines(L, ops, leaf_orders=()):
    """Hermite Coulomb integrals r_N^(0) from g_m = (2 rho)^m F_m and the separation D = Q - P: with
    q^(m) = (-1)^m R^(m), q_{N+1_i}^(m) = D_i q_N^(m+1) - N_i q_{N-1_i}^(m+1).  Returns (lines, name of r_N,
    terms), terms(N) = [(axis or None, factor, name)]: r_N as a sum of D_axis * name and -factor * name.  No other
    r depends on an r_N^(0), so those of leaf_orders are not formed: the caller accumulates their terms."""
    recipe = {}

    def need(t, m):
        if (t, m) in recipe:
            return
        if t == Z3:
            recipe[(t, m)] = None
            return
        ones = [i for i in range(3) if t[i] == 1]
        i = ones[0] if ones else min((i for i in range(3) if t[i]), key=lambda i: t[i])
        recipe[(t, m)] = i
        need(add(t, i, -1), m + 1)
        if t[i] >= 2:
            need(add(t, i, -2), m + 1)

    for t in hermites(L):
        need(t, 0)
    nm = lambda t, m: f"g{m}" if t == Z3 else f"r{tname(t)}_{m}"  # noqa: E731
    lines = []
    for (t, m), i in sorted(recipe.items(), key=lambda kv: (sum(kv[0][0]), -kv[0][1])):
        if i is None:
            continue
        if m == 0 and sum(t) in leaf_orders:
            continue
        e = f"D{AX[i]} * {nm(add(t, i, -1), m + 1)}"
        ops.n += 1
        if t[i] >= 2:
            c = t[i] - 1
            e += (" - " if c == 1 else f" - {c}.0 * ") + nm(add(t, i, -2), m + 1)
            ops.n += 1 if c == 1 else 2
        lines.append(f"const double {nm(t, m)} = {e};")

    def terms(t):
        i = recipe[(t, 0)]
        out = [(i, 1, nm(add(t, i, -1), 1))]
        if t[i] >= 2:
            out.append((None, t[i] - 1, nm(add(t, i, -2), 1)))
        return out

    return lines, (lambda t: nm(t, 0)), terms


def prim_lines(la, lb, lc, ld, ops, leaf_orders=()):
    """One primitive quartet up to g_m, the scalings and r_N: (lines, r name, r terms, bra names, ket names).  The
    prefactor is part of the bra scalings."""
    L = la + lb + lc + ld
    lines = ["const double Dx = kp.Px - bp.Px, Dy = kp.Py - bp.Py, Dz = kp.Pz - bp.Pz;",
             "double rs, a2;",
             "herm_exponents(bp, kp, etab, ntype, rs, a2);",
             "const double pf = bp.K * kp.K * rs;",
             "double F[%d];" % (L + 1),
             "boys_eval_2t<%d>(a2 * (Dx * Dx + Dy * Dy + Dz * Dz), boys_tab, F);" % L]
    ops.n += 3 + 2 + 6 + (5 + 7 * (L + 1) + 2 if L <= 1 else 24 + 2 * L)
    lines.append("const double g0 = F[0];")
    pw = "a2"
    for m in range(1, L + 1):
        lines.append(f"const double g{m} = {pw} * F[{m}];")
        ops.n += 1
        if m < L:
            lines.append(f"const double a2_{m + 1} = {pw} * a2;")
            ops.n += 1
            pw = f"a2_{m + 1}"
    b, bn = scale_lines(la, lb, "bp", "sb", ops, "pf")
    k, kn = scale_lines(lc, ld, "kp", "uk", ops)
    r, rname, terms = r_lines(L, ops, leaf_orders)
    return lines + b + k + r, rname, terms, bn, kn


def transform(la, lb, src, ab, ket, ops, pre):
    """Straight-line [e| from the pair items: src(k, s, N) names the inputs; ab: prefix of the separation;
    returns (lines, {e: name})."""
    lines, memo = [], {}

    def need(e, k, s, t):
        if e == Z3:
            return src(k, s, t)
        key = (e, k, s, t)
        if key in memo:
            return memo[key]
        i = next(x for x in range(3) if e[x])
        e1 = add(e, i, -1)
        sg = "-" if ket else "+"
        ex = f"-{ab}{AX[i]} * {need(e1, k + 1, s, t)} {sg} {need(e1, k, s + 1, add(t, i))}"
        ops.n += 2
        if t[i]:
            x = need(e1, k, s, add(t, i, -1))
            ex += f" {sg} {x}" if t[i] == 1 else f" {sg} {t[i]}.0 * {x}"
            ops.n += 1 if t[i] == 1 else 2
        nm = f"{pre}{tname(e)}_{k}_{s}_{tname(t)}"
        lines.append(f"const double {nm} = {ex};")
        memo[key] = nm
        return nm

    return lines, {e: need(e, 0, 0, Z3) for n in range(la, la + lb + 1) for e in CART[n]}


def hrr(la, lb, src, ab, ops, pre):
    """(a b| from [e0|, (a b+1_i| = (a+1_i b| + AB_i (a b|: (lines, {(a, b): name})."""
    lines, memo = [], {}

    def need(a, b):
        if b == Z3:
            return src(a)
        if (a, b) in memo:
            return memo[(a, b)]
        i = next(x for x in range(3) if b[x])
        x, y = need(add(a, i), add(b, i, -1)), need(a, add(b, i, -1))
        nm = f"{pre}{tname(a)}_{tname(b)}"
        lines.append(f"const double {nm} = {x} + {ab}{AX[i]} * {y};")
        ops.n += 2
        memo[(a, b)] = nm
        return nm

    return lines, {(a, b): need(a, b) for a in CART[la] for b in CART[lb]}


def gen_thread(name, la, lb, lc, ld, hrr_digest):
    """Quartet function of the thread kernel; hrr_digest(acc name of (e, f)) -> (lines, op count) is the
    shared horizontal recurrence and digestion.  Returns (source, primitive ops, contracted ops)."""
    L = la + lb + lc + ld
    acc = accumulators(la, lb, lc, ld)
    po, co = Ops(), Ops()
    # r_N that few scalings use are accumulated from their terms with the scaling folded into D (p D_i once per
    # scaling): the top order, which one scaling uses, and order 1 when fewer than three do
    uses = {}
    for (i, j) in {(i, j) for i, j, _ in acc}:
        for n in {sum(t) for a, b, t in acc if (a, b) == (i, j)}:
            uses[n] = uses.get(n, 0) + 1
    leaf = {n for n in uses if n >= 1 and ((n == L and L != 2) or (n == 1 and uses[n] < 3))}
    lines, rname, terms, bn, kn = prim_lines(la, lb, lc, ld, po, leaf)
    body = list(lines)
    order = {}
    for idx, (i, j, t) in enumerate(acc):
        order.setdefault((i, j), []).append((idx, t))
    for (i, j), ts in order.items():
        if kn[j] is None:
            p = bn[i]
        else:
            p = f"s{i}_{j}"
            body.append(f"const double {p} = {bn[i]} * {kn[j]};")
            po.n += 1
        made = set()

        def coef(name, expr):
            if name not in made:
                made.add(name)
                body.append(f"const double {name} = {expr};")
                po.n += 1
            return name

        for idx, t in ts:
            if sum(t) not in leaf:
                body.append(f"h{idx} = fma({p}, {rname(t)}, h{idx});")
                po.n += 2
            elif sum(t) == 1:  # D_i (p g_1)
                ax, _, nm = terms(t)[0]
                body.append(f"h{idx} = fma(D{AX[ax]}, {coef(f'pg{i}_{j}', f'{p} * {nm}')}, h{idx});")
                po.n += 2
            else:
                for ax, c, nm in terms(t):
                    if ax is not None:
                        k = coef(f"pD{AX[ax]}{i}_{j}", f"{p} * D{AX[ax]}")
                    elif c == 1:
                        k = f"-{p}"
                    else:
                        k = coef(f"pn{c}_{i}_{j}", f"-{c}.0 * {p}")
                    body.append(f"h{idx} = fma({k}, {nm}, h{idx});")
                    po.n += 2
    B, K = list(scalings(la, lb)), list(scalings(lc, ld))
    where = {(B[i], K[j], t): f"h{idx}" for idx, (i, j, t) in enumerate(acc)}
    cont = []
    # bra transform once per ket item, then ket transform once per e
    mid = {}
    for (k2, s2, t2) in items(lc, ld):
        ls, out = transform(la, lb, lambda k, s, t: where[((k, s), (k2, s2), plus(t, t2))], "AB", False, co,
                            f"x{k2}{s2}{tname(t2)}_")
        cont += ls
        for e, nm in out.items():
            mid[(e, k2, s2, t2)] = nm
    final = {}
    for n in range(la, la + lb + 1):
        for e in CART[n]:
            ls, out = transform(lc, ld, lambda k, s, t: mid[(e, k, s, t)], "CD", True, co, f"y{tname(e)}_")
            cont += ls
            for f, nm in out.items():
                final[(e, f)] = nm
    tail, cops = hrr_digest(final)
    co.n += cops
    need_ab = any("AB" in l for l in cont + tail)
    need_cd = any("CD" in l for l in cont + tail)
    o = []
    o.append("template <int G>")
    o.append(f"__device__ __forceinline__ int quartet_h_{name}(const PairHdr& hb, const PairHdr& hk, const HermView& hv,"
             " const double* __restrict__ boys_tab, const double* __restrict__ Pd, int N, double fscale,"
             " double* __restrict__ Jt, double* __restrict__ Kt, double* qout, float ptau, int lane, bool valid)")
    o.append("{")
    o.append("    using real = double;")
    o.append("    const HermPair* __restrict__ bpp = hv.rec + hb.prim0;")
    o.append("    const HermPair* __restrict__ kpp = hv.rec + hk.prim0;")
    o.append("    const float* __restrict__ bB = hv.B + hb.prim0;")
    o.append("    const float* __restrict__ kB = hv.B + hk.prim0;")
    o.append("    const double2* __restrict__ etab = hv.etab;")
    o.append("    const int ntype = hv.ntype;")
    o.append("    // surviving primitive quartets, ket-major: ket primitive ik with the first nb(ik) bra primitives")
    o.append("    int nbb = hb.nprim;")
    o.append("    const int total = valid ? herm_total(bB, hb.nprim, kB, hk.nprim, ptau) : 0;")
    o.append("    if (valid) while (nbb > 0 && bB[nbb - 1] * kB[0] < ptau) nbb--;")
    o += [f"    double h{i} = 0.0;" for i in range(len(acc))]
    o.append("    int ib = 0, ik = 0, lk = -1, nq = 0;")
    o.append("    HermPair kp;")
    o.append("    auto advance = [&]() {")
    o.append("        if (++ib == nbb) {")
    o.append("            ib = 0;")
    o.append("            ik++;")
    o.append("            if (ik < hk.nprim)")
    o.append("                while (nbb > 0 && bB[nbb - 1] * kB[ik] < ptau) nbb--;")
    o.append("        }")
    o.append("    };")
    o.append("    if (G > 1)")
    o.append("        for (int s = 0; s < lane && s < total; s++) advance();")
    o.append("    for (int it = (G > 1 ? lane : 0); it < total; it += G) {")
    o.append("        if (ik != lk) {  // a lane reloads its ket record only when its ket primitive changes")
    o.append("            kp = kpp[ik];")
    o.append("            lk = ik;")
    o.append("        }")
    o.append("        const HermPair bp = bpp[ib];")
    o.append("#pragma unroll 1")
    o.append("        for (int s = 0; s < G && it + s + 1 < total; s++) advance();")
    o.append("        nq++;")
    o += ["        " + l for l in body]
    o.append("    }")
    o.append("    if constexpr (G > 1) {")
    o.append("#pragma unroll")
    o.append("        for (int o = 1; o < G; o <<= 1) {")
    o += [f"            h{i} += __shfl_xor_sync(0xffffffffu, h{i}, o);" for i in range(len(acc))]
    o.append("        }")
    o.append("    }")
    o.append("    if (!valid || lane != 0) return nq;")
    if need_ab:
        o.append("    const double ABx = hb.ABx, ABy = hb.ABy, ABz = hb.ABz;")
    if need_cd:
        o.append("    const double CDx = hk.ABx, CDy = hk.ABy, CDz = hk.ABz;")
    o += ["    " + l for l in cont]
    o += ["    " + l for l in tail]
    o.append("    return nq;")
    o.append("}")
    o.append(f"struct HermThread_{name} {{")
    o.append("    template <int G>")
    o.append("    static __device__ __forceinline__ int run(const PairHdr& hb, const PairHdr& hk, const HermView& hv,"
             " const double* bt, const double* Pd, int N, double f, double* Jt, double* Kt, double* qout, float ptau,"
             " int lane, bool valid)")
    o.append(f"    {{ return quartet_h_{name}<G>(hb, hk, hv, bt, Pd, N, f, Jt, Kt, qout, ptau, lane, valid); }}")
    o.append("};")
    return "\n".join(o) + "\n", po.n, co.n


def gen_warp(name, la, lb, lc, ld):
    """Traits of the warp kernel (herm_warp in eri_herm.cuh): sizes, index tables and straight-line steps."""
    L = la + lb + lc + ld
    acc = accumulators(la, lb, lc, ld)
    hs = hermites(L)
    hidx = {t: i for i, t in enumerate(hs)}
    B, K = list(scalings(la, lb)), list(scalings(lc, ld))
    BI, KI = items(la, lb), items(lc, ld)
    where = {(B[i], K[j], t): a for a, (i, j, t) in enumerate(acc)}
    po, co = Ops(), Ops()
    lines, rname, _, bn, kn = prim_lines(la, lb, lc, ld, po)
    po.n += sum(1 for n in kn if n is not None) * len(bn) + 2 * len(acc)
    es = [e for n in range(la, la + lb + 1) for e in CART[n]]
    fs = [f for n in range(lc, lc + ld + 1) for f in CART[n]]
    nslot = (len(acc) + 31) // 32
    o = []
    slot = []
    for a in range(nslot * 32):
        i, j, t = acc[a] if a < len(acc) else (0, 0, Z3)
        slot.append((i * len(K) + j) | (hidx[t] << 8))
    tab = []
    for (k, s, t) in BI:
        for (k2, s2, t2) in KI:
            tab.append(where[((k, s), (k2, s2), plus(t, t2))])
    fmt = lambda v: ",\n    ".join(", ".join(map(str, v[i:i + 24])) for i in range(0, len(v), 24))  # noqa: E731
    o.append("// accumulator 32 s + l: scaling pair in the low byte, Hermite index in the high byte")
    o.append(f"__device__ const unsigned short kHermSlot_{name}[{len(slot)}] = {{\n    {fmt(slot)}}};")
    o.append("// accumulator of (bra item, ket item)")
    o.append(f"__device__ const unsigned short kHermItem_{name}[{len(tab)}] = {{\n    {fmt(tab)}}};")
    o.append(f"struct HermWarp_{name} {{")
    nrp = len(hs) | 1
    o.append(f"    static constexpr int NR = {len(hs)}, NRP = {nrp}, NBS = {len(B)}, NKS = {len(K)}, NACC = {len(acc)},"
             f" NSLOT = {nslot}, NKI = {len(KI)}, NE = {len(es)}, NF = {len(fs)};")
    o.append(f"    static constexpr int LA = {la}, LB = {lb}, LC = {lc}, LD = {ld};")
    # quartets per group: about a warp's worth of (quartet, ket item) columns, or more where one quartet exceeds it (11
    # items: 33 columns, the last of them in a round of its own); one where L >= 7 needs the shared memory
    ng = 1 if L >= 7 else {1: 8, 4: 8, 11: 3, 15: 2, 35: 2}[len(KI)]
    o.append(f"    static constexpr int NQ = {ng};")
    o.append("    static __device__ __forceinline__ const unsigned short* slots() { return kHermSlot_%s; }" % name)
    o.append("    // one primitive quartet: R[0..NR), scalings sc[0..NBS + NKS)")
    o.append("    static __device__ __forceinline__ void prim(const HermPair& bp, const HermPair& kp, const double2* __restrict__ etab,"
             " int ntype, const double* __restrict__ boys_tab, double live, double* __restrict__ R, double* __restrict__ sc)")
    o.append("    {")
    # a padding lane's prefactor is zero
    o += ["        " + l.replace("const double pf = bp.K * kp.K * rs;", "const double pf = bp.K * kp.K * rs * live;")
          for l in lines]
    for i, t in enumerate(hs):
        o.append(f"        R[{i}] = {rname(t)};")
    for i, n in enumerate(bn):
        o.append(f"        sc[{i}] = {n};")
    for j, n in enumerate(kn):
        o.append(f"        sc[{len(bn) + j}] = {n if n else '1.0'};")
    o.append("    }")

    def step(fname, args, loads, lns, outs):
        o.append(f"    static __device__ __forceinline__ void {fname}({args})")
        o.append("    {")
        o.extend("        " + l for l in loads + lns + outs)
        o.append("    }")

    bpos = {it: i for i, it in enumerate(BI)}
    kpos = {it: i for i, it in enumerate(KI)}
    lns, out = transform(la, lb, lambda k, s, t: f"i{bpos[(k, s, t)]}", "AB", False, co, "x")
    step("bra", "const double* __restrict__ H, int j, double ABx, double ABy, double ABz, double* __restrict__ U",
         [f"const double i{b} = H[__ldg(kHermItem_{name} + {b * len(KI)} + j)];" for b in range(len(BI))], lns,
         [f"U[{i * len(KI)} + j] = {out[e]};" for i, e in enumerate(es)])
    n1 = co.n
    co.n = n1 * len(KI)
    k1 = Ops()
    lns, out = transform(lc, ld, lambda k, s, t: f"i{kpos[(k, s, t)]}", "CD", True, k1, "y")
    step("ket", "const double* __restrict__ U, double CDx, double CDy, double CDz, double* __restrict__ V",
         [f"const double i{j} = U[{j}];" for j in range(len(KI))], lns,
         [f"V[{i}] = {out[f]};" for i, f in enumerate(fs)])
    co.n += k1.n * len(es)
    k2 = Ops()
    epos = {e: i for i, e in enumerate(es)}
    lns, out = hrr(la, lb, lambda e: f"i{epos[e]}", "AB", k2, "p")
    step("hrr_bra", "const double* __restrict__ V, double ABx, double ABy, double ABz, double* __restrict__ Wd",
         [f"const double i{i} = V[{i * len(fs)}];" for i in range(len(es))], lns,
         [f"Wd[{i * len(fs)}] = {out[ab]};" for i, ab in enumerate((a, b) for a in CART[la] for b in CART[lb])])
    co.n += k2.n * len(fs)
    k3 = Ops()
    fpos = {f: i for i, f in enumerate(fs)}
    lns, out = hrr(lc, ld, lambda f: f"i{fpos[f]}", "CD", k3, "q")
    step("hrr_ket", "const double* __restrict__ Wd, double CDx, double CDy, double CDz, double* __restrict__ X",
         [f"const double i{i} = Wd[{i}];" for i in range(len(fs))], lns,
         [f"X[{i}] = {out[cd]};" for i, cd in enumerate((c, d) for c in CART[lc] for d in CART[ld])])
    nab, ncd = len(CART[la]) * len(CART[lb]), len(CART[lc]) * len(CART[ld])
    co.n += k3.n * nab + 12 * nab * ncd
    o.append("};")
    return "\n".join(o) + "\n", po.n, co.n


def gen_onee(la, lb):
    """Traits of the one-electron kernel of a pair class (one_electron_pair in onee_herm.cuh): nuclear attraction
    with the same Hermite accumulators, a point charge in the ket's place."""
    L = la + lb
    hs, sc, its = hermites(L), list(scalings(la, lb)), items(la, lb)
    hidx = {t: i for i, t in enumerate(hs)}
    ops = Ops()
    o = [f"struct OneE_{la}{lb} {{",
         f"    static constexpr int LA = {la}, LB = {lb}, NR = {len(hs)}, NI = {len(its)};",
         "    // RS += Z R_N(P - C)",
         "    static __device__ __forceinline__ void nucleus(const HermPair& bp, double Cx, double Cy, double Cz, double Z,"
         " const double* __restrict__ boys_tab, double (&RS)[NR])",
         "    {",
         "        const double Dx = Cx - bp.Px, Dy = Cy - bp.Py, Dz = Cz - bp.Pz;",
         f"        double F[{L + 1}];",
         f"        boys_eval_2t<{L}>(bp.v * (Dx * Dx + Dy * Dy + Dz * Dz), boys_tab, F);",
         "        double zp = Z;"]
    for m in range(L + 1):
        if m:
            o.append("        zp *= bp.v;")
        o.append(f"        const double g{m} = zp * F[{m}];")
    lines, rname, _ = r_lines(L, ops)
    o += ["        " + l for l in lines]
    o += [f"        RS[{i}] += {rname(t)};" for i, t in enumerate(hs)]
    o += ["    }", "    // acc += pf sigma RS_N of every scaling and order",
          "    static __device__ __forceinline__ void scale(const HermPair& bp, double pf, const double (&RS)[NR], double (&acc)[NI])",
          "    {"]
    lines, names = scale_lines(la, lb, "bp", "sb", ops, "pf")
    o += ["        " + l for l in lines]
    o += [f"        acc[{x}] = fma({names[sc.index((k, s))]}, RS[{hidx[t]}], acc[{x}]);" for x, (k, s, t) in enumerate(its)]
    o += ["    }", "    // (a|b) from the accumulators",
          "    static __device__ __forceinline__ void finish(const double (&acc)[NI], double ABx, double ABy, double ABz, double* __restrict__ V)",
          "    {"]
    pos = {it: x for x, it in enumerate(its)}
    lines, out = transform(la, lb, lambda k, s, t: f"acc[{pos[(k, s, t)]}]", "AB", False, ops, "x")
    l2, ab = hrr(la, lb, lambda e: out[e], "AB", ops, "p")
    o += ["        " + l for l in lines + l2]
    o += [f"        V[{i}] = {ab[k]};" for i, k in enumerate((a, b) for a in CART[la] for b in CART[lb])]
    o += ["    }", "};", f"ONEE_KERNEL({la}, {lb})", ""]
    return "\n".join(o)
