// Device-side building blocks of the Hermite-accumulator class kernels (gen_herm.py has the method).
#pragma once
#include "eri_common.cuh"

namespace hf {

// The pair exponents' part of one primitive quartet: rs = 1/sqrt(p + q) and a2 = 2 p q / (p + q).  A basis
// has few distinct exponents (25 for the water basis, 325 sums p), so both come from a table over
// (type of p, type of q): one 16-byte load instead of about 11 FP64 instructions, of 30 to 60 that a
// low-angular-momentum primitive quartet takes in all.  Bases with more than kHermMaxTypes sums (table
// above 32 MB) evaluate them directly.
__device__ __forceinline__ void herm_exponents(const HermPair& bp, const HermPair& kp,
                                               const double2* __restrict__ etab, int ntype, double& rs, double& a2)
{
    if (etab) {  // launch-uniform
        const double2 e = __ldg(etab + (size_t)bp.type * ntype + kp.type);
        rs = e.x;
        a2 = e.y;
    } else {
        // v = 2p: p + q = (v + v') / 2, 2 p q / (p + q) = v v' / (v + v')
        const double s = bp.v + kp.v;
        const double r = rsqrt(s);
        rs = 1.41421356237309504880 * r;
        a2 = bp.v * kp.v * (r * r);
    }
}

// F_m(T) from T2 = 2T (the argument the Hermite kernels form): T by an exponent decrement, no FP64 instruction.
template <int L>
__device__ __forceinline__ void boys_eval_2t(double T2, const double* __restrict__ tab, double* F)
{
    const int hi = __double2hiint(T2);
    const double T = hi >= 0x00200000 ? __hiloint2double(hi - 0x00100000, __double2loint(T2)) : 0.0;
    boys_eval<L>(T, tab, F);
}

// Number of surviving primitive quartets: bra primitive ib pairs with the first c(ib) ket primitives whose bound
// product reaches ptau, c non-increasing (bounds sorted descending).
__device__ __forceinline__ int herm_total(const float* __restrict__ bB, int nbp, const float* __restrict__ kB, int nkp,
                                          float ptau)
{
    int total = 0;
    for (int ib = 0, c = nkp; ib < nbp; ib++) {
        const float Bb = bB[ib];
        while (c > 0 && Bb * kB[c - 1] < ptau) c--;
        if (c == 0) break;
        total += c;
    }
    return total;
}

// bra and ket of quartet q of a launch
__device__ __forceinline__ void quartet_pair(const EriArgs& a, long long q, int& b, int& k)
{
    const long long c = q >> kChunkShift;
    b = a.chunk ? find_bra_in(a.offsets, a.chunk[c], a.chunk[c + 1], q) : find_bra(a.offsets, a.n_bra, q);
    k = (int)(q - a.offsets[b]) + (a.kstart ? a.kstart[b] : 0);
}

// Digestion weight f = 1/((1+d_AB)(1+d_CD)(1+d_AB,CD)) of a unique quartet.
__device__ __forceinline__ double quartet_weight(const PairHdr& hb, const PairHdr& hk, bool same)
{
    return (hb.A == hb.B ? 0.5 : 1.0) * (hk.A == hk.B ? 0.5 : 1.0) * (same ? 0.5 : 1.0);
}

// Density-weighted screening of one quartet (see density_block_max): whether it lives, and its primitive threshold.
__device__ __forceinline__ bool quartet_lives(const EriArgs& a, const PairHdr& hb, const PairHdr& hk, float& pt)
{
    if (!a.dsh) return true;
    const float dm = density_block_max(a, hb, hk);
    pt = pt / fmaxf(dm, 1e-30f);
    return 4.0f * (float)(hb.Q * hk.Q) * dm >= a.dtau;
}

// ------------------------------------------------------------ thread kernel --
// One quartet per lane group of GK lanes.  Each warp sorts its window of a.rounds * 32 / GK quartets by staircase
// length and runs it in a.rounds rounds of similar lengths.
template <class C, int GK>
__device__ __forceinline__ void herm_thread_kernel(const EriArgs& a)
{
    if (a.bad && *a.bad) return;
    const float ptau = (float)a.prim_tau;
    const size_t cofs = a.n_copies > 1 ? (size_t)(blockIdx.x % a.n_copies) * a.copy_stride : 0;
    const HermView hv = a.herm;
    unsigned nprimq = 0;
    constexpr int gpw = 32 / GK;
    constexpr int kWmax = kSortRounds * gpw;
    __shared__ unsigned skeys[(kEriThreads / 32) * kWmax];
    unsigned* const wkeys = skeys + (threadIdx.x >> 5) * kWmax;
    const int lane32 = threadIdx.x & 31;
    const int lane = threadIdx.x & (GK - 1);
    const int grp = lane32 / GK;
    const long long warp = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const long long nwarps = ((long long)gridDim.x * blockDim.x) >> 5;
    const int R = a.rounds, W = R * gpw;
    for (long long wb = a.q_begin + warp * W; wb < a.n_quartets; wb += nwarps * W) {  // warp-uniform
        if (R > 1) {
            for (int pos = lane32; pos < W; pos += 32) {
                unsigned key = (unsigned)pos;
                if (wb + pos < a.n_quartets) {
                    int b, k;
                    quartet_pair(a, wb + pos, b, k);
                    const PairHdr& hb = a.bhdr[b];
                    const PairHdr& hk = a.khdr[k];
                    const int t = herm_total(hv.B + hb.prim0, hb.nprim, hv.B + hk.prim0, hk.nprim, ptau);
                    key |= (unsigned)min(t, 0xFFFF) << 16;
                }
                wkeys[pos] = key;
            }
            __syncwarp();
            warp_bitonic_sort(wkeys, W, lane32);
        }
        for (int r = 0; r < R; r++) {
            const int s = r * gpw + grp;
            const long long q = wb + (R > 1 ? (long long)(wkeys[s] & 0xFFFFu) : (long long)s);
            const bool valid = q < a.n_quartets;
            PairHdr hb, hk;
            int b = 0, k = 0;
            if (valid) quartet_pair(a, q, b, k);
            hb = a.bhdr[b];
            hk = valid ? a.khdr[k] : hb;
            float pt = ptau;
            const bool live = valid && quartet_lives(a, hb, hk, pt);
            nprimq += C::template run<GK>(hb, hk, hv, a.boys64, a.P64, a.N, quartet_weight(hb, hk, a.same && b == k),
                                          a.Jt + cofs, a.Kt + cofs, nullptr, pt, lane, live);
        }
        __syncwarp();
    }
    if (a.prim_count) {
        const unsigned long long w = __reduce_add_sync(0xffffffffu, nprimq);
        if (lane32 == 0 && w) atomicAdd(a.prim_count, w);
    }
}

// -------------------------------------------------------------- warp kernel --
constexpr int kHermBatch = 32;  // primitive quartets whose R_N a warp holds at a time (one per lane)
constexpr int kHermSub = 4;     // of which the scaling products are expanded at a time

__host__ __device__ constexpr int herm_ncart(int l) { return (l + 1) * (l + 2) / 2; }

// One quartet of a warp's group, in shared memory.
struct HermQuartet {
    const HermPair *bp, *kp;
    const float *bB, *kB;
    const double* P;
    double *J, *K;
    double AB[3], CD[3], f;
    int N, bA, bB_, bC, bD, nb, nk;
    float ptau;
    int first;  // first primitive quartet of the quartet in the group's list
    int pad;
    __device__ __forceinline__ void set(const PairHdr& hb, const PairHdr& hk, const HermView& hv)
    {
        bp = hv.rec + hb.prim0;
        kp = hv.rec + hk.prim0;
        bB = hv.B + hb.prim0;
        kB = hv.B + hk.prim0;
        nb = hb.nprim;
        nk = hk.nprim;
        AB[0] = hb.ABx, AB[1] = hb.ABy, AB[2] = hb.ABz;
        CD[0] = hk.ABx, CD[1] = hk.ABy, CD[2] = hk.ABz;
        bA = hb.bfA, bB_ = hb.bfB, bC = hk.bfA, bD = hk.bfB;
    }
};

// Shared memory of one warp, in doubles.  Primitive phase: R_N, scalings and scaling products; contracted steps: per
// quartet H -> V -> X and U -> W.  U lies over the primitive phase's part; so does H for groups of one (NQ == 1),
// whose H is written when the primitive phase is over.  Then the density blocks, row prefixes and descriptors.
template <class C>
struct HermShape {
    static constexpr int NA = herm_ncart(C::LA), NB = herm_ncart(C::LB), NC = herm_ncart(C::LC), ND = herm_ncart(C::LD);
    static constexpr int NAB = NA * NB, NCD = NC * ND;
    static constexpr int NS = C::NBS * C::NKS, NSC = (C::NBS + C::NKS) | 1;
    static constexpr int cmax(int x, int y) { return x > y ? x : y; }
    static constexpr int oSc = kHermBatch * C::NRP, oS = oSc + kHermBatch * NSC, prim = oS + kHermSub * NS;
    static constexpr int nH = cmax(C::NACC, cmax(C::NE * C::NF, NAB * NCD));
    static constexpr int nU = cmax(C::NE * C::NKI, NAB * C::NF);
    static constexpr int oH = C::NQ == 1 ? 0 : cmax(prim, C::NQ * nU);
    static constexpr int oU = C::NQ == 1 ? nH : 0;
    static constexpr int nP = NC * ND + NA * NB + NB * ND + NA * NC + NB * NC + NA * ND;
    static constexpr int oP = C::NQ == 1 ? cmax(prim, nH + nU) : oH + C::NQ * nH;
    static constexpr int oPre = oP + C::NQ * nP;
    static constexpr int nPre = kMaxPrim * kMaxPrim;  // ints per quartet
    static constexpr int oQ = oPre + (C::NQ * nPre + 1) / 2;
    static constexpr int total = oQ + C::NQ * (int)(sizeof(HermQuartet) / 8);
    static constexpr size_t bytes = (size_t)total * sizeof(double);
};
static_assert(sizeof(HermQuartet) % 8 == 0, "HermQuartet in an array of doubles");

// the slot table's entry, read where it is used: hoisted out of the loop the entries would fill the registers
__device__ __forceinline__ unsigned herm_slot(const unsigned short* p)
{
    unsigned short v;
    asm volatile("ld.global.nc.u16 %0, [%1];" : "=h"(v) : "l"(p));
    return v;
}

// component-normalisation factor of component c of angular momentum l, squared (see comp_norm)
__device__ __forceinline__ double herm_norm2(int l, int c) { return l == 2 && (c == 0 || c == 3 || c == 5) ? 1.0 / 3.0 : 1.0; }

// A group of g <= C::NQ shell quartets by one warp.  fetch(i, descriptor), called by lane i < g, fills the
// descriptor of quartet i (nb = 0: nothing to do).  The primitive quartets of the whole group form one list, so that
// phase 1 fills its 32 lanes across quartet boundaries (a quartet keeps 33 of 81 on average: alone, every second
// batch of 32 would be nearly empty), and the contracted steps take (quartet, column) per lane, so that a ket with
// four Hermite items does not leave 28 lanes idle.
// part of nparts (groups of one): the warp takes batches part, part + nparts, ... of the quartet's primitive quartets
// and digests their share of the integrals, which is linear in them; launches with fewer quartets than the GPU has
// room for warps run several parts per quartet.
template <class C, class Fetch>
__device__ __forceinline__ int herm_warp(int g, Fetch fetch, const double2* __restrict__ etab, int ntype,
                                         const double* __restrict__ boys_tab, bool schwarz, int part, int nparts,
                                         double* __restrict__ sh)
{
    using Z = HermShape<C>;
    constexpr unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    HermQuartet* const Q = (HermQuartet*)(sh + Z::oQ);
    int* const pre = (int*)(sh + Z::oPre);
    if (lane < g) {
        Q[lane].nb = 0;
        fetch(lane, Q[lane]);
    }
    __syncwarp();
    // row ib of a quartet's staircase: the first c(ib) ket primitives; pre = exclusive prefix of c
    int T = 0;
    for (int q = 0; q < g; q++) {
        const float* __restrict__ const bB = Q[q].bB;
        const float* __restrict__ const kB = Q[q].kB;
        const int nb = Q[q].nb, nk = Q[q].nk;
        const float ptau = Q[q].ptau;
        int total = 0;
        for (int r0 = 0; r0 < nb; r0 += 32) {
            const int ib = r0 + lane;
            int c = 0;
            if (ib < nb) {
                const float Bb = bB[ib];
                while (c < nk && Bb * kB[c] >= ptau) c++;
            }
            int x = c;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(full, x, o);
                if (lane >= o) x += y;
            }
            if (ib < nb) pre[q * Z::nPre + ib] = total + x - c;
            total += __shfl_sync(full, x, 31);
        }
        if (lane == 0) Q[q].first = T;
        T += total;
    }
    __syncwarp();
    if (kHermBatch * part >= T) return 0;
    auto first = [&](int q) { return q < g ? Q[q].first : T; };
    double* const R = sh;
    double* const sc = sh + Z::oSc;
    double* const S = sh + Z::oS;
    double* const H = sh + Z::oH;
    double* const U = sh + Z::oU;
    double acc[C::NSLOT];
#pragma unroll
    for (int s = 0; s < C::NSLOT; s++) acc[s] = 0.0;
    auto flush = [&](int q) {
#pragma unroll
        for (int s = 0; s < C::NSLOT; s++) {
            if (32 * s + lane < C::NACC) H[q * Z::nH + 32 * s + lane] = acc[s];
            acc[s] = 0.0;
        }
    };
    int nq = 0, cur = 0;
    for (int base = kHermBatch * part; base < T; base += kHermBatch * nparts) {
        const bool live = base + lane < T;
        const int t = live ? base + lane : base;
        int q = 0;
        while (t >= first(q + 1)) q++;
        const int tq = t - Q[q].first;
        const int* const pq = pre + q * Z::nPre;
        int lo = 0, hi = Q[q].nb - 1;  // the row that holds tq (empty rows are last, with prefix total > tq)
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (pq[mid] <= tq)
                lo = mid;
            else
                hi = mid - 1;
        }
        nq += live;
        C::prim(Q[q].bp[lo], Q[q].kp[tq - pq[lo]], etab, ntype, boys_tab, live ? 1.0 : 0.0, R + lane * C::NRP,
                sc + lane * Z::NSC);
        __syncwarp();
        const int bend = min(kHermBatch, T - base);
        for (int pos = 0; pos < bend;) {  // one quartet's part of the batch at a time
            int end = bend;
            if constexpr (C::NQ > 1) {
                while (first(cur + 1) <= base + pos) cur++;
                end = min(bend, first(cur + 1) - base);
            }
            for (int i0 = pos; i0 < end; i0 += kHermSub) {
                for (int x = lane; x < kHermSub * Z::NS; x += 32) {
                    const int i = x / Z::NS, p = x - i * Z::NS;
                    const double* const si = sc + (i0 + i) * Z::NSC;
                    S[x] = i0 + i < end ? si[p / C::NKS] * si[C::NBS + p % C::NKS] : 0.0;
                }
                __syncwarp();
                const double* const Ri = R + i0 * C::NRP;
#pragma unroll
                for (int s = 0; s < C::NSLOT; s++) {
                    const unsigned ix = herm_slot(C::slots() + 32 * s + lane);
                    const double* const r = Ri + (ix >> 8);
                    const double* const p = S + (ix & 255u);
#pragma unroll
                    for (int i = 0; i < kHermSub; i++)  // past the batch's end: any finite R, S = 0
                        acc[s] = fma(p[i * Z::NS], r[min(i, kHermBatch - 1 - i0) * C::NRP], acc[s]);
                }
                __syncwarp();
            }
            if constexpr (C::NQ > 1) {
                if (nparts == 1 && base + end == first(cur + 1)) flush(cur);
            }
            pos = end;
        }
    }
    if (C::NQ == 1 || nparts > 1) flush(0);
    __syncwarp();
    for (int x = lane; x < g * C::NKI; x += 32) {
        const int q = x / C::NKI;
        C::bra(H + q * Z::nH, x - q * C::NKI, Q[q].AB[0], Q[q].AB[1], Q[q].AB[2], U + q * Z::nU);
    }
    __syncwarp();
    for (int x = lane; x < g * C::NE; x += 32) {  // V over H
        const int q = x / C::NE, e = x - q * C::NE;
        C::ket(U + q * Z::nU + e * C::NKI, Q[q].CD[0], Q[q].CD[1], Q[q].CD[2], H + q * Z::nH + e * C::NF);
    }
    __syncwarp();
    for (int x = lane; x < g * C::NF; x += 32) {  // W over U
        const int q = x / C::NF, f = x - q * C::NF;
        C::hrr_bra(H + q * Z::nH + f, Q[q].AB[0], Q[q].AB[1], Q[q].AB[2], U + q * Z::nU + f);
    }
    __syncwarp();
    for (int x = lane; x < g * Z::NAB; x += 32) {  // X[ab][cd] over V
        const int q = x / Z::NAB, ab = x - q * Z::NAB;
        C::hrr_ket(U + q * Z::nU + ab * C::NF, Q[q].CD[0], Q[q].CD[1], Q[q].CD[2], H + q * Z::nH + ab * Z::NCD);
    }
    __syncwarp();
    if constexpr (C::LA == C::LC && C::LB == C::LD) {
        if (schwarz) {  // Schwarz bound sqrt(max |(ab|ab)|) of normalised components, to the descriptor's J
            for (int q = 0; q < g; q++) {
                if (Q[q].nb == 0) continue;
                double m = 0.0;
                for (int ab = lane; ab < Z::NAB; ab += 32)
                    m = fmax(m, fabs(H[q * Z::nH + ab * Z::NCD + ab]) * herm_norm2(C::LA, ab / Z::NB) *
                                    herm_norm2(C::LB, ab % Z::NB));
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(full, m, o));
                if (lane == 0) *Q[q].J = sqrt(m);
            }
            __syncwarp();
            return nq;
        }
    }
    // digestion: one Fock element per lane and round, from the density blocks in shared memory
    double* const Ps = sh + Z::oP;
    constexpr int nCD = Z::NC * Z::ND, nAB = Z::NA * Z::NB, nBD = Z::NB * Z::ND, nAC = Z::NA * Z::NC, nBC = Z::NB * Z::NC;
    constexpr int pCD = 0, pAB = pCD + nCD, pBD = pAB + nAB, pAC = pBD + nBD, pBC = pAC + nAC, pAD = pBC + nBC;
    // block of element o in the order cd, ab, bd, ac, bc, ad: first functions, row length and position in it
    auto where = [&](const HermQuartet& d, int o, int& blk, int& u, int& v) -> size_t {
        int r0, c0, n1;
        if (o < pAB) blk = 0, o -= pCD, r0 = d.bC, c0 = d.bD, n1 = Z::ND;
        else if (o < pBD) blk = 1, o -= pAB, r0 = d.bA, c0 = d.bB_, n1 = Z::NB;
        else if (o < pAC) blk = 2, o -= pBD, r0 = d.bB_, c0 = d.bD, n1 = Z::ND;
        else if (o < pBC) blk = 3, o -= pAC, r0 = d.bA, c0 = d.bC, n1 = Z::NC;
        else if (o < pAD) blk = 4, o -= pBC, r0 = d.bB_, c0 = d.bC, n1 = Z::NC;
        else blk = 5, o -= pAD, r0 = d.bA, c0 = d.bD, n1 = Z::ND;
        u = o / n1;
        v = o - u * n1;
        return (size_t)(r0 + u) * d.N + c0 + v;
    };
    auto empty = [&](int q) { return first(q + 1) == Q[q].first; };  // no primitive quartet survived: H was not written
    for (int x = lane; x < g * Z::nP; x += 32) {
        const int q = x / Z::nP;
        int blk, u, v;
        if (!empty(q)) Ps[x] = Q[q].P[where(Q[q], x - q * Z::nP, blk, u, v)];
    }
    __syncwarp();
    constexpr int sA = Z::NB * Z::NCD, sB = Z::NCD, sC = Z::ND, sD = 1;  // strides of X
    for (int y = lane; y < g * Z::nP; y += 32) {
        const int q = y / Z::nP;
        if (empty(q)) continue;
        int blk, u, v;
        const size_t e = where(Q[q], y - q * Z::nP, blk, u, v);
        int x0, s1, s2, n1, n2, p0;
        switch (blk) {
            case 0: x0 = u * sC + v * sD, s1 = sA, s2 = sB, n1 = Z::NA, n2 = Z::NB, p0 = pAB; break;  // J_cd
            case 1: x0 = u * sA + v * sB, s1 = sC, s2 = sD, n1 = Z::NC, n2 = Z::ND, p0 = pCD; break;  // J_ab
            case 2: x0 = u * sB + v * sD, s1 = sA, s2 = sC, n1 = Z::NA, n2 = Z::NC, p0 = pAC; break;  // K_bd
            case 3: x0 = u * sA + v * sC, s1 = sB, s2 = sD, n1 = Z::NB, n2 = Z::ND, p0 = pBD; break;  // K_ac
            case 4: x0 = u * sB + v * sC, s1 = sA, s2 = sD, n1 = Z::NA, n2 = Z::ND, p0 = pAD; break;  // K_bc
            default: x0 = u * sA + v * sD, s1 = sB, s2 = sC, n1 = Z::NB, n2 = Z::NC, p0 = pBC; break;  // K_ad
        }
        double sum = 0.0;
        const double* p = Ps + q * Z::nP + p0;
        const double* const X = H + q * Z::nH + x0;
        for (int i = 0; i < n1; i++)
            for (int j = 0; j < n2; j++) sum = fma(X[i * s1 + j * s2], *p++, sum);
        red_add((blk < 2 ? Q[q].J : Q[q].K) + e, (blk < 2 ? 4.0 : 2.0) * Q[q].f * sum);
    }
    __syncwarp();  // the next group reuses the shared memory
    return nq;
}

// Units of `g` consecutive quartets (nparts == 1) or of one part of a quartet (g == 1).
template <class C>
__device__ __forceinline__ void herm_warp_kernel(const EriArgs& a, int g, int nparts, double* sh)
{
    if (a.bad && *a.bad) return;
    const size_t cofs = a.n_copies > 1 ? (size_t)(blockIdx.x % a.n_copies) * a.copy_stride : 0;
    const HermView hv = a.herm;
    const long long units = (a.n_quartets - a.q_begin + g - 1) / g * nparts;
    unsigned nprimq = 0;
    for (long long w = blockIdx.x; w < units; w += gridDim.x) {
        const long long q0 = a.q_begin + w / nparts * g;
        auto fetch = [&](int i, HermQuartet& d) {
            int b, k;
            quartet_pair(a, q0 + i, b, k);
            const PairHdr hb = a.bhdr[b], hk = a.khdr[k];
            d.ptau = (float)a.prim_tau;
            if (!quartet_lives(a, hb, hk, d.ptau)) return;
            d.set(hb, hk, hv);
            d.f = quartet_weight(hb, hk, a.same && b == k);
            d.P = a.P64;
            d.J = a.Jt + cofs;
            d.K = a.Kt + cofs;
            d.N = a.N;
        };
        nprimq += herm_warp<C>((int)min((long long)g, a.n_quartets - q0), fetch, hv.etab, hv.ntype, a.boys64, false,
                               (int)(w % nparts), nparts, sh);
    }
    if (a.prim_count) {
        const unsigned long long s = __reduce_add_sync(0xffffffffu, nprimq);
        if (threadIdx.x == 0 && s) atomicAdd(a.prim_count, s);
    }
}

// Schwarz bounds: item 0 of a pair is Q = sqrt(max |(ab|ab)|) of the contracted pair, item i > 0 the same bound of
// primitive pair i - 1 alone
struct SchwarzItem {
    PairHdr h;
    double* out;
    bool valid;
    __device__ __forceinline__ SchwarzItem(const SchwarzArgs& a, long long t)
    {
        valid = t < (long long)a.n * a.items;
        const int pid = a.ids[valid ? t / a.items : 0];
        const int item = valid ? (int)(t % a.items) : 0;
        h = a.pairs[pid];
        if (item > h.nprim) valid = false;
        out = a.Q + pid;
        if (item > 0 && valid) {
            h.prim0 += item - 1;
            h.nprim = 1;
            out = a.Bprim + h.prim0;
        }
    }
};

// Batched build: (molecule, bra, ket) of quartet q of the batch's index space.
__device__ __forceinline__ void batch_quartet(const BatchArgs& a, long long q, int& m, int& b, int& k)
{
    m = find_bra(a.mol_off, a.n_mol, q);
    const long long ql = q - a.mol_off[m];
    const MolClass& mc = a.mols[m];
    b = find_bra(mc.offsets, mc.n_bra, ql);
    k = (int)(ql - mc.offsets[b]);
}

// Thread form of the batched kernels: each warp sorts windows of its chunk (up to 256 quartets, of any molecules)
// by staircase length, as herm_thread_kernel does; unsorted, 20 of 32 lanes worked on the small molecules of a batch.
template <class C>
__device__ __forceinline__ void herm_thread_batch(const BatchArgs& a)
{
    __shared__ unsigned skeys[8 * kSortRounds * 32];
    unsigned* const wkeys = skeys + (threadIdx.x >> 5) * (kSortRounds * 32);
    const int wl = threadIdx.x & 31;
    const float ptau = (float)a.prim_tau;
    int W = 32;  // window: the largest power of two of warps' worth within the chunk
    while (W < kSortRounds * 32 && 2 * W <= a.chunk) W *= 2;
    for (;;) {
        unsigned long long base = 0;
        if (wl == 0) base = atomicAdd(a.counter, (unsigned long long)a.chunk);
        base = __shfl_sync(0xffffffffu, base, 0);
        if (base >= (unsigned long long)a.n_total) break;
        const long long end = min((long long)base + a.chunk, a.n_total);
        for (long long wb = (long long)base; wb < end; wb += W) {  // warp-uniform
            if (W > 32) {
                for (int pos = wl; pos < W; pos += 32) {
                    unsigned key = (unsigned)pos;
                    if (wb + pos < end) {
                        int m, b, k;
                        batch_quartet(a, wb + pos, m, b, k);
                        const MolClass& mc = a.mols[m];
                        const PairHdr &hb = mc.bhdr[b], &hk = mc.khdr[k];
                        const int t = herm_total(mc.herm.B + hb.prim0, hb.nprim, mc.herm.B + hk.prim0, hk.nprim, ptau);
                        key |= (unsigned)min(t, 0xFFFF) << 16;
                    }
                    wkeys[pos] = key;
                }
                __syncwarp();
                warp_bitonic_sort(wkeys, W, wl);
            }
            for (int r = 0; r < W / 32; r++) {
                const long long q = wb + (W > 32 ? (long long)(wkeys[32 * r + wl] & 0xFFFFu) : (long long)wl);
                const bool valid = q < end;
                int m, b, k;
                batch_quartet(a, valid ? q : wb, m, b, k);
                const MolClass& mc = a.mols[m];
                const PairHdr hb = mc.bhdr[b], hk = mc.khdr[k];
                C::template run<1>(hb, hk, mc.herm, a.boys64, mc.P64, mc.N, quartet_weight(hb, hk, mc.same && b == k),
                                   mc.Jt, mc.Kt, nullptr, ptau, 0, valid);
            }
            __syncwarp();
        }
    }
}

// Warp form of the batched kernels: groups of C::NQ quartets (of any molecules) from the device counter.
template <class C>
__device__ __forceinline__ void herm_warp_batch(const BatchArgs& a, double* sh)
{
    const HermView hv = a.mols[0].herm;  // the exponent table, shared by the molecules
    for (;;) {
        unsigned long long q0 = 0;
        if (threadIdx.x == 0) q0 = atomicAdd(a.counter, (unsigned long long)C::NQ);
        q0 = __shfl_sync(0xffffffffu, q0, 0);
        if (q0 >= (unsigned long long)a.n_total) break;
        auto fetch = [&](int i, HermQuartet& d) {
            int m, b, k;
            batch_quartet(a, (long long)q0 + i, m, b, k);
            const MolClass& mc = a.mols[m];
            const PairHdr hb = mc.bhdr[b], hk = mc.khdr[k];
            d.set(hb, hk, mc.herm);
            d.ptau = (float)a.prim_tau;
            d.f = quartet_weight(hb, hk, mc.same && b == k);
            d.P = mc.P64;
            d.J = mc.Jt;
            d.K = mc.Kt;
            d.N = mc.N;
        };
        herm_warp<C>((int)min((long long)C::NQ, a.n_total - (long long)q0), fetch, hv.etab, hv.ntype, a.boys64, false, 0,
                     1, sh);
    }
}

// Largest per-thread local memory of a list of kernels.
template <typename... K>
inline size_t herm_local_bytes(K... kernels)
{
    size_t m = 0;
    cudaFuncAttributes fa;
    for (const void* fn : {(const void*)kernels...})
        if (cudaFuncGetAttributes(&fa, fn) == cudaSuccess && fa.localSizeBytes > m) m = fa.localSizeBytes;
    cudaGetLastError();
    return m;
}

}  // namespace hf

// Kernels and host launchers of one class with a thread kernel: GL lanes per quartet in small launches.
#define HERM_THREAD_KERNELS(NAME, GL)                                                                        \
    template <int GK>                                                                                        \
    __global__ void __launch_bounds__(kEriThreads) k_herm_##NAME(const EriArgs a)                           \
    {                                                                                                        \
        herm_thread_kernel<HermThread_##NAME, GK>(a);                                                        \
    }                                                                                                        \
    void launch_herm_##NAME(const EriArgs& a, int grid, cudaStream_t s, int lanes)                          \
    {                                                                                                        \
        if (lanes > 1)                                                                                       \
            k_herm_##NAME<(GL)><<<grid, kEriThreads, 0, s>>>(a);                                             \
        else                                                                                                 \
            k_herm_##NAME<1><<<grid, kEriThreads, 0, s>>>(a);                                                \
    }

// ... and with a warp kernel: one warp per block, grid = quartets x parts (bounded).
#define HERM_WARP_KERNELS(NAME)                                                                              \
    __global__ void __launch_bounds__(32) k_hermw_##NAME(const EriArgs a, int g, int nparts)                \
    {                                                                                                        \
        extern __shared__ double hsh[];                                                                      \
        herm_warp_kernel<HermWarp_##NAME>(a, g, nparts, hsh);                                                \
    }                                                                                                        \
    int prepare_hermw_##NAME()                                                                               \
    {                                                                                                        \
        return cudaFuncSetAttribute(k_hermw_##NAME, cudaFuncAttributeMaxDynamicSharedMemorySize,             \
                                    (int)HermShape<HermWarp_##NAME>::bytes) == cudaSuccess ? 0 : -1;         \
    }                                                                                                        \
    void launch_hermw_##NAME(const EriArgs& a, cudaStream_t s, int group, int nparts)                       \
    {                                                                                                        \
        const int g = group ? HermWarp_##NAME::NQ : 1;                                                       \
        const long long units = (a.n_quartets - a.q_begin + g - 1) / g * nparts;                             \
        const int grid = (int)(units < (1 << 20) ? units : (1 << 20));                                       \
        k_hermw_##NAME<<<grid, 32, HermShape<HermWarp_##NAME>::bytes, s>>>(a, g, nparts);                    \
    }

// Schwarz bounds of a diagonal class: 8 lanes (thread form) per item or one warp per group of items.
#define HERM_THREAD_SCHWARZ(NAME)                                                                            \
    __global__ void __launch_bounds__(kEriThreads) k_schwarz_##NAME(const SchwarzArgs a)                    \
    {                                                                                                        \
        const long long t = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 3;                         \
        const SchwarzItem it(a, t);                                                                          \
        double qm = 0.0;                                                                                     \
        HermThread_##NAME::run<8>(it.h, it.h, a.herm, a.boys64, nullptr, 0, 1.0, nullptr, nullptr, &qm, 0.0f, \
                                  threadIdx.x & 7, it.valid);                                                \
        if (it.valid && (threadIdx.x & 7) == 0) *it.out = sqrt(qm);                                          \
    }                                                                                                        \
    void launch_schwarz_##NAME(const SchwarzArgs& a, int block, cudaStream_t s)                             \
    {                                                                                                        \
        const long long thr = (long long)a.n * a.items * 8;                                                  \
        if (thr > 0) k_schwarz_##NAME<<<(unsigned)((thr + block - 1) / block), block, 0, s>>>(a);            \
    }
#define HERM_WARP_SCHWARZ(NAME)                                                                              \
    __global__ void __launch_bounds__(32) k_schwarz_##NAME(const SchwarzArgs a)                             \
    {                                                                                                        \
        extern __shared__ double hsh[];                                                                      \
        constexpr int g = HermWarp_##NAME::NQ; /* items per warp: most are single primitive pairs */         \
        auto fetch = [&](int i, HermQuartet& d) {                                                            \
            const SchwarzItem it(a, (long long)blockIdx.x * g + i);                                          \
            if (!it.valid) return;                                                                           \
            d.set(it.h, it.h, a.herm);                                                                       \
            d.ptau = 0.0f;                                                                                   \
            d.J = it.out;                                                                                    \
        };                                                                                                   \
        herm_warp<HermWarp_##NAME>(g, fetch, a.herm.etab, a.herm.ntype, a.boys64, true, 0, 1, hsh);          \
    }                                                                                                        \
    void launch_schwarz_##NAME(const SchwarzArgs& a, int, cudaStream_t s)                                   \
    {                                                                                                        \
        if (cudaFuncSetAttribute(k_schwarz_##NAME, cudaFuncAttributeMaxDynamicSharedMemorySize,              \
                                 (int)HermShape<HermWarp_##NAME>::bytes) != cudaSuccess) return;             \
        const long long items = ((long long)a.n * a.items + HermWarp_##NAME::NQ - 1) / HermWarp_##NAME::NQ;  \
        if (items > 0) k_schwarz_##NAME<<<(unsigned)items, 32, HermShape<HermWarp_##NAME>::bytes, s>>>(a);   \
    }

// Batched build: warps take chunks of the batch's quartet index space from a device counter.
#define HERM_THREAD_BATCH(NAME)                                                                              \
    __global__ void __launch_bounds__(256) k_eri_batch_##NAME(const BatchArgs a)                            \
    {                                                                                                        \
        herm_thread_batch<HermThread_##NAME>(a);                                                             \
    }                                                                                                        \
    void launch_eri_batch_##NAME(const BatchArgs& a, int grid, int block, cudaStream_t s)                   \
    {                                                                                                        \
        k_eri_batch_##NAME<<<grid, block, 0, s>>>(a);                                                        \
    }
#define HERM_WARP_BATCH(NAME)                                                                                \
    __global__ void __launch_bounds__(32) k_eri_batch_##NAME(const BatchArgs a)                             \
    {                                                                                                        \
        extern __shared__ double hsh[];                                                                      \
        herm_warp_batch<HermWarp_##NAME>(a, hsh);                                                            \
    }                                                                                                        \
    void launch_eri_batch_##NAME(const BatchArgs& a, int grid, int, cudaStream_t s)                         \
    {                                                                                                        \
        k_eri_batch_##NAME<<<grid, 32, HermShape<HermWarp_##NAME>::bytes, s>>>(a);                           \
    }                                                                                                        \
    int prepare_batch_##NAME()                                                                               \
    {                                                                                                        \
        return cudaFuncSetAttribute(k_eri_batch_##NAME, cudaFuncAttributeMaxDynamicSharedMemorySize,         \
                                    (int)HermShape<HermWarp_##NAME>::bytes) == cudaSuccess ? 0 : -1;         \
    }
