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
// One quartet per lane group of GK lanes.  Each warp sorts its window of quartets by staircase length and runs
// it in rounds, as the Obara-Saika kernels do (ERI_KERNEL_BODY).
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
    int R = 1;
    while (R < kSortRounds && (long long)(2 * R) * gpw * nwarps * 2 <= a.n_quartets - a.q_begin) R *= 2;
    const int W = R * gpw;
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

// Shared memory of one warp, in doubles: the primitive phase's R_N, scalings and scaling products, and in the
// same space the contracted steps' H -> V -> X and U -> W; then the density blocks and the row prefix.
template <class C>
struct HermShape {
    static constexpr int NA = herm_ncart(C::LA), NB = herm_ncart(C::LB), NC = herm_ncart(C::LC), ND = herm_ncart(C::LD);
    static constexpr int NAB = NA * NB, NCD = NC * ND;
    static constexpr int NS = C::NBS * C::NKS, NSC = (C::NBS + C::NKS) | 1;
    static constexpr int cmax(int x, int y) { return x > y ? x : y; }
    static constexpr int oSc = kHermBatch * C::NRP, oS = oSc + kHermBatch * NSC, prim = oS + kHermSub * NS;
    static constexpr int nH = cmax(C::NACC, cmax(C::NE * C::NF, NAB * NCD));
    static constexpr int oU = nH, nU = cmax(C::NE * C::NKI, NAB * C::NF);
    static constexpr int oP = cmax(prim, oU + nU);
    static constexpr int nP = NC * ND + NA * NB + NB * ND + NA * NC + NB * NC + NA * ND;
    static constexpr int oPre = oP + nP;
    static constexpr int total = oPre + (kMaxPrim * kMaxPrim + 2) / 2 + 1;
    static constexpr size_t bytes = (size_t)total * sizeof(double);
};

// the slot table's entry, read where it is used: hoisted out of the loop the entries would fill the registers
__device__ __forceinline__ unsigned herm_slot(const unsigned short* p)
{
    unsigned short v;
    asm volatile("ld.global.nc.u16 %0, [%1];" : "=h"(v) : "l"(p));
    return v;
}

// component-normalisation factor of component c of angular momentum l, squared (see comp_norm)
__device__ __forceinline__ double herm_norm2(int l, int c) { return l == 2 && (c == 0 || c == 3 || c == 5) ? 1.0 / 3.0 : 1.0; }

// One shell quartet by one warp (uniform arguments).  part of nparts: the warp takes batches part,
// part + nparts, ... of the primitive quartets and digests their share of the integrals, which is linear in
// them; launches with fewer quartets than the GPU has room for warps run several parts per quartet.
template <class C>
__device__ __forceinline__ int herm_warp(const PairHdr& hb, const PairHdr& hk, const HermView& hv,
                                         const double* __restrict__ boys_tab, const double* __restrict__ Pd, int N,
                                         double f, double* __restrict__ Jt, double* __restrict__ Kt, double* qout,
                                         float ptau, int part, int nparts, double* __restrict__ sh)
{
    using Z = HermShape<C>;
    constexpr unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const HermPair* __restrict__ bpp = hv.rec + hb.prim0;
    const HermPair* __restrict__ kpp = hv.rec + hk.prim0;
    const float* __restrict__ bB = hv.B + hb.prim0;
    const float* __restrict__ kB = hv.B + hk.prim0;
    int* const pre = (int*)(sh + Z::oPre);
    // row ib of the staircase: the first c(ib) ket primitives; pre = exclusive prefix of c
    int total = 0;
    for (int r0 = 0; r0 < hb.nprim; r0 += 32) {
        const int ib = r0 + lane;
        int c = 0;
        if (ib < hb.nprim) {
            const float Bb = bB[ib];
            while (c < hk.nprim && Bb * kB[c] >= ptau) c++;
        }
        int x = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(full, x, o);
            if (lane >= o) x += y;
        }
        if (ib < hb.nprim) pre[ib] = total + x - c;
        total += __shfl_sync(full, x, 31);
    }
    __syncwarp();
    if (32 * part >= total) return 0;
    double* const R = sh;
    double* const sc = sh + Z::oSc;
    double* const S = sh + Z::oS;
    double acc[C::NSLOT];
#pragma unroll
    for (int s = 0; s < C::NSLOT; s++) acc[s] = 0.0;
    int nq = 0;
    for (int base = kHermBatch * part; base < total; base += kHermBatch * nparts) {
        const bool live = base + lane < total;
        const int t = live ? base + lane : base;
        int lo = 0, hi = hb.nprim - 1;  // the row that holds t (empty rows are last, with prefix total > t)
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (pre[mid] <= t)
                lo = mid;
            else
                hi = mid - 1;
        }
        nq += live;
        C::prim(bpp[lo], kpp[t - pre[lo]], hv.etab, hv.ntype, boys_tab, live ? 1.0 : 0.0, R + lane * C::NRP,
                sc + lane * Z::NSC);
        __syncwarp();
        const int cnt = min(kHermBatch, total - base);
        for (int i0 = 0; i0 < cnt; i0 += kHermSub) {
            for (int x = lane; x < kHermSub * Z::NS; x += 32) {
                const int i = x / Z::NS, p = x - i * Z::NS;
                const double* const si = sc + (i0 + i) * Z::NSC;
                S[x] = si[p / C::NKS] * si[C::NBS + p % C::NKS];
            }
            __syncwarp();
            const double* const Ri = R + i0 * C::NRP;
#pragma unroll
            for (int s = 0; s < C::NSLOT; s++) {
                const unsigned ix = herm_slot(C::slots() + 32 * s + lane);
                const double* const r = Ri + (ix >> 8);
                const double* const p = S + (ix & 255u);
#pragma unroll
                for (int i = 0; i < kHermSub; i++) acc[s] = fma(p[i * Z::NS], r[i * C::NRP], acc[s]);
            }
            __syncwarp();
        }
    }
    double* const H = sh;
    double* const U = sh + Z::oU;
#pragma unroll
    for (int s = 0; s < C::NSLOT; s++)
        if (32 * s + lane < C::NACC) H[32 * s + lane] = acc[s];
    __syncwarp();
    const double ABx = hb.ABx, ABy = hb.ABy, ABz = hb.ABz;
    const double CDx = hk.ABx, CDy = hk.ABy, CDz = hk.ABz;
    for (int j = lane; j < C::NKI; j += 32) C::bra(H, j, ABx, ABy, ABz, U);
    __syncwarp();
    double* const V = sh;  // H is done
    for (int e = lane; e < C::NE; e += 32) C::ket(U + e * C::NKI, CDx, CDy, CDz, V + e * C::NF);
    __syncwarp();
    double* const Wd = U;  // U is done
    for (int g = lane; g < C::NF; g += 32) C::hrr_bra(V + g, ABx, ABy, ABz, Wd + g);
    __syncwarp();
    double* const X = sh;  // V is done; X[ab][cd]
    for (int ab = lane; ab < Z::NAB; ab += 32) C::hrr_ket(Wd + ab * C::NF, CDx, CDy, CDz, X + ab * Z::NCD);
    __syncwarp();
    if constexpr (C::LA == C::LC && C::LB == C::LD) {
        if (qout) {  // Schwarz bound: max |(ab|ab)| of normalised components
            double m = 0.0;
            for (int ab = lane; ab < Z::NAB; ab += 32)
                m = fmax(m, fabs(X[ab * Z::NCD + ab]) * herm_norm2(C::LA, ab / Z::NB) * herm_norm2(C::LB, ab % Z::NB));
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(full, m, o));
            if (lane == 0) *qout = m;
            __syncwarp();
            return nq;
        }
    }
    // digestion: one Fock element per lane and round, from the density blocks in shared memory
    const int bA = hb.bfA, bB_ = hb.bfB, bC = hk.bfA, bD = hk.bfB;
    double* const Ps = sh + Z::oP;
    constexpr int nCD = Z::NC * Z::ND, nAB = Z::NA * Z::NB, nBD = Z::NB * Z::ND, nAC = Z::NA * Z::NC, nBC = Z::NB * Z::NC,
                  nAD = Z::NA * Z::ND;
    constexpr int pCD = 0, pAB = pCD + nCD, pBD = pAB + nAB, pAC = pBD + nBD, pBC = pAC + nAC, pAD = pBC + nBC;
    // block of element o in the order cd, ab, bd, ac, bc, ad: first functions, row length and position in it
    auto where = [&](int o, int& blk, int& u, int& v) -> size_t {
        int r0, c0, n1;
        if (o < pAB) blk = 0, o -= pCD, r0 = bC, c0 = bD, n1 = Z::ND;
        else if (o < pBD) blk = 1, o -= pAB, r0 = bA, c0 = bB_, n1 = Z::NB;
        else if (o < pAC) blk = 2, o -= pBD, r0 = bB_, c0 = bD, n1 = Z::ND;
        else if (o < pBC) blk = 3, o -= pAC, r0 = bA, c0 = bC, n1 = Z::NC;
        else if (o < pAD) blk = 4, o -= pBC, r0 = bB_, c0 = bC, n1 = Z::NC;
        else blk = 5, o -= pAD, r0 = bA, c0 = bD, n1 = Z::ND;
        u = o / n1;
        v = o - u * n1;
        return (size_t)(r0 + u) * N + c0 + v;
    };
    for (int o = lane; o < Z::nP; o += 32) {
        int blk, u, v;
        Ps[o] = Pd[where(o, blk, u, v)];
    }
    __syncwarp();
    constexpr int sA = Z::NB * Z::NCD, sB = Z::NCD, sC = Z::ND, sD = 1;  // strides of X
    for (int o = lane; o < Z::nP; o += 32) {
        int blk, u, v;
        const size_t g = where(o, blk, u, v);
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
        const double* p = Ps + p0;
        for (int i = 0; i < n1; i++)
            for (int j = 0; j < n2; j++) sum = fma(X[x0 + i * s1 + j * s2], *p++, sum);
        red_add((blk < 2 ? Jt : Kt) + g, (blk < 2 ? 4.0 : 2.0) * f * sum);
    }
    __syncwarp();  // the next quartet reuses the shared memory
    return nq;
}

template <class C>
__device__ __forceinline__ void herm_warp_kernel(const EriArgs& a, int nparts, double* sh)
{
    if (a.bad && *a.bad) return;
    const size_t cofs = a.n_copies > 1 ? (size_t)(blockIdx.x % a.n_copies) * a.copy_stride : 0;
    const HermView hv = a.herm;
    const long long units = (a.n_quartets - a.q_begin) * nparts;
    unsigned nprimq = 0;
    for (long long w = blockIdx.x; w < units; w += gridDim.x) {
        const long long q = a.q_begin + w / nparts;
        int b, k;
        quartet_pair(a, q, b, k);
        const PairHdr hb = a.bhdr[b], hk = a.khdr[k];
        float pt = (float)a.prim_tau;
        if (!quartet_lives(a, hb, hk, pt)) continue;
        nprimq += herm_warp<C>(hb, hk, hv, a.boys64, a.P64, a.N, quartet_weight(hb, hk, a.same && b == k), a.Jt + cofs,
                               a.Kt + cofs, nullptr, pt, (int)(w % nparts), nparts, sh);
    }
    if (a.prim_count) {
        const unsigned long long s = __reduce_add_sync(0xffffffffu, nprimq);
        if (threadIdx.x == 0 && s) atomicAdd(a.prim_count, s);
    }
}

// item 0 of a pair: its contracted bound; item i > 0: primitive pair i - 1 alone (see SCHWARZ_KERNEL)
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

// Work queue of a batched build (see ERI_BATCH_KERNEL): (molecule, bra, ket) of quartet q.
__device__ __forceinline__ void batch_quartet(const BatchArgs& a, long long q, int& m, int& b, int& k)
{
    m = find_bra(a.mol_off, a.n_mol, q);
    const long long ql = q - a.mol_off[m];
    const MolClass& mc = a.mols[m];
    b = find_bra(mc.offsets, mc.n_bra, ql);
    k = (int)(ql - mc.offsets[b]);
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
    __global__ void __launch_bounds__(32) k_hermw_##NAME(const EriArgs a, int nparts)                       \
    {                                                                                                        \
        extern __shared__ double hsh[];                                                                      \
        herm_warp_kernel<HermWarp_##NAME>(a, nparts, hsh);                                                   \
    }                                                                                                        \
    int prepare_hermw_##NAME()                                                                               \
    {                                                                                                        \
        return cudaFuncSetAttribute(k_hermw_##NAME, cudaFuncAttributeMaxDynamicSharedMemorySize,             \
                                    (int)HermShape<HermWarp_##NAME>::bytes) == cudaSuccess ? 0 : -1;         \
    }                                                                                                        \
    void launch_hermw_##NAME(const EriArgs& a, int grid, cudaStream_t s, int nparts)                        \
    {                                                                                                        \
        k_hermw_##NAME<<<grid, 32, HermShape<HermWarp_##NAME>::bytes, s>>>(a, nparts);                       \
    }

// Schwarz bounds of a diagonal class: 8 lanes (thread form) or one warp per item.
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
        const SchwarzItem it(a, blockIdx.x);                                                                 \
        if (!it.valid) return; /* block-uniform */                                                           \
        double qm = 0.0;                                                                                     \
        herm_warp<HermWarp_##NAME>(it.h, it.h, a.herm, a.boys64, nullptr, 0, 1.0, nullptr, nullptr, &qm, 0.0f, \
                                   0, 1, hsh);                                                               \
        if (threadIdx.x == 0) *it.out = sqrt(qm);                                                            \
    }                                                                                                        \
    void launch_schwarz_##NAME(const SchwarzArgs& a, int, cudaStream_t s)                                   \
    {                                                                                                        \
        if (cudaFuncSetAttribute(k_schwarz_##NAME, cudaFuncAttributeMaxDynamicSharedMemorySize,              \
                                 (int)HermShape<HermWarp_##NAME>::bytes) != cudaSuccess) return;             \
        const long long items = (long long)a.n * a.items;                                                    \
        if (items > 0) k_schwarz_##NAME<<<(unsigned)items, 32, HermShape<HermWarp_##NAME>::bytes, s>>>(a);   \
    }

// Batched build: warps take chunks of the batch's quartet index space from a device counter.
#define HERM_THREAD_BATCH(NAME)                                                                              \
    __global__ void __launch_bounds__(256) k_eri_batch_##NAME(const BatchArgs a)                            \
    {                                                                                                        \
        const int wl = threadIdx.x & 31;                                                                     \
        for (;;) {                                                                                           \
            unsigned long long base = 0;                                                                     \
            if (wl == 0) base = atomicAdd(a.counter, (unsigned long long)a.chunk);                          \
            base = __shfl_sync(0xffffffffu, base, 0);                                                        \
            if (base >= (unsigned long long)a.n_total) break;                                                \
            const long long end = min((long long)base + a.chunk, a.n_total);                                 \
            for (long long wq = (long long)base; wq < end; wq += 32) { /* warp-uniform */                   \
                const bool valid = wq + wl < end;                                                            \
                int m, b, k;                                                                                 \
                batch_quartet(a, valid ? wq + wl : wq, m, b, k);                                             \
                const MolClass& mc = a.mols[m];                                                              \
                const PairHdr hb = mc.bhdr[b], hk = mc.khdr[k];                                              \
                HermThread_##NAME::run<1>(hb, hk, mc.herm, a.boys64, mc.P64, mc.N,                           \
                                          quartet_weight(hb, hk, mc.same && b == k), mc.Jt, mc.Kt, nullptr,  \
                                          (float)a.prim_tau, 0, valid);                                      \
            }                                                                                                \
        }                                                                                                    \
    }                                                                                                        \
    void launch_eri_batch_##NAME(const BatchArgs& a, int grid, int block, cudaStream_t s)                   \
    {                                                                                                        \
        k_eri_batch_##NAME<<<grid, block, 0, s>>>(a);                                                        \
    }
#define HERM_WARP_BATCH(NAME)                                                                                \
    __global__ void __launch_bounds__(32) k_eri_batch_##NAME(const BatchArgs a)                             \
    {                                                                                                        \
        extern __shared__ double hsh[];                                                                      \
        for (;;) {                                                                                           \
            unsigned long long q = 0;                                                                        \
            if (threadIdx.x == 0) q = atomicAdd(a.counter, 1ull);                                            \
            q = __shfl_sync(0xffffffffu, q, 0);                                                              \
            if (q >= (unsigned long long)a.n_total) break;                                                   \
            int m, b, k;                                                                                     \
            batch_quartet(a, (long long)q, m, b, k);                                                         \
            const MolClass& mc = a.mols[m];                                                                  \
            const PairHdr hb = mc.bhdr[b], hk = mc.khdr[k];                                                  \
            herm_warp<HermWarp_##NAME>(hb, hk, mc.herm, a.boys64, mc.P64, mc.N,                              \
                                       quartet_weight(hb, hk, mc.same && b == k), mc.Jt, mc.Kt, nullptr,     \
                                       (float)a.prim_tau, 0, 1, hsh);                                        \
        }                                                                                                    \
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
