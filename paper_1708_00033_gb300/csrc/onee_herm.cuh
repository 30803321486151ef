// One-electron matrices S and H = T + V of one pair class, one warp per shell pair.
//
//   S, T: per primitive pair the 1-D overlaps of the three directions,
//      s_{i+1,j} = PA s_ij + (i s_{i-1,j} + j s_{i,j-1}) / 2p (and the same with PB on the second index),
//      s_00 = sqrt(pi/p) exp(-mu X_AB^2); one (primitive pair, direction) per lane, then one component per lane with
//      T as half the gradient overlap, t_ij = (i j s_{i-1,j-1} - 2b i s_{i-1,j+1} - 2a j s_{i+1,j-1} + 4ab s_{i+1,j+1}) / 2;
//   V: Hermite Coulomb integrals of the nuclei (gen_herm.py), lanes over nuclei (and over primitive pairs when there
//      are fewer nuclei than lanes), contracted over the primitives before the pair geometry enters.
// One thread per shell pair walked every primitive pair and nucleus through arrays indexed at run time (local memory)
// and took 12.4 ms of a 20-water set-up; these six kernels, run beside the Schwarz bounds, take 0.3 to 0.5 ms each.
#pragma once
#include <math.h>

#include "eri_herm.cuh"

namespace hf {

constexpr int kOneEChunk = 10;  // primitive pairs whose 1-D tables a warp holds: 30 lanes make them

template <int L>
struct CartPow {
    int x[herm_ncart(L)], y[herm_ncart(L)], z[herm_ncart(L)];
    constexpr CartPow() : x(), y(), z()
    {
        int k = 0;
        for (int a = L; a >= 0; a--)
            for (int b = L - a; b >= 0; b--, k++) {
                x[k] = a;
                y[k] = b;
                z[k] = L - a - b;
            }
    }
    __device__ __forceinline__ int get(int c, int d) const { return d == 0 ? x[c] : d == 1 ? y[c] : z[c]; }
};

template <class C>
__device__ __forceinline__ void one_electron_pair(const OneEArgs& a, int pid, double* __restrict__ sh)
{
    constexpr int LA = C::LA, LB = C::LB, NA = herm_ncart(LA), NB = herm_ncart(LB), NAB = NA * NB;
    constexpr int U = LA + 2, W = LB + 2, NT = 3 * U * W;  // 1-D table of a primitive pair
    constexpr CartPow<LA> pa{};
    constexpr CartPow<LB> pb{};
    const int lane = threadIdx.x & 31;
    const PairHdr h = a.pairs[pid];
    const int nb_prim = a.nprim[h.B];
    const double* const ea = a.exps + a.prim0[h.A];
    const double* const eb = a.exps + a.prim0[h.B];
    const double* const ca = a.cn + a.prim0[h.A];
    const double* const cb = a.cn + a.prim0[h.B];
    const double AB[3] = {h.ABx, h.ABy, h.ABz};
    const double R2 = AB[0] * AB[0] + AB[1] * AB[1] + AB[2] * AB[2];
    // primitive pairs whose Gaussian-product factor exp(-x), x = ab/(a+b) |AB|^2, is below exp(-60) ~ 9e-27 are
    // skipped.  Functions and primitives are normalised, so with two contraction coefficients below 10 each, the
    // components' polynomials ((4 x)^2 at most for two d functions, 6e4 here) and 1e6 for total charge times
    // 2 sqrt(p), what is dropped from an element stays below 6e-14, a hundredth of the 1e-11 parity tolerance
    auto skipped = [&](double x, double y) { return x * y / (x + y) * R2 > 60.0; };
    double sa[(NAB + 31) / 32], ta[(NAB + 31) / 32];
#pragma unroll
    for (int i = 0; i < (NAB + 31) / 32; i++) sa[i] = ta[i] = 0.0;
    for (int k0 = 0; k0 < h.nprim; k0 += kOneEChunk) {
        const int nk = min(kOneEChunk, h.nprim - k0);
        if (lane < 3 * nk) {
            const int k = k0 + lane / 3, d = lane % 3;
            const double x = ea[k / nb_prim], y = eb[k % nb_prim];
            const double ip = 1.0 / (x + y), X = AB[d], o2p = 0.5 * ip;
            const double PA = -y * ip * X, PB = x * ip * X;
            double s[U][W];
            s[0][0] = skipped(x, y) ? 0.0 : sqrt(M_PI * ip) * exp(-x * y * ip * X * X);
#pragma unroll
            for (int v = 1; v < W; v++)
                s[0][v] = PB * s[0][v - 1] + (v >= 2 ? o2p * (v - 1) * s[0][v - 2] : 0.0);
#pragma unroll
            for (int u = 1; u < U; u++)
#pragma unroll
                for (int v = 0; v < W; v++)
                    s[u][v] = PA * s[u - 1][v] + o2p * ((u >= 2 ? (u - 1) * s[u - 2][v] : 0.0) + (v >= 1 ? v * s[u - 1][v - 1] : 0.0));
            double* const o = sh + (lane / 3) * NT + d * U * W;
#pragma unroll
            for (int u = 0; u < U; u++)
#pragma unroll
                for (int v = 0; v < W; v++) o[u * W + v] = s[u][v];
        }
        __syncwarp();
#pragma unroll
        for (int i = 0; i < (NAB + 31) / 32; i++) {
            const int c = lane + 32 * i;
            if (c < NAB) {
                const int c1 = c / NB, c2 = c % NB;
                for (int kk = 0; kk < nk; kk++) {
                    const int k = k0 + kk;
                    const double x = ea[k / nb_prim], y = eb[k % nb_prim];
                    const double cc = ca[k / nb_prim] * cb[k % nb_prim];
                    double sd[3], td[3];
#pragma unroll
                    for (int d = 0; d < 3; d++) {
                        const int u = pa.get(c1, d), v = pb.get(c2, d);
                        const double* const s = sh + kk * NT + d * U * W + u * W + v;
                        double t = 4.0 * x * y * s[W + 1];
                        if (u > 0) t -= 2.0 * y * u * s[-W + 1];
                        if (v > 0) t -= 2.0 * x * v * s[W - 1];
                        if (u > 0 && v > 0) t += (double)(u * v) * s[-W - 1];
                        sd[d] = s[0];
                        td[d] = 0.5 * t;
                    }
                    sa[i] += cc * sd[0] * sd[1] * sd[2];
                    ta[i] += cc * (td[0] * sd[1] * sd[2] + sd[0] * td[1] * sd[2] + sd[0] * sd[1] * td[2]);
                }
            }
        }
        __syncwarp();
    }
    // nuclear attraction
    const HermPair* const rec = a.herm.rec + h.prim0;
    int gn = 32;  // lanes over nuclei; the others take further primitive pairs
    while (gn > 1 && gn / 2 >= a.n_atoms) gn >>= 1;
    const int nslot = lane & (gn - 1), pslot = lane / gn, np = 32 / gn;
    double acc[C::NI];
#pragma unroll
    for (int i = 0; i < C::NI; i++) acc[i] = 0.0;
    for (int k = pslot; k < h.nprim; k += np) {
        const HermPair bp = rec[k];
        const double y = 0.5 * bp.u, x = 0.5 * bp.v - y;
        if (skipped(x, y)) continue;
        double RS[C::NR];
#pragma unroll
        for (int i = 0; i < C::NR; i++) RS[i] = 0.0;
        for (int nuc = nslot; nuc < a.n_atoms; nuc += gn)
            C::nucleus(bp, a.xyz[3 * nuc], a.xyz[3 * nuc + 1], a.xyz[3 * nuc + 2], a.Z[nuc], a.boys64, RS);
        C::scale(bp, -kNuclearPrefactor * bp.K, RS, acc);  // the record's sqrt(2) pi^(5/4) / p to -2 pi / p
    }
#pragma unroll
    for (int i = 0; i < C::NI; i++)
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) acc[i] += __shfl_xor_sync(0xffffffffu, acc[i], o);
    if (lane == 0) C::finish(acc, h.ABx, h.ABy, h.ABz, sh);
    __syncwarp();
#pragma unroll
    for (int i = 0; i < (NAB + 31) / 32; i++) {
        const int c = lane + 32 * i;
        // the two halves of a diagonal block (A == B) mirror each other: one of them writes both
        if (c < NAB && (h.A != h.B || c / NB >= c % NB)) {
            const int r = h.bfA + c / NB, q = h.bfB + c % NB;
            const double nrm = a.comp_norm[r] * a.comp_norm[q];
            a.S[(size_t)r * a.N + q] = a.S[(size_t)q * a.N + r] = nrm * sa[i];
            a.H[(size_t)r * a.N + q] = a.H[(size_t)q * a.N + r] = nrm * (ta[i] + sh[c]);
        }
    }
}

}  // namespace hf

#define ONEE_KERNEL(LA_, LB_)                                                                                \
    __global__ void __launch_bounds__(32) k_one_electron_##LA_##LB_(const OneEArgs a)                       \
    {                                                                                                        \
        constexpr int NT = 3 * (LA_ + 2) * (LB_ + 2) * kOneEChunk;                                           \
        constexpr int NAB = herm_ncart(LA_) * herm_ncart(LB_);                                               \
        __shared__ double sh[NT > NAB ? NT : NAB];                                                           \
        one_electron_pair<OneE_##LA_##LB_>(a, a.ids[blockIdx.x], sh);                                        \
    }                                                                                                        \
    int launch_one_electron_##LA_##LB_(const OneEArgs& a, cudaStream_t s)                                   \
    {                                                                                                        \
        if (a.n > 0) k_one_electron_##LA_##LB_<<<a.n, 32, 0, s>>>(a);                                        \
        return cudaGetLastError() == cudaSuccess ? 0 : -1;                                                   \
    }
