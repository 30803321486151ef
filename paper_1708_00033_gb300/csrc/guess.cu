// Learned initial guess: a small MLP maps per-atom-pair geometric features
// to the corresponding block of the density matrix.  Training and inference
// run in these kernels: BF16 weights (with FP32 master copies for Adam),
// FP32 activations and FP32 accumulation.
//
//   features (16): R, u_x, u_y, u_z, the 9 products u_i u_j, one-hot of the
//                  element pair (O-O, O-H, H-H); u = (r_b - r_a) / R, zero
//                  for on-site pairs (a == b, R = 0)
//   network:       16 -> 256 (SiLU) -> 256 (SiLU) -> 325 = 225 (O-O head)
//                  + 75 (O-H head) + 25 (H-H head); a sample's loss only sees
//                  its own head
//   density:       each unordered pair's predicted block is placed at
//                  P[a, b] (and its transpose at P[b, a]); on-site blocks are
//                  symmetrised; P is finally scaled so that tr(PS) = N_e.
#include <cuda_bf16.h>
#include <math.h>
#include <string.h>

#include <algorithm>
#include <string>
#include <vector>

#include "hf_internal.h"

namespace hf {
namespace {

constexpr int kFeat = 16;
constexpr int kWidth = 256;
constexpr int kOut = 325;
__host__ __device__ __forceinline__ int head_off(int h) { return h == 0 ? 0 : (h == 1 ? 225 : 300); }
__host__ __device__ __forceinline__ int head_rows(int h) { return h == 2 ? 5 : 15; }
__host__ __device__ __forceinline__ int head_cols(int h) { return h == 0 ? 15 : 5; }

__device__ __forceinline__ float silu(float z) { return z / (1.0f + __expf(-z)); }
__device__ __forceinline__ float dsilu(float z)
{
    const float s = 1.0f / (1.0f + __expf(-z));
    return s * (1.0f + z * (1.0f - s));
}

constexpr int kOutLd = 328;  // row length of the output gradients (325 padded to 16 bytes, zero-filled)

// ------------------------------------------------------------- MLP products --
// Every product of the network is a 64 x 64 tile per block of 256 threads, 4 x 4 outputs per thread, FP32
// FMAs on k-major shared tiles read with 16-byte loads, the next k-tile's global loads in flight meanwhile.
// FP32 stays on the FMA units: activations and gradients are FP32, the whole step is 1.9 GFLOP (25 us at the
// FP32 rate), and what bound it was elsewhere: weight gradients as 4 to 24 blocks walking the whole minibatch,
// column sums by one thread per column, and separate passes for the loss, its gradient and SiLU'.  These are
// now epilogues or part of the weight-gradient product, which is split over the minibatch.
// Measured: a training step on 2,048 samples 1,345 us before, 173 us with these kernels (127 us of kernel time).
constexpr int kGT = 64, kGK = 32, kGLd = kGT + 4;

struct GemmTile {
    float a[kGK][kGLd];
    float b[kGK][kGLd];
};

// 8 values of a 64 x 32 tile per thread: rows of op(A) with k contiguous (row = e / 4, k = 8 (e % 4)) or
// k-rows with the tile's 64 columns contiguous (k = e / 8, column = 8 (e % 8)), e = threadIdx.x.
template <typename T>
__device__ __forceinline__ void load8(const T* __restrict__ p, int n_ok, bool vec, float* v)
{
    if constexpr (sizeof(T) == 4) {
        if (vec && n_ok >= 8) {
            const float4 x = *(const float4*)p, y = *(const float4*)(p + 4);
            v[0] = x.x, v[1] = x.y, v[2] = x.z, v[3] = x.w, v[4] = y.x, v[5] = y.y, v[6] = y.z, v[7] = y.w;
            return;
        }
#pragma unroll
        for (int i = 0; i < 8; i++) v[i] = i < n_ok ? (float)p[i] : 0.0f;
    } else {
        if (vec && n_ok >= 8) {
            const uint4 x = *(const uint4*)p;
            const unsigned w[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
            for (int i = 0; i < 4; i++) {
                v[2 * i] = __uint_as_float(w[i] << 16);
                v[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u);
            }
            return;
        }
#pragma unroll
        for (int i = 0; i < 8; i++) v[i] = i < n_ok ? __bfloat162float(p[i]) : 0.0f;
    }
}

// acc += op(A)[m0.., k0..k1) op(B)[k0..k1), n0..).  AK: A stored [M][K] (k contiguous), else [K][M]; BK the same
// for B ([N][K] or [K][N]).  vecA / vecB: 16-byte loads allowed (base and row length aligned).  colsum: threads
// below 64 also add up their column of op(A) over k.
template <bool AK, bool BK, typename TB>
__device__ __forceinline__ void tile_gemm(GemmTile& sm, float (&acc)[4][4], const float* __restrict__ A, int lda, int M,
                                          int m0, bool vecA, const TB* __restrict__ B, int ldb, int N, int n0, bool vecB,
                                          int k0, int k1, float* colsum)
{
    const int e = threadIdx.x, tx = e % 16, ty = e / 16;
    float va[8], vb[8];
    auto load = [&](int k) {
        if constexpr (AK) {
            const int m = m0 + e / 4, kk = k + 8 * (e % 4);
            load8(A + (size_t)m * lda + kk, m < M ? k1 - kk : 0, vecA, va);
        } else {
            const int kk = k + e / 8, m = m0 + 8 * (e % 8);
            load8(A + (size_t)kk * lda + m, kk < k1 ? M - m : 0, vecA, va);
        }
        if constexpr (BK) {
            const int n = n0 + e / 4, kk = k + 8 * (e % 4);
            load8(B + (size_t)n * ldb + kk, n < N ? k1 - kk : 0, vecB, vb);
        } else {
            const int kk = k + e / 8, n = n0 + 8 * (e % 8);
            load8(B + (size_t)kk * ldb + n, kk < k1 ? N - n : 0, vecB, vb);
        }
    };
    load(k0);
    for (int k = k0; k < k1; k += kGK) {
        __syncthreads();
        if constexpr (AK) {
#pragma unroll
            for (int i = 0; i < 8; i++) sm.a[8 * (e % 4) + i][e / 4] = va[i];
        } else {
            *(float4*)&sm.a[e / 8][8 * (e % 8)] = make_float4(va[0], va[1], va[2], va[3]);
            *(float4*)&sm.a[e / 8][8 * (e % 8) + 4] = make_float4(va[4], va[5], va[6], va[7]);
        }
        if constexpr (BK) {
#pragma unroll
            for (int i = 0; i < 8; i++) sm.b[8 * (e % 4) + i][e / 4] = vb[i];
        } else {
            *(float4*)&sm.b[e / 8][8 * (e % 8)] = make_float4(vb[0], vb[1], vb[2], vb[3]);
            *(float4*)&sm.b[e / 8][8 * (e % 8) + 4] = make_float4(vb[4], vb[5], vb[6], vb[7]);
        }
        __syncthreads();
        if (k + kGK < k1) load(k + kGK);
#pragma unroll 8
        for (int kk = 0; kk < kGK; kk++) {
            const float4 x = *(const float4*)&sm.a[kk][4 * ty], y = *(const float4*)&sm.b[kk][4 * tx];
            const float xa[4] = {x.x, x.y, x.z, x.w}, yb[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
            for (int i = 0; i < 4; i++)
#pragma unroll
                for (int j = 0; j < 4; j++) acc[i][j] = fmaf(xa[i], yb[j], acc[i][j]);
        }
        if (colsum && e < kGT) {
            float c = 0.0f;
#pragma unroll 8
            for (int kk = 0; kk < kGK; kk++) c += sm.a[kk][e];
            *colsum += c;
        }
    }
}

// Hidden layer: Z = A W^T + b, H = SiLU(Z).  A [n][K], W bf16 [256][K].
__global__ void __launch_bounds__(256) k_layer_hidden(int n, int K, const float* __restrict__ A, bool vecA,
                                                      const __nv_bfloat16* __restrict__ W, const float* __restrict__ bias,
                                                      float* __restrict__ Z, float* __restrict__ H)
{
    __shared__ GemmTile sm;
    const int m0 = blockIdx.y * kGT, n0 = blockIdx.x * kGT, tx = threadIdx.x % 16, ty = threadIdx.x / 16;
    float acc[4][4] = {};
    tile_gemm<true, true>(sm, acc, A, K, n, m0, vecA, W, K, kWidth, n0, true, 0, K, nullptr);
    const float4 b = *(const float4*)(bias + n0 + 4 * tx);
#pragma unroll
    for (int i = 0; i < 4; i++) {
        const int m = m0 + 4 * ty + i;
        if (m >= n) continue;
        const float4 z = make_float4(acc[i][0] + b.x, acc[i][1] + b.y, acc[i][2] + b.z, acc[i][3] + b.w);
        *(float4*)(Z + (size_t)m * kWidth + n0 + 4 * tx) = z;
        *(float4*)(H + (size_t)m * kWidth + n0 + 4 * tx) = make_float4(silu(z.x), silu(z.y), silu(z.z), silu(z.w));
    }
}

// Output layer: Y = H W^T + b into Y [n][325], or (training) straight into dY = 2 (Y - T) mask / n, [n][328],
// with one partial of sum mask (Y - T)^2 per block.
__global__ void __launch_bounds__(256) k_layer_output(int n, const float* __restrict__ H,
                                                      const __nv_bfloat16* __restrict__ W, const float* __restrict__ bias,
                                                      float* __restrict__ Y, const float* __restrict__ T,
                                                      const float* __restrict__ mask, float inv_count,
                                                      float* __restrict__ dY, double* __restrict__ part)
{
    __shared__ GemmTile sm;
    __shared__ double wsum[8];
    const int m0 = blockIdx.y * kGT, n0 = blockIdx.x * kGT, tx = threadIdx.x % 16, ty = threadIdx.x / 16;
    float acc[4][4] = {};
    tile_gemm<true, true>(sm, acc, H, kWidth, n, m0, true, W, kWidth, kOut, n0, true, 0, kWidth, nullptr);
    double loss = 0.0;
#pragma unroll
    for (int i = 0; i < 4; i++) {
        const int m = m0 + 4 * ty + i;
        if (m >= n) continue;
#pragma unroll
        for (int j = 0; j < 4; j++) {
            const int c = n0 + 4 * tx + j;
            if (c < kOut) {
                const float y = acc[i][j] + bias[c];
                const size_t o = (size_t)m * kOut + c;
                if (Y) {
                    Y[o] = y;
                } else {
                    const float d = (y - T[o]) * mask[o];
                    dY[(size_t)m * kOutLd + c] = 2.0f * d * inv_count;
                    loss += (double)d * d;
                }
            } else if (c < kOutLd && !Y) {
                dY[(size_t)m * kOutLd + c] = 0.0f;
            }
        }
    }
    if (!Y) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) loss += __shfl_xor_sync(0xffffffffu, loss, o);
        if (threadIdx.x % 32 == 0) wsum[threadIdx.x / 32] = loss;
        __syncthreads();
        if (threadIdx.x == 0) {
            double a = 0.0;
            for (int w = 0; w < 8; w++) a += wsum[w];
            part[blockIdx.y * gridDim.x + blockIdx.x] = a;
        }
    }
}

// Gradient through a layer: dZ = (G W) SiLU'(Z), G [n][ldg] with K columns, W bf16 [K][256].
__global__ void __launch_bounds__(256) k_layer_backward(int n, int K, const float* __restrict__ G, int ldg,
                                                        const __nv_bfloat16* __restrict__ W, const float* __restrict__ Z,
                                                        float* __restrict__ dZ)
{
    __shared__ GemmTile sm;
    const int m0 = blockIdx.y * kGT, n0 = blockIdx.x * kGT, tx = threadIdx.x % 16, ty = threadIdx.x / 16;
    float acc[4][4] = {};
    tile_gemm<true, false>(sm, acc, G, ldg, n, m0, true, W, kWidth, kWidth, n0, true, 0, K, nullptr);
#pragma unroll
    for (int i = 0; i < 4; i++) {
        const int m = m0 + 4 * ty + i;
        if (m >= n) continue;
        const float4 z = *(const float4*)(Z + (size_t)m * kWidth + n0 + 4 * tx);
        *(float4*)(dZ + (size_t)m * kWidth + n0 + 4 * tx) =
            make_float4(acc[i][0] * dsilu(z.x), acc[i][1] * dsilu(z.y), acc[i][2] * dsilu(z.z), acc[i][3] * dsilu(z.w));
    }
}

// Weight and bias gradients of all three layers, dW = G^T A and db = column sums of G, in one launch: block
// (tile, split) sums the samples [split chunk, (split + 1) chunk) into its own partial gradient vector.
struct WGradLayer {
    const float* G;  // [n][ldg] gradient of the layer's pre-activation, M columns
    const float* A;  // [n][N] the layer's input
    int ldg, M, N, tiles_n, tile0;
    long long off_w, off_b;
};
struct WGradArgs {
    WGradLayer l[3];
    int n, chunk;
    bool vec_x;  // the network's input may be read in 16-byte loads
    float* part;
    long long n_params;
};

__global__ void __launch_bounds__(256) k_weight_grads(const WGradArgs a)
{
    __shared__ GemmTile sm;
    const int t = blockIdx.x;
    const int li = t >= a.l[2].tile0 ? 2 : t >= a.l[1].tile0 ? 1 : 0;
    const WGradLayer& l = a.l[li];
    const int tile = t - l.tile0, m0 = tile / l.tiles_n * kGT, n0 = tile % l.tiles_n * kGT;
    const int k0 = blockIdx.y * a.chunk, k1 = min(a.n, k0 + a.chunk);
    float acc[4][4] = {};
    float cs = 0.0f;
    tile_gemm<false, false>(sm, acc, l.G, l.ldg, l.ldg, m0, true, l.A, l.N, l.N, n0, li != 2 || a.vec_x, k0, k1,
                            n0 == 0 ? &cs : nullptr);
    const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
    float* const out = a.part + (size_t)blockIdx.y * a.n_params;
#pragma unroll
    for (int i = 0; i < 4; i++)
#pragma unroll
        for (int j = 0; j < 4; j++) {
            const int m = m0 + 4 * ty + i, c = n0 + 4 * tx + j;
            if (m < l.M && c < l.N) out[l.off_w + (size_t)m * l.N + c] = acc[i][j];
        }
    if (n0 == 0 && threadIdx.x < kGT && m0 + (int)threadIdx.x < l.M) out[l.off_b + m0 + threadIdx.x] = cs;
}

// Gradient = sum of the partials, then (lr > 0) Adam on the FP32 master weights and their BF16 copy.  The last
// block sums the loss partials instead.
__global__ void k_reduce_adam(long long n, int nsplit, const float* __restrict__ part, float* __restrict__ w,
                              float* __restrict__ g, float* __restrict__ m, float* __restrict__ v,
                              __nv_bfloat16* __restrict__ wb, float lr, float b1, float b2, float eps, float c1, float c2,
                              int n_loss, const double* __restrict__ loss_part, float loss_scale, float* __restrict__ loss)
{
    if (blockIdx.x == gridDim.x - 1) {
        __shared__ double sm[256];
        double a = 0.0;
        for (int i = threadIdx.x; i < n_loss; i += blockDim.x) a += loss_part[i];
        sm[threadIdx.x] = a;
        __syncthreads();
        for (int s = blockDim.x / 2; s > 0; s >>= 1) {
            if (threadIdx.x < s) sm[threadIdx.x] += sm[threadIdx.x + s];
            __syncthreads();
        }
        if (threadIdx.x == 0 && loss) *loss = (float)(sm[0] * loss_scale);
        return;
    }
    const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= n) return;
    float gg = 0.0f;
    for (int s = 0; s < nsplit; s++) gg += part[(size_t)s * n + e];
    g[e] = gg;
    if (!(lr > 0.0f)) return;
    const float mm = b1 * m[e] + (1.0f - b1) * gg;
    const float vv = b2 * v[e] + (1.0f - b2) * gg * gg;
    m[e] = mm;
    v[e] = vv;
    const float wn = w[e] - lr * (mm * c1) / (sqrtf(vv * c2) + eps);
    w[e] = wn;
    wb[e] = __float2bfloat16(wn);
}

__global__ void k_to_bf16(long long n, const float* __restrict__ w, __nv_bfloat16* __restrict__ wb)
{
    const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (e < n) wb[e] = __float2bfloat16(w[e]);
}

// per unordered atom pair (a <= b): features and block placement
struct PairMeta {
    int row0, col0;  // first basis function of the block's row atom and column atom
    int head;        // 0 O-O, 1 O-H (O rows), 2 H-H
    int onsite;
};

__device__ __forceinline__ int element_class(int Z) { return Z == 8 ? 0 : (Z == 1 ? 1 : -1); }

__global__ void k_guess_features(int n_atoms, const double* __restrict__ xyz, const int* __restrict__ Z,
                                 const int* __restrict__ atom_bf0, float* __restrict__ X,
                                 PairMeta* __restrict__ meta, int* __restrict__ bad)
{
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long np = (long long)n_atoms * (n_atoms + 1) / 2;
    if (t >= np) return;
    long long ii = (long long)((sqrt(8.0 * (double)t + 1.0) - 1.0) * 0.5);
    while (ii * (ii + 1) / 2 > t) ii--;
    while ((ii + 1) * (ii + 2) / 2 <= t) ii++;
    int a = (int)(t - ii * (ii + 1) / 2), b = (int)ii;  // a <= b
    int ca = element_class(Z[a]), cb = element_class(Z[b]);
    if (ca < 0 || cb < 0) {
        atomicOr(bad, 1);
        ca = cb = 1;
    }
    if (ca == 1 && cb == 0) {  // O-H blocks have the O atom first
        const int t2 = a;
        a = b;
        b = t2;
        ca = 0;
        cb = 1;
    }
    float u[3] = {0.f, 0.f, 0.f}, R = 0.f;
    if (a != b) {
        const double d0 = xyz[3 * b] - xyz[3 * a], d1 = xyz[3 * b + 1] - xyz[3 * a + 1], d2 = xyz[3 * b + 2] - xyz[3 * a + 2];
        const double r = sqrt(d0 * d0 + d1 * d1 + d2 * d2);
        R = (float)r;
        u[0] = (float)(d0 / r);
        u[1] = (float)(d1 / r);
        u[2] = (float)(d2 / r);
    }
    float* x = X + t * kFeat;
    x[0] = R;
    x[1] = u[0];
    x[2] = u[1];
    x[3] = u[2];
    for (int i = 0; i < 3; i++)
        for (int j = 0; j < 3; j++) x[4 + 3 * i + j] = u[i] * u[j];
    const int head = ca == 0 ? (cb == 0 ? 0 : 1) : 2;
    x[13] = head == 0;
    x[14] = head == 1;
    x[15] = head == 2;
    PairMeta pm;
    pm.row0 = atom_bf0[a];
    pm.col0 = atom_bf0[b];
    pm.head = head;
    pm.onsite = a == b;
    meta[t] = pm;
}

// place each pair's predicted block; on-site blocks symmetrised
__global__ void k_guess_scatter(long long np, int N, const float* __restrict__ Y, const PairMeta* __restrict__ meta,
                                double* __restrict__ P)
{
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= np) return;
    const PairMeta pm = meta[t];
    const int h = pm.head, nr = head_rows(h), nc = head_cols(h);
    const float* y = Y + t * kOut + head_off(h);
    for (int r = 0; r < nr; r++)
        for (int c = 0; c < nc; c++) {
            double v = y[r * nc + c];
            if (pm.onsite) v = 0.5 * (v + (double)y[c * nc + r]);
            P[(size_t)(pm.row0 + r) * N + pm.col0 + c] = v;
            P[(size_t)(pm.col0 + c) * N + pm.row0 + r] = v;
        }
}

// Training targets of every atom pair: T[t][head block] = the pair's block of P, mask 1 there, 0 elsewhere.
__global__ void k_guess_targets(long long np, int N, const double* __restrict__ P, const PairMeta* __restrict__ meta,
                                float* __restrict__ T, float* __restrict__ mask)
{
    const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= np * kOut) return;
    const long long t = e / kOut;
    const int o = (int)(e - t * kOut);
    const PairMeta pm = meta[t];
    const int h = pm.head, o0 = head_off(h), nc = head_cols(h);
    const int r = (o - o0) / nc, c = (o - o0) % nc;
    const bool in = o >= o0 && o < o0 + head_rows(h) * nc;
    T[e] = in ? (float)P[(size_t)(pm.row0 + r) * N + pm.col0 + c] : 0.0f;
    mask[e] = in ? 1.0f : 0.0f;
}

// SplitMix64 output function (Steele, Lea and Flood, OOPSLA 2014) applied to seed + (i + 1) * golden gamma.
__host__ __device__ __forceinline__ unsigned long long splitmix64(unsigned long long seed, unsigned long long i)
{
    unsigned long long z = seed + (i + 1ull) * 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

// Minibatch of step k: sample j is row splitmix64(seed, k * batch + j) mod n of the dataset.
__global__ void k_draw_batch(long long n, int batch, unsigned long long seed, long long step,
                             const float* __restrict__ X, const float* __restrict__ T, const float* __restrict__ M,
                             float* __restrict__ Xb, float* __restrict__ Tb, float* __restrict__ Mb)
{
    const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (long long)batch * kOut) return;
    const int j = (int)(e / kOut), o = (int)(e % kOut);
    const long long row = (long long)(splitmix64(seed, (unsigned long long)(step * batch + j)) % (unsigned long long)n);
    Tb[e] = T[row * kOut + o];
    Mb[e] = M[row * kOut + o];
    if (o < kFeat) Xb[(size_t)j * kFeat + o] = X[row * kFeat + o];
}

__global__ void k_trace_ps(int N, const double* __restrict__ P, const double* __restrict__ S, double* __restrict__ part)
{
    __shared__ double sm[256];
    double acc = 0.0;
    for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < (long long)N * N;
         e += (long long)gridDim.x * blockDim.x)
        acc += P[e] * S[e];  // tr(PS) = sum_ij P_ij S_ji, S symmetric
    sm[threadIdx.x] = acc;
    __syncthreads();
    for (int s = blockDim.x / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s) sm[threadIdx.x] += sm[threadIdx.x + s];
        __syncthreads();
    }
    if (threadIdx.x == 0) part[blockIdx.x] = sm[0];
}

__global__ void k_scale_density_to(int N, const double* __restrict__ part, double n_el, double* __restrict__ P,
                                   int* __restrict__ bad)
{
    __shared__ double tr;
    if (threadIdx.x == 0) {
        double a = 0.0;
        for (int i = 0; i < 256; i++) a += part[i];
        tr = a;
        if (!(a > 0.0) || !isfinite(a)) atomicOr(bad, 2);
    }
    __syncthreads();
    const double f = (tr > 0.0 && isfinite(tr)) ? n_el / tr : 0.0;
    for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < (long long)N * N;
         e += (long long)gridDim.x * blockDim.x) {
        const double v = P[e] * f;
        if (!isfinite(v)) atomicOr(bad, 4);
        P[e] = v;
    }
}

int gfail(int code, const std::string& msg)
{
    set_error(code, msg);
    return code;
}

struct GuessDevice {
    int prev = -1;
    explicit GuessDevice(int dev)
    {
        if (cudaGetDevice(&prev) != cudaSuccess) prev = -1;
        if (prev != dev) cudaSetDevice(dev);
    }
    ~GuessDevice()
    {
        if (prev >= 0) cudaSetDevice(prev);
    }
};

}  // namespace
}  // namespace hf

using namespace hf;

constexpr int kOutTiles = (kOut + kGT - 1) / kGT;
constexpr int kMaxSplit = 8;  // splits of the minibatch in the weight gradients: 44 tiles x 8 blocks fill the GPU twice

struct hf_model {
    hf_ctx* ctx = nullptr;
    // FP32 master weights, BF16 copies, gradients, Adam moments: W1 [256x16], b1, W2 [256x256], b2, W3 [325x256], b3
    DevBuf w, wb, g, m, v;
    long long n_params = 0;
    long long off[6] = {};
    int step = 0;
    // activation workspace
    DevBuf Z1, H1, Z2, H2, Y, dY, dH, dZ, part, lossbuf, gpart;
    DevBuf Xb, Tb, Mb;  // minibatch drawn by hf_guess_train
    long long cap = 0, bcap = 0;
    int reserve(long long n)
    {
        if (n <= cap) return HF_OK;
        const long long c = std::max(n, 1024LL);
        int rc;
        if ((rc = Z1.alloc(sizeof(float) * c * kWidth)) || (rc = H1.alloc(sizeof(float) * c * kWidth)) ||
            (rc = Z2.alloc(sizeof(float) * c * kWidth)) || (rc = H2.alloc(sizeof(float) * c * kWidth)) ||
            (rc = Y.alloc(sizeof(float) * c * kOut)) || (rc = dY.alloc(sizeof(float) * c * kOutLd)) ||
            (rc = dH.alloc(sizeof(float) * c * kWidth)) || (rc = dZ.alloc(sizeof(float) * c * kWidth)) ||
            (rc = part.alloc(sizeof(double) * ((c + kGT - 1) / kGT) * kOutTiles)) ||
            (rc = gpart.alloc(sizeof(float) * kMaxSplit * n_params)))
            return rc;
        cap = c;
        return HF_OK;
    }
    float* W(int i) { return w.as<float>() + off[i]; }
    __nv_bfloat16* Wb(int i) { return wb.as<__nv_bfloat16>() + off[i]; }
    float* G(int i) { return g.as<float>() + off[i]; }
};

static const long long kSizes[6] = {(long long)kWidth * kFeat, kWidth, (long long)kWidth * kWidth, kWidth,
                                    (long long)kOut * kWidth, kOut};

static bool aligned16(const void* p) { return ((uintptr_t)p & 15) == 0; }

// Hidden layers into M's Z1, H1, Z2, H2.
static void forward_hidden(hf_model* M, int n, const float* X, cudaStream_t st)
{
    const dim3 grid(kWidth / kGT, (n + kGT - 1) / kGT);
    k_layer_hidden<<<grid, 256, 0, st>>>(n, kFeat, X, aligned16(X), M->Wb(0), M->W(1), M->Z1.as<float>(), M->H1.as<float>());
    k_layer_hidden<<<grid, 256, 0, st>>>(n, kWidth, M->H1.as<float>(), true, M->Wb(2), M->W(3), M->Z2.as<float>(),
                                         M->H2.as<float>());
}

static int forward(hf_model* M, int n, const float* X, cudaStream_t st)
{
    forward_hidden(M, n, X, st);
    k_layer_output<<<dim3(kOutTiles, (n + kGT - 1) / kGT), 256, 0, st>>>(n, M->H2.as<float>(), M->Wb(4), M->W(5),
                                                                         M->Y.as<float>(), nullptr, nullptr, 0.0f, nullptr,
                                                                         nullptr);
    return cudaGetLastError() == cudaSuccess ? HF_OK : cuda_status(cudaGetLastError(), "guess forward");
}

// One training step: loss = (1/n) sum_samples sum_outputs mask (Y - T)^2 (masks are 0/1 per output) into loss_dev
// (nullable), its gradients into M->g, and for lr > 0 one Adam step (beta 0.9 / 0.999, eps 1e-8).
static int train_step(hf_model* M, int n, const float* X, const float* T, const float* mask, float lr, float* loss_dev,
                      cudaStream_t st)
{
    const int rows = (n + kGT - 1) / kGT;
    const float inv = 1.0f / (float)n;
    forward_hidden(M, n, X, st);
    k_layer_output<<<dim3(kOutTiles, rows), 256, 0, st>>>(n, M->H2.as<float>(), M->Wb(4), M->W(5), nullptr, T, mask, inv,
                                                          M->dY.as<float>(), M->part.as<double>());
    const dim3 grid(kWidth / kGT, rows);
    k_layer_backward<<<grid, 256, 0, st>>>(n, kOut, M->dY.as<float>(), kOutLd, M->Wb(4), M->Z2.as<float>(),
                                           M->dH.as<float>());
    k_layer_backward<<<grid, 256, 0, st>>>(n, kWidth, M->dH.as<float>(), kWidth, M->Wb(2), M->Z1.as<float>(),
                                           M->dZ.as<float>());
    WGradArgs a;
    a.l[0] = {M->dY.as<float>(), M->H2.as<float>(), kOutLd, kOut, kWidth, kWidth / kGT, 0, M->off[4], M->off[5]};
    a.l[1] = {M->dH.as<float>(), M->H1.as<float>(), kWidth, kWidth, kWidth, kWidth / kGT, kOutTiles * (kWidth / kGT),
              M->off[2], M->off[3]};
    a.l[2] = {M->dZ.as<float>(), X, kWidth, kWidth, kFeat, 1, a.l[1].tile0 + (kWidth / kGT) * (kWidth / kGT), M->off[0],
              M->off[1]};
    const int tiles = a.l[2].tile0 + kWidth / kGT;
    // as many splits as leave each at least 128 samples, up to kMaxSplit; whole k-tiles
    const int want = std::max(1, std::min(kMaxSplit, n / 128));
    a.n = n;
    a.chunk = ((n + want - 1) / want + kGK - 1) / kGK * kGK;
    const int nsplit = (n + a.chunk - 1) / a.chunk;
    a.vec_x = aligned16(X);
    a.part = M->gpart.as<float>();
    a.n_params = M->n_params;
    k_weight_grads<<<dim3(tiles, nsplit), 256, 0, st>>>(a);
    const float b1 = 0.9f, b2 = 0.999f;
    if (lr > 0.0f) M->step++;
    const float c1 = 1.0f / (1.0f - powf(b1, (float)M->step)), c2 = 1.0f / (1.0f - powf(b2, (float)M->step));
    k_reduce_adam<<<(unsigned)((M->n_params + 255) / 256) + 1, 256, 0, st>>>(
        M->n_params, nsplit, M->gpart.as<float>(), M->w.as<float>(), M->g.as<float>(), M->m.as<float>(), M->v.as<float>(),
        M->wb.as<__nv_bfloat16>(), lr, b1, b2, 1e-8f, c1, c2, kOutTiles * rows, M->part.as<double>(), inv, loss_dev);
    return cudaGetLastError() == cudaSuccess ? HF_OK : cuda_status(cudaGetLastError(), "guess training step");
}

extern "C" {

int hf_model_create(hf_ctx* ctx, const float* init_weights, hf_model** out)
{
    if (!ctx || !init_weights || !out) return gfail(HF_E_INVALID, "hf_model_create: NULL argument");
    *out = nullptr;
    GuessDevice gd(ctx->device);
    hf_model* M = new hf_model();
    M->ctx = ctx;
    long long o = 0;
    for (int i = 0; i < 6; i++) {
        M->off[i] = o;
        o += kSizes[i];
    }
    M->n_params = o;
    int rc;
    if ((rc = M->w.alloc(sizeof(float) * o)) || (rc = M->wb.alloc(sizeof(__nv_bfloat16) * o)) ||
        (rc = M->g.alloc(sizeof(float) * o)) || (rc = M->m.alloc(sizeof(float) * o)) ||
        (rc = M->v.alloc(sizeof(float) * o)) ||
        (rc = M->lossbuf.alloc(sizeof(float) * 4))) {
        delete M;
        return rc;
    }
    cudaStream_t st = ctx->stream;
    HF_CUDA(cudaMemcpyAsync(M->w.p, init_weights, sizeof(float) * o, cudaMemcpyHostToDevice, st));
    HF_CUDA(cudaMemsetAsync(M->m.p, 0, sizeof(float) * o, st));
    HF_CUDA(cudaMemsetAsync(M->v.p, 0, sizeof(float) * o, st));
    k_to_bf16<<<(unsigned)((o + 255) / 256), 256, 0, st>>>(o, M->w.as<float>(), M->wb.as<__nv_bfloat16>());
    HF_CUDA(cudaStreamSynchronize(st));
    *out = M;
    return HF_OK;
}

void hf_model_destroy(hf_model* M)
{
    if (!M) return;
    GuessDevice gd(M->ctx->device);
    cudaStreamSynchronize(M->ctx->stream);
    delete M;
}

int64_t hf_model_num_params(void) { return kSizes[0] + kSizes[1] + kSizes[2] + kSizes[3] + kSizes[4] + kSizes[5]; }

int hf_model_get_weights(hf_model* M, float* w, float* grad)
{
    if (!M) return gfail(HF_E_INVALID, "hf_model_get_weights: NULL model");
    GuessDevice gd(M->ctx->device);
    cudaStream_t st = M->ctx->stream;
    if (w) HF_CUDA(cudaMemcpyAsync(w, M->w.p, sizeof(float) * M->n_params, cudaMemcpyDeviceToHost, st));
    if (grad) HF_CUDA(cudaMemcpyAsync(grad, M->g.p, sizeof(float) * M->n_params, cudaMemcpyDeviceToHost, st));
    HF_CUDA(cudaStreamSynchronize(st));
    return HF_OK;
}

int hf_model_forward(hf_model* M, int n, const float* X, float* Y, int flags)
{
    if (!M || !X || !Y || n <= 0) return gfail(HF_E_INVALID, "hf_model_forward: bad arguments");
    GuessDevice gd(M->ctx->device);
    cudaStream_t st = M->ctx->stream;
    int rc = M->reserve(n);
    if (rc != HF_OK) return rc;
    const bool dev = (flags & HF_PTR_DEVICE) != 0;
    DevBuf Xd;
    const float* xp = X;
    if (!dev) {
        if ((rc = Xd.alloc(sizeof(float) * (size_t)n * kFeat))) return rc;
        HF_CUDA(cudaMemcpyAsync(Xd.p, X, sizeof(float) * (size_t)n * kFeat, cudaMemcpyHostToDevice, st));
        xp = Xd.as<float>();
    }
    if ((rc = forward(M, n, xp, st)) != HF_OK) return rc;
    HF_CUDA(cudaMemcpyAsync(Y, M->Y.p, sizeof(float) * (size_t)n * kOut,
                            dev ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost, st));
    HF_CUDA(cudaStreamSynchronize(st));
    return HF_OK;
}

int hf_model_train_step(hf_model* M, int n, const float* X, const float* T, const float* mask, float lr,
                        float* loss, int flags)
{
    if (!M || !X || !T || !mask || n <= 0) return gfail(HF_E_INVALID, "hf_model_train_step: bad arguments");
    GuessDevice gd(M->ctx->device);
    cudaStream_t st = M->ctx->stream;
    int rc = M->reserve(n);
    if (rc != HF_OK) return rc;
    if (!(flags & HF_PTR_DEVICE)) return gfail(HF_E_INVALID, "hf_model_train_step: device pointers required");
    if ((rc = train_step(M, n, X, T, mask, lr, M->lossbuf.as<float>(), st)) != HF_OK) return rc;
    if (loss) HF_CUDA(cudaMemcpyAsync(loss, M->lossbuf.p, sizeof(float), cudaMemcpyDeviceToHost, st));
    HF_CUDA(cudaStreamSynchronize(st));
    HF_CUDA(cudaGetLastError());
    return HF_OK;
}

int hf_guess_train(hf_model* M, int64_t n, const float* X, const float* T, const float* mask,
                   const hf_train_opts* opts, float* losses, int flags)
{
    if (!M || !X || !T || !mask || !opts || n <= 0) return gfail(HF_E_INVALID, "hf_guess_train: bad arguments");
    if (!(flags & HF_PTR_DEVICE)) return gfail(HF_E_INVALID, "hf_guess_train: the dataset must be in device memory");
    if (opts->steps <= 0 || opts->batch < 0 || !(opts->lr >= 0.0f) || !isfinite(opts->lr))
        return gfail(HF_E_INVALID, "hf_guess_train: bad options");
    GuessDevice gd(M->ctx->device);
    cudaStream_t st = M->ctx->stream;
    const int batch = (int)std::min<int64_t>(opts->batch > 0 ? opts->batch : 2048, n);
    const float lr = opts->lr > 0.0f ? opts->lr : 1e-3f;
    int rc = M->reserve(batch);
    if (rc != HF_OK) return rc;
    if (batch > M->bcap) {
        if ((rc = M->Xb.alloc(sizeof(float) * (size_t)batch * kFeat)) ||
            (rc = M->Tb.alloc(sizeof(float) * (size_t)batch * kOut)) ||
            (rc = M->Mb.alloc(sizeof(float) * (size_t)batch * kOut))) {
            M->bcap = 0;
            return rc;
        }
        M->bcap = batch;
    }
    DevBuf ldev;
    if ((rc = ldev.alloc(sizeof(float) * (size_t)opts->steps))) return rc;
    const long long ne = (long long)batch * kOut;
    const double pi = 3.14159265358979323846;
    for (int k = 0; k < opts->steps; k++) {
        k_draw_batch<<<(unsigned)((ne + 255) / 256), 256, 0, st>>>(n, batch, (unsigned long long)opts->seed, k, X, T,
                                                                  mask, M->Xb.as<float>(), M->Tb.as<float>(),
                                                                  M->Mb.as<float>());
        // cosine decay from lr to 0 over the run
        const float lr_k = (float)(lr * 0.5 * (1.0 + cos(pi * (double)k / (double)opts->steps)));
        if ((rc = train_step(M, batch, M->Xb.as<float>(), M->Tb.as<float>(), M->Mb.as<float>(), lr_k,
                             ldev.as<float>() + k, st)) != HF_OK)
            return rc;
    }
    HF_CUDA(cudaGetLastError());
    if (losses) HF_CUDA(cudaMemcpyAsync(losses, ldev.p, sizeof(float) * (size_t)opts->steps, cudaMemcpyDeviceToHost, st));
    HF_CUDA(cudaStreamSynchronize(st));
    HF_CUDA(cudaGetLastError());
    return HF_OK;
}

// Check that every atom is H (5 functions) or O (15 functions) with contiguous shells.
static int check_guess_basis(const hf_system* S)
{
    for (int a = 0; a < S->n_atoms; a++) {
        const int z = S->Z_h[a], nb = S->atom_nbf_h[a];
        if (!((z == 8 && nb == 15) || (z == 1 && nb == 5)) || S->atom_bf0_h[a] < 0)
            return gfail(HF_E_UNSUPPORTED, "learned guess: every atom must be O with 15 or H with 5 contiguous "
                                           "Cartesian functions (the synthetic water basis)");
    }
    return HF_OK;
}

// per-pair features of a system: X [n_pairs x 16] floats, meta [n_pairs x 4] ints
// (row atom's first function, column atom's first function, head, on-site flag)
int hf_guess_features(hf_system* S, float* X, int32_t* meta, int64_t* n_pairs, int flags)
{
    if (!S || !n_pairs) return gfail(HF_E_INVALID, "hf_guess_features: NULL argument");
    const long long np = (long long)S->n_atoms * (S->n_atoms + 1) / 2;
    *n_pairs = np;
    if (!X || !meta) return HF_OK;  // size query
    int rc = check_guess_basis(S);
    if (rc != HF_OK) return rc;
    GuessDevice gd(S->device);
    cudaStream_t st = S->stream;
    DevBuf bf0, Zi, bad, Xd, Md;
    if ((rc = bf0.alloc(sizeof(int) * S->n_atoms)) || (rc = Zi.alloc(sizeof(int) * S->n_atoms)) ||
        (rc = bad.alloc(sizeof(int))))
        return rc;
    HF_CUDA(cudaMemcpyAsync(Zi.p, S->Z_h.data(), sizeof(int) * S->n_atoms, cudaMemcpyHostToDevice, st));
    HF_CUDA(cudaMemcpyAsync(bf0.p, S->atom_bf0_h.data(), sizeof(int) * S->n_atoms, cudaMemcpyHostToDevice, st));
    HF_CUDA(cudaMemsetAsync(bad.p, 0, sizeof(int), st));
    const bool dev = (flags & HF_PTR_DEVICE) != 0;
    float* xp = X;
    PairMeta* mp = (PairMeta*)meta;
    if (!dev) {
        if ((rc = Xd.alloc(sizeof(float) * np * kFeat)) || (rc = Md.alloc(sizeof(PairMeta) * np))) return rc;
        xp = Xd.as<float>();
        mp = Md.as<PairMeta>();
    }
    k_guess_features<<<(unsigned)((np + 127) / 128), 128, 0, st>>>(S->n_atoms, S->atom_xyz.as<double>(), Zi.as<int>(),
                                                                  bf0.as<int>(), xp, mp, bad.as<int>());
    int hb = 0;
    HF_CUDA(cudaMemcpyAsync(&hb, bad.p, sizeof(int), cudaMemcpyDeviceToHost, st));
    if (!dev) {
        HF_CUDA(cudaMemcpyAsync(X, xp, sizeof(float) * np * kFeat, cudaMemcpyDeviceToHost, st));
        HF_CUDA(cudaMemcpyAsync(meta, mp, sizeof(PairMeta) * np, cudaMemcpyDeviceToHost, st));
    }
    HF_CUDA(cudaStreamSynchronize(st));
    if (hb) return gfail(HF_E_UNSUPPORTED, "hf_guess_features: only H and O atoms are supported");
    return HF_OK;
}

int hf_guess_targets(hf_system* S, const double* P, float* T, float* mask, int flags)
{
    if (!S || !P || !T || !mask) return gfail(HF_E_INVALID, "hf_guess_targets: NULL argument");
    GuessDevice gd(S->device);
    cudaStream_t st = S->stream;
    int64_t np = 0;
    hf_guess_features(S, nullptr, nullptr, &np, 0);
    const int N = S->n_bf;
    const bool dev = (flags & HF_PTR_DEVICE) != 0;
    DevBuf X, meta, Pd, Td, Md;
    int rc;
    if ((rc = X.alloc(sizeof(float) * np * kFeat)) || (rc = meta.alloc(sizeof(PairMeta) * np))) return rc;
    if ((rc = hf_guess_features(S, X.as<float>(), (int32_t*)meta.p, &np, HF_PTR_DEVICE)) != HF_OK) return rc;
    const double* pp = P;
    float *tp = T, *mp = mask;
    if (!dev) {
        if ((rc = Pd.alloc(sizeof(double) * (size_t)N * N)) || (rc = Td.alloc(sizeof(float) * np * kOut)) ||
            (rc = Md.alloc(sizeof(float) * np * kOut)))
            return rc;
        HF_CUDA(cudaMemcpyAsync(Pd.p, P, sizeof(double) * (size_t)N * N, cudaMemcpyHostToDevice, st));
        pp = Pd.as<double>();
        tp = Td.as<float>();
        mp = Md.as<float>();
    }
    const long long ne = np * kOut;
    k_guess_targets<<<(unsigned)((ne + 255) / 256), 256, 0, st>>>(np, N, pp, meta.as<PairMeta>(), tp, mp);
    HF_CUDA(cudaGetLastError());
    if (!dev) {
        HF_CUDA(cudaMemcpyAsync(T, tp, sizeof(float) * ne, cudaMemcpyDeviceToHost, st));
        HF_CUDA(cudaMemcpyAsync(mask, mp, sizeof(float) * ne, cudaMemcpyDeviceToHost, st));
    }
    HF_CUDA(cudaStreamSynchronize(st));
    return HF_OK;
}

int hf_guess_predict(hf_model* M, hf_system* S, double* P, int flags)
{
    if (!M || !S || !P) return gfail(HF_E_INVALID, "hf_guess_predict: NULL argument");
    GuessDevice gd(S->device);
    cudaStream_t st = S->stream;
    int64_t np = 0;
    hf_guess_features(S, nullptr, nullptr, &np, 0);
    DevBuf X, meta, Pd, part, bad;
    int rc;
    if ((rc = X.alloc(sizeof(float) * np * kFeat)) || (rc = meta.alloc(sizeof(PairMeta) * np)) ||
        (rc = part.alloc(sizeof(double) * 256)) || (rc = bad.alloc(sizeof(int))))
        return rc;
    if ((rc = hf_guess_features(S, X.as<float>(), (int32_t*)meta.p, &np, HF_PTR_DEVICE)) != HF_OK)
        return rc;
    if ((rc = M->reserve(np)) != HF_OK) return rc;
    if ((rc = forward(M, (int)np, X.as<float>(), st)) != HF_OK) return rc;
    const int N = S->n_bf;
    const bool dev = (flags & HF_PTR_DEVICE) != 0;
    double* pp = P;
    if (!dev) {
        if ((rc = Pd.alloc(sizeof(double) * (size_t)N * N))) return rc;
        pp = Pd.as<double>();
    }
    HF_CUDA(cudaMemsetAsync(pp, 0, sizeof(double) * (size_t)N * N, st));
    HF_CUDA(cudaMemsetAsync(bad.p, 0, sizeof(int), st));
    k_guess_scatter<<<(unsigned)((np + 127) / 128), 128, 0, st>>>(np, N, M->Y.as<float>(), meta.as<PairMeta>(), pp);
    k_trace_ps<<<256, 256, 0, st>>>(N, pp, S->S.as<double>(), part.as<double>());
    k_scale_density_to<<<256, 256, 0, st>>>(N, part.as<double>(), (double)S->n_electrons, pp, bad.as<int>());
    int hb = 0;
    HF_CUDA(cudaMemcpyAsync(&hb, bad.p, sizeof(int), cudaMemcpyDeviceToHost, st));
    if (!dev) HF_CUDA(cudaMemcpyAsync(P, pp, sizeof(double) * (size_t)N * N, cudaMemcpyDeviceToHost, st));
    HF_CUDA(cudaStreamSynchronize(st));
    HF_CUDA(cudaGetLastError());
    if (hb) return gfail(HF_E_INVALID, "hf_guess_predict: the predicted density is not finite or has tr(PS) <= 0");
    return HF_OK;
}

}  // extern "C"
