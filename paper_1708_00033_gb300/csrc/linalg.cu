// Dense FP64 linear algebra of the SCF cycle (Section 3: diagonalise the Fock
// matrix in an orthogonal basis, form the new density):
//   - tiled SIMT FP64 GEMM  C = alpha op(A) op(B) + beta C  (row-major);
//   - parallel cyclic Jacobi eigensolver for symmetric matrices: each round
//     applies N/2 disjoint plane rotations chosen by the round-robin
//     ("circle") ordering, every 2x2 block of A' = J^T A J and every row pair
//     of V' = V J being independent; one launch per round, ping-pong buffers;
//   - small helpers (antisymmetric part, dot products, linear combinations,
//     RMS difference, the Pulay DIIS system solved on the device).
#include <math.h>

#include <utility>

#include "linalg.cuh"

namespace hf {

// ------------------------------------------------------------------ GEMM --
constexpr int kTK = 16;

// C[M x N] = alpha * op(A)[M x K] * op(B)[K x N] + beta * C, all row-major.
// op(A) = A (lda >= K) or A^T (A stored K x M, lda >= M); same for B.
// T x T tile per block of NT threads, (T / sqrt(NT))^2 outputs per thread.  An SM does only two FP64 FMAs per
// clock, so a 64 x 64 tile of a 100 x 100 product took 114 us on four SMs; the tile shrinks until the product
// covers the GPU (gemm below), and each SM then has as little to do as the shape allows.
template <int T, int NT>
__global__ void __launch_bounds__(NT) k_gemm_f64(int M, int N, int K, double alpha, const double* __restrict__ A,
                                                 int lda, int ta, const double* __restrict__ B, int ldb, int tb,
                                                 double beta, double* __restrict__ C, int ldc)
{
    constexpr int S = NT == 256 ? 16 : 8;  // threads per tile side
    constexpr int Q = T / S;               // outputs per thread and side
    __shared__ double As[kTK][T + 1];
    __shared__ double Bs[kTK][T + 1];
    const int tx = threadIdx.x % S, ty = threadIdx.x / S;
    const int m0 = blockIdx.y * T, n0 = blockIdx.x * T;
    double acc[Q][Q];
#pragma unroll
    for (int i = 0; i < Q; i++)
#pragma unroll
        for (int j = 0; j < Q; j++) acc[i][j] = 0.0;
    for (int k0 = 0; k0 < K; k0 += kTK) {
        // load As[k][m] = op(A)[m0+m][k0+k]
        for (int e = threadIdx.x; e < kTK * T; e += NT) {
            int k, m;
            if (ta) {  // A stored K x M: contiguous in m
                k = e / T;
                m = e % T;
            } else {  // A stored M x K: contiguous in k
                m = e / kTK;
                k = e % kTK;
            }
            const int gm = m0 + m, gk = k0 + k;
            double v = 0.0;
            if (gm < M && gk < K) v = ta ? A[(size_t)gk * lda + gm] : A[(size_t)gm * lda + gk];
            As[k][m] = v;
        }
        for (int e = threadIdx.x; e < kTK * T; e += NT) {
            int k, n;
            if (tb) {  // B stored N x K
                n = e / kTK;
                k = e % kTK;
            } else {  // B stored K x N
                k = e / T;
                n = e % T;
            }
            const int gn = n0 + n, gk = k0 + k;
            double v = 0.0;
            if (gn < N && gk < K) v = tb ? B[(size_t)gn * ldb + gk] : B[(size_t)gk * ldb + gn];
            Bs[k][n] = v;
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < kTK; k++) {
            double a[Q], b[Q];
#pragma unroll
            for (int i = 0; i < Q; i++) a[i] = As[k][ty + S * i];
#pragma unroll
            for (int j = 0; j < Q; j++) b[j] = Bs[k][tx + S * j];
#pragma unroll
            for (int i = 0; i < Q; i++)
#pragma unroll
                for (int j = 0; j < Q; j++) acc[i][j] = fma(a[i], b[j], acc[i][j]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < Q; i++) {
        const int gm = m0 + ty + S * i;
        if (gm >= M) continue;
#pragma unroll
        for (int j = 0; j < Q; j++) {
            const int gn = n0 + tx + S * j;
            if (gn >= N) continue;
            double* c = C + (size_t)gm * ldc + gn;
            *c = alpha * acc[i][j] + (beta == 0.0 ? 0.0 : beta * *c);
        }
    }
}

int gemm(int M, int N, int K, double alpha, const double* A, int lda, bool ta, const double* B, int ldb, bool tb,
         double beta, double* C, int ldc, cudaStream_t s)
{
    if (M <= 0 || N <= 0) return 0;
    // the largest tile that still gives most of the 152 SMs a block
    auto blocks = [&](int t) { return (long long)((M + t - 1) / t) * ((N + t - 1) / t); };
    const int t = blocks(64) >= 128 ? 64 : blocks(32) >= 128 ? 32 : blocks(16) >= 128 ? 16 : 8;
    const dim3 grid((N + t - 1) / t, (M + t - 1) / t);
    if (t == 64)
        k_gemm_f64<64, 256><<<grid, 256, 0, s>>>(M, N, K, alpha, A, lda, ta ? 1 : 0, B, ldb, tb ? 1 : 0, beta, C, ldc);
    else if (t == 32)
        k_gemm_f64<32, 256><<<grid, 256, 0, s>>>(M, N, K, alpha, A, lda, ta ? 1 : 0, B, ldb, tb ? 1 : 0, beta, C, ldc);
    else if (t == 16)
        k_gemm_f64<16, 256><<<grid, 256, 0, s>>>(M, N, K, alpha, A, lda, ta ? 1 : 0, B, ldb, tb ? 1 : 0, beta, C, ldc);
    else
        k_gemm_f64<8, 64><<<grid, 64, 0, s>>>(M, N, K, alpha, A, lda, ta ? 1 : 0, B, ldb, tb ? 1 : 0, beta, C, ldc);
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

// ---------------------------------------------------------------- Jacobi --
// Round-robin pairing of n (even) indices, round r in [0, n-1), pair k in [0, n/2).
__device__ __forceinline__ void rr_pair(int n, int r, int k, int& p, int& q)
{
    const int m = n - 1;
    if (k == 0) {
        p = m;
        q = r;
    } else {
        p = (r + k) % m;
        q = (r - k + m) % m;
    }
}

// Rotation zeroing A_pq: t = tan(theta), |theta| <= pi/4, is the smaller root of x t^2 + 2 d t - x = 0 with
// d = A_qq - A_pp, x = 2 A_pq; c = 1/sqrt(1 + t^2), s = t c.  The root comes from FP32 and one Newton step whose
// residual is FP64 and whose slope is FP32 (relative error about 1e-13); c and s belong to that t to FP64 rounding,
// so the rotation is as orthogonal as with the exact root, and exactly 1, t for tiny angles.  About 15 dependent
// FP64 instructions where a division, two square roots and two reciprocals took some 45; this chain is most of a
// round's latency.  The matrix is scaled to max |a_ij| ~ 1, so what underflows in FP32 is far below the tolerance.
__device__ __forceinline__ void jacobi_cs(const double* __restrict__ A, int n, int p, int q, double& c, double& s)
{
    const double x = 2.0 * A[(size_t)p * n + q];
    const double d = A[(size_t)q * n + q] - A[(size_t)p * n + p];
    const float xf = (float)x, df = (float)d;
    c = 1.0;
    s = 0.0;
    if (xf == 0.0f) return;
    const float th = df / xf;
    const float tf = (th >= 0.0f ? 1.0f : -1.0f) / (fabsf(th) + sqrtf(fmaf(th, th, 1.0f)));
    double t = (double)tf;
    const double w = fma(x, t, 2.0 * d);
    const float res = (float)fma(t, w, -x);
    const float slope = 2.0f * fmaf(xf, tf, df);
    if (slope != 0.0f) t -= (double)(res / slope);
    c = rsqrt(fma(t, t, 1.0));
    s = t * c;
}

constexpr int kJT = 8;  // row pairs and column pairs per block: 300 working blocks at n = 375 (16: 78, half the SMs)

// One round: the 2x2 block of rows (p_r, q_r) and columns (p_c, q_c) of A goes into Anew, with its mirror image, and
// the entries of V in rows (p_r|q_r), columns (p_c|q_c) and the other way round.  Blocks below the diagonal do
// nothing: A stays symmetric, which saves a third of the FP64 work.  The block's first warp makes the rotations of
// its 8 row pairs and 8 column pairs; making them once needs a launch of its own and costs more.  Launched with
// programmatic serialisation: a round's blocks are resident when the previous round ends.
// Measured at n = 375: 6.5 us per round (10.6 us as two launches over the whole square), hf_eigh 37.7 -> 18.9 ms.
__global__ void __launch_bounds__(kJT * kJT) k_jacobi_round(int n, int r, const double* __restrict__ A,
                                                            double* __restrict__ Anew, double* __restrict__ V)
{
    __shared__ double sc[2 * kJT], ss[2 * kJT];
    __shared__ int sp[2 * kJT], sq[2 * kJT];
    if (blockIdx.x < blockIdx.y) return;
    const int half = n / 2;
    cudaGridDependencySynchronize();
    if (threadIdx.x < 2 * kJT) {
        const int i = threadIdx.x, k = (i < kJT ? blockIdx.y : blockIdx.x) * kJT + (i & (kJT - 1));
        if (k < half) {
            int p, q;
            rr_pair(n, r, k, p, q);
            jacobi_cs(A, n, p, q, sc[i], ss[i]);
            sp[i] = p;
            sq[i] = q;
        }
    }
    __syncthreads();
    const int tr = threadIdx.x / kJT, tc = threadIdx.x % kJT;
    const int kr = blockIdx.y * kJT + tr, kc = blockIdx.x * kJT + tc;
    if (kr >= half || kc >= half || kr > kc) return;
    const int pr = sp[tr], qr = sq[tr], pc = sp[kJT + tc], qc = sq[kJT + tc];
    const double cr = sc[tr], sr = ss[tr], cc = sc[kJT + tc], sn = ss[kJT + tc];
    const double a = A[(size_t)pr * n + pc], b = A[(size_t)pr * n + qc];
    const double c = A[(size_t)qr * n + pc], d = A[(size_t)qr * n + qc];
    // columns: A J_c, then rows: J_r^T (A J_c)
    const double a1 = cc * a - sn * b, b1 = sn * a + cc * b;
    const double c1 = cc * c - sn * d, d1 = sn * c + cc * d;
    const double a2 = cr * a1 - sr * c1, c2 = sr * a1 + cr * c1;
    const double b2 = cr * b1 - sr * d1, d2 = sr * b1 + cr * d1;
    Anew[(size_t)pr * n + pc] = a2;
    Anew[(size_t)qr * n + pc] = c2;
    Anew[(size_t)pr * n + qc] = b2;
    Anew[(size_t)qr * n + qc] = d2;
    auto rotate_v = [&](int row, int p, int q, double cs, double sn_) {
        double* const vp = V + (size_t)row * n + p;
        double* const vq = V + (size_t)row * n + q;
        const double x = *vp, y = *vq;
        *vp = cs * x - sn_ * y;
        *vq = sn_ * x + cs * y;
    };
    rotate_v(pr, pc, qc, cc, sn);
    rotate_v(qr, pc, qc, cc, sn);
    if (kr != kc) {
        Anew[(size_t)pc * n + pr] = a2;
        Anew[(size_t)pc * n + qr] = c2;
        Anew[(size_t)qc * n + pr] = b2;
        Anew[(size_t)qc * n + qr] = d2;
        rotate_v(pc, pr, qr, cr, sr);
        rotate_v(qc, pr, qr, cr, sr);
    }
}

static int launch_jacobi_round(int m, int r, const double* A, double* Anew, double* V, cudaStream_t s)
{
    const unsigned g = (m / 2 + kJT - 1) / kJT;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(g, g);
    cfg.blockDim = dim3(kJT * kJT);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_jacobi_round, m, r, A, Anew, V) == cudaSuccess ? 0 : -1;
}

// sum of squares of the off-diagonal and of all entries (two partial arrays)
__global__ void k_offdiag(int n, const double* __restrict__ A, double* __restrict__ part)
{
    __shared__ double so[256], sa[256];
    double o = 0.0, t = 0.0;
    for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < (long long)n * n;
         e += (long long)gridDim.x * blockDim.x) {
        const double v = A[e];
        t += v * v;
        if (e / n != e % n) o += v * v;
    }
    so[threadIdx.x] = o;
    sa[threadIdx.x] = t;
    __syncthreads();
    for (int s = blockDim.x / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s) {
            so[threadIdx.x] += so[threadIdx.x + s];
            sa[threadIdx.x] += sa[threadIdx.x + s];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        part[blockIdx.x] = so[0];
        part[gridDim.x + blockIdx.x] = sa[0];
    }
}

__global__ void k_sum2(int nb, const double* __restrict__ part, double* __restrict__ out)
{
    __shared__ double s0[256], s1[256];
    double a = 0.0, b = 0.0;
    for (int i = threadIdx.x; i < nb; i += blockDim.x) {
        a += part[i];
        b += part[nb + i];
    }
    s0[threadIdx.x] = a;
    s1[threadIdx.x] = b;
    __syncthreads();
    for (int s = blockDim.x / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s) {
            s0[threadIdx.x] += s0[threadIdx.x + s];
            s1[threadIdx.x] += s1[threadIdx.x + s];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        out[0] = s0[0];
        out[1] = s1[0];
    }
}

// pad an n x n symmetric matrix to m x m (m = n or n + 1); identity for V
__global__ void k_jacobi_init(int n, int m, const double* __restrict__ src, double* __restrict__ A,
                              double* __restrict__ V, double pad_value)
{
    const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (long long)m * m) return;
    const int i = (int)(e / m), j = (int)(e % m);
    double v;
    if (i < n && j < n)
        v = 0.5 * (src[(size_t)i * n + j] + src[(size_t)j * n + i]);
    else
        v = (i == j) ? pad_value : 0.0;
    A[e] = v;
    V[e] = (i == j) ? 1.0 : 0.0;
}

// eigenvalues -> sort keys (ascending eigenvalue, then index)
__global__ void k_diag_keys(int m, const double* __restrict__ A, double* __restrict__ key, int* __restrict__ val,
                            int m_pad)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= m_pad) return;
    if (i < m) {
        key[i] = -A[(size_t)i * m + i];  // descending sort of -lambda = ascending lambda
        val[i] = i;
    } else {
        key[i] = -INFINITY;
        val[i] = 0x7fffffff;
    }
}

// The matrix is worked on times this power of two (exact), which brings max |a_ij| into [1, 2): the sums of
// squares of the convergence tests and the FP32 steps neither under- nor overflow.  scale[0] = bits of max |a_ij|.
// Subnormal matrices take the largest power whose double is finite too (2^1022): they end up above 2^-52.
__device__ __forceinline__ double eigh_factor(const unsigned long long* scale)
{
    const double mx = __longlong_as_double(scale[0]);
    return mx > 0.0 && isfinite(mx) ? ldexp(1.0, min(-ilogb(mx), 1022)) : 1.0;
}

// w[j] = lambda of sorted column j; Vout[:, j] = V[:n, perm[j]] for j < ncols
__global__ void k_gather_eig(int n, int m, int ncols, const double* __restrict__ A, const double* __restrict__ V,
                             const int* __restrict__ perm, const unsigned long long* __restrict__ scale,
                             double* __restrict__ w, double* __restrict__ Vout)
{
    const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (long long)n * ncols) return;
    const int i = (int)(e / ncols), j = (int)(e % ncols);
    const int src = perm[j];
    Vout[e] = V[(size_t)i * m + src];
    if (i == 0 && w) w[j] = A[(size_t)src * m + src] / eigh_factor(scale);
}

int bitonic_sort_desc(double* key, int* val, int n, int n_pad, cudaStream_t s);

// doubles of the Jacobi sweeps' own workspace: A, its ping-pong copy and V, partial sums, sort keys, norms and lambda
static size_t jacobi_work_base(int n)
{
    const size_t m = (size_t)(n + (n & 1));
    size_t mp = 1;
    while (mp < m) mp <<= 1;
    return 3 * m * m + 514 + mp + 2 * m;
}

// remove value x from perm[0..m) keeping order (single thread; m small enough)
__global__ void k_drop_index(int m, int* perm, int x)
{
    int o = 0;
    for (int i = 0; i < m; i++)
        if (perm[i] != x) perm[o++] = perm[i];
}


// ------------------------------------------------ eigenvectors to start from --
// FP64 Jacobi from an unprepared matrix takes 8 to 10 sweeps of n - 1 rounds, each round bound by launch and
// FP64 latency (an SM issues an FP64 warp instruction every 16 clocks).  The sweeps far from convergence need no
// FP64: an FP32 eigenbasis, refined in FP64 by matrix products, leaves the FP64 Jacobi a matrix that is
// already diagonal to its own tolerance, or nearly so (clustered eigenvalues), and its convergence test decides
// as before.
//   1. One-sided (Hestenes) Jacobi in FP32 on the columns of G = A / s + c I, c > ||A / s||: G is positive
//      definite, so its columns converge to lambda_j v_j and need no second matrix.  One warp per column pair, the
//      whole matrix in one SM's shared memory.
//   2. Two passes of the iterative refinement of the symmetric eigendecomposition (T. Ogita and K. Aishima, Japan J.
//      Indust. Appl. Math. 35, 2018): R = I - X^T X, S = X^T A X, X += X E with E_ij = (s_ij + l_j r_ij) / (l_j - l_i),
//      or r_ij / 2 for eigenvalues closer than 1e-4 (second pass: 1e-8) of the spectrum's RMS, where the quotient
//      would be noise, and where the quotient exceeds kPreMaxTurn.  The FP32 phase resolves eigenvectors to 1e-7 of the
//      norm over the gap, so pairs with gaps below about 1e-5 ask for turns that a first-order step cannot make.
//   3. Two Newton-Schulz steps X = X (3 I - X^T X) / 2 make X orthonormal to rounding: g turns E in a column leave
//      d = g E^2, two steps take that to 0.4 d^4, which is 3e-15 for 20 turns of the largest E allowed.
// Then off(X^T A X) is near 1e-15 |A| for separated eigenvalues (no Jacobi sweep) and below 1e-5 |A| where some pairs
// were left alone (up to five sweeps, measured on groups of four).  Without the limit on E, matrices with groups of
// eigenvalues 1e-8 to 1e-4 apart lost X's orthonormality and with it everything done here: the sweeps then start from A.
// An eigenvector's sign (and a basis of an exactly degenerate space) is whatever the method happens to give:
// hf_eigh, whose eigenvectors the caller sees, keeps the plain Jacobi start and with it its signs; the SCF, which
// only uses the density they span, starts here (EighStart) up to the size that fits one SM.  Beyond it (the matrix in
// L2, the pairs over a cluster of 8 SMs) the phase took longer than the four or five sweeps that a start from the last
// iteration's eigenvectors leaves: n = 800 0.17 s a diagonalisation against 0.125 s.  Measured in a 4-water SCF (n = 100, 11
// diagonalisations): 29 ms of Jacobi kernels and their launch gaps before, 12.5 ms with this start.
constexpr int kPre32MinN = 4, kPre32MaxN = 240;
static bool uses_basis32(int n, EighStart start)
{
    return start == EighStart::kBasis32 && n >= kPre32MinN && n <= kPre32MaxN;
}
constexpr int kPre32Sweeps = 15;
constexpr double kPreMaxTurn = 1.0 / 256;

// scale[0] = max |a_ij|, scale[1] = max row sum of |a_ij|
__global__ void __launch_bounds__(256) k_pre_norms(int n, const double* __restrict__ A, unsigned long long* __restrict__ scale)
{
    const int i = blockIdx.x;
    double sum = 0.0, mx = 0.0;
    for (int j = threadIdx.x; j < n; j += 256) {
        const double v = fabs(A[(size_t)i * n + j]);
        sum += v;
        mx = fmax(mx, v);
    }
    __shared__ double s0[256], s1[256];
    s0[threadIdx.x] = sum;
    s1[threadIdx.x] = mx;
    __syncthreads();
    for (int s = 128; s > 0; s >>= 1) {
        if (threadIdx.x < s) {
            s0[threadIdx.x] += s0[threadIdx.x + s];
            s1[threadIdx.x] = fmax(s1[threadIdx.x], s1[threadIdx.x + s]);
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {  // non-negative doubles order as their bits
        atomicMax(&scale[0], (unsigned long long)__double_as_longlong(s1[0]));
        atomicMax(&scale[1], (unsigned long long)__double_as_longlong(s0[0]));
    }
}

// As = factor (A + A^T) / 2
__global__ void k_symmetrise(int n, const double* __restrict__ A, const unsigned long long* __restrict__ scale,
                             double* __restrict__ As)
{
    const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (long long)n * n) return;
    const int i = (int)(e / n), j = (int)(e % n);
    const double f = 0.5 * eigh_factor(scale);
    As[e] = f * A[e] + f * A[(size_t)j * n + i];
}

// G = A / s + c I with s = max |a_ij| and c = 1.25 max row sum / s: eigenvalues between 0.25 and 2.25 of the norm
__global__ void k_pre_shift(int n, const double* __restrict__ As, const unsigned long long* __restrict__ scale,
                            float* __restrict__ G)
{
    const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (long long)n * n) return;
    const double f = eigh_factor(scale), s = f * __longlong_as_double(scale[0]), rows = f * __longlong_as_double(scale[1]);
    const double inv = s > 0.0 ? 1.0 / s : 0.0;
    G[e] = (float)(As[e] * inv + (e / n == e % n ? 1.25 * rows * inv + (s > 0.0 ? 0.0 : 1.0) : 0.0));
}

__device__ __forceinline__ float warp_sum(float v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// One-sided Jacobi sweeps on the n <= 240 columns of G (column j at G + j n), eight elements of a column per lane.
__global__ void __launch_bounds__(1024) k_pre_sweeps(int n, float* __restrict__ Gg)
{
    constexpr int NC = (kPre32MaxN + 31) / 32;
    extern __shared__ float G[];
    __shared__ int changed;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int e = threadIdx.x; e < n * n; e += 1024) G[e] = Gg[e];
    const int m = n + (n & 1);
    for (int sweep = 0; sweep < kPre32Sweeps; sweep++) {
        if (threadIdx.x == 0) changed = 0;
        __syncthreads();
        for (int r = 0; r < m - 1; r++) {
            for (int k = warp; k < m / 2; k += 32) {
                int p, q;
                rr_pair(m, r, k, p, q);
                if (p >= n || q >= n) continue;  // the padding index of an odd n
                float* const gp = G + p * n;
                float* const gq = G + q * n;
                float x[NC], y[NC];
                float aa = 0.0f, bb = 0.0f, ab = 0.0f;
#pragma unroll
                for (int i = 0; i < NC; i++) {
                    const int e = lane + 32 * i;
                    x[i] = e < n ? gp[e] : 0.0f;
                    y[i] = e < n ? gq[e] : 0.0f;
                    aa = fmaf(x[i], x[i], aa);
                    bb = fmaf(y[i], y[i], bb);
                    ab = fmaf(x[i], y[i], ab);
                }
                aa = warp_sum(aa);
                bb = warp_sum(bb);
                ab = warp_sum(ab);
                const float lim = sqrtf(aa * bb);
                if (!(fabsf(ab) > 2e-7f * lim)) continue;  // warp-uniform
                // a pair this far from orthogonal asks for another sweep; the others end at its square or less
                if (fabsf(ab) > 3e-4f * lim && lane == 0) changed = 1;
                const float z = (bb - aa) / (2.0f * ab);
                const float t = copysignf(1.0f, z) / (fabsf(z) + sqrtf(1.0f + z * z));
                const float c = rsqrtf(1.0f + t * t), s = c * t;
#pragma unroll
                for (int i = 0; i < NC; i++) {
                    const int e = lane + 32 * i;
                    if (e < n) {
                        gp[e] = c * x[i] - s * y[i];
                        gq[e] = s * x[i] + c * y[i];
                    }
                }
            }
            __syncthreads();
        }
        const bool any = changed != 0;
        __syncthreads();
        if (!any) break;
    }
    for (int e = threadIdx.x; e < n * n; e += 1024) Gg[e] = G[e];
}

// X[:, j] = g_j / |g_j| (one warp per column), X row-major
__global__ void k_pre_normalise(int n, const float* __restrict__ G, double* __restrict__ X)
{
    const int j = (int)(((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
    if (j >= n) return;
    const float* const g = G + (size_t)j * n;
    double s = 0.0;
    for (int i = lane; i < n; i += 32) s += (double)g[i] * g[i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    const double r = 1.0 / sqrt(s);
    for (int i = lane; i < n; i += 32) X[(size_t)i * n + j] = g[i] * r;
}

// part[b] = partial sum of squares of S, lambda_i = s_ii / q_ii for Q = X^T X
__global__ void k_refine_norm(int n, const double* __restrict__ S, const double* __restrict__ Q, double* __restrict__ part,
                              double* __restrict__ lam)
{
    double t = 0.0;
    for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < (long long)n * n;
         e += (long long)gridDim.x * blockDim.x) {
        const double v = S[e];
        t += v * v;
        if (e / n == e % n) lam[e / n] = v / Q[e];
    }
    __shared__ double sm[256];
    sm[threadIdx.x] = t;
    __syncthreads();
    for (int s = blockDim.x / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s) sm[threadIdx.x] += sm[threadIdx.x + s];
        __syncthreads();
    }
    if (threadIdx.x == 0) part[blockIdx.x] = sm[0];
}

// Q (= X^T X) is overwritten with I + E: X (I + E) is the refined basis
__global__ void k_refine_correction(int n, int nb, double guard, const double* __restrict__ S, double* __restrict__ Q,
                                    const double* __restrict__ lam, const double* __restrict__ part)
{
    __shared__ double close;
    if (threadIdx.x < 32) {
        double a = 0.0;
        for (int i = threadIdx.x; i < nb; i += 32) a += part[i];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
        if (threadIdx.x == 0) close = guard * sqrt(a / n);
    }
    __syncthreads();
    const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (long long)n * n) return;
    const int i = (int)(e / n), j = (int)(e % n);
    const double r = (i == j ? 1.0 : 0.0) - Q[e];
    const double d = lam[j] - lam[i], t = S[e] + lam[j] * r;
    const bool turn = i != j && fabs(d) > close && fabs(t) <= kPreMaxTurn * fabs(d);
    Q[e] = (i == j ? 1.0 : 0.0) + (turn ? t / d : 0.5 * r);
}

// Q = X^T X -> (3 I - Q) / 2
__global__ void k_schulz(int n, double* __restrict__ Q)
{
    const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (e < (long long)n * n) Q[e] = (e / n == e % n ? 1.5 : 0.0) - 0.5 * Q[e];
}

// X (n x n, row-major) from the FP32 basis, S = X^T As X and Q = X^T X; -1 on a CUDA failure.
static int pre_eigenbasis(int n, const double* As, double*& X, double*& T, double* S, double* Q, float* G, double* part,
                          double* scal, cudaStream_t s)
{
    const unsigned long long* scale = (const unsigned long long*)scal;  // 2 words, then lambda
    double* lam = scal + 2;
    const unsigned nb = (unsigned)(((long long)n * n + 255) / 256);
    k_pre_shift<<<nb, 256, 0, s>>>(n, As, scale, G);
    if (cudaFuncSetAttribute(k_pre_sweeps, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             kPre32MaxN * kPre32MaxN * (int)sizeof(float)) != cudaSuccess) return -1;
    k_pre_sweeps<<<1, 1024, n * n * (int)sizeof(float), s>>>(n, G);
    k_pre_normalise<<<(n + 7) / 8, 256, 0, s>>>(n, G, X);
    for (int it = 0; it < 4; it++) {
        if (gemm(n, n, n, 1.0, X, n, true, X, n, false, 0.0, Q, n, s)) return -1;
        if (it < 2) {
            if (gemm(n, n, n, 1.0, As, n, false, X, n, false, 0.0, T, n, s)) return -1;
            if (gemm(n, n, n, 1.0, X, n, true, T, n, false, 0.0, S, n, s)) return -1;
            k_refine_norm<<<128, 256, 0, s>>>(n, S, Q, part, lam);
            k_refine_correction<<<nb, 256, 0, s>>>(n, 128, it == 0 ? 1e-4 : 1e-8, S, Q, lam, part);
        } else {
            k_schulz<<<nb, 256, 0, s>>>(n, Q);
        }
        if (gemm(n, n, n, 1.0, X, n, false, Q, n, false, 0.0, T, n, s)) return -1;
        std::swap(X, T);
    }
    if (gemm(n, n, n, 1.0, As, n, false, X, n, false, 0.0, T, n, s)) return -1;
    if (gemm(n, n, n, 1.0, X, n, true, T, n, false, 0.0, S, n, s)) return -1;
    if (gemm(n, n, n, 1.0, X, n, true, X, n, false, 0.0, Q, n, s)) return -1;
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

// Vout[:, j] = X[:, perm[j]]
__global__ void k_gather_cols(int n, int ncols, const double* __restrict__ X, const int* __restrict__ perm,
                              double* __restrict__ Vout)
{
    const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (long long)n * ncols) return;
    Vout[e] = X[(e / ncols) * n + perm[e % ncols]];
}

int jacobi_eigh(int n, const double* Ain, double* w, double* Vout, int ncols, double* work, int* iwork, int max_sweeps,
                double tol, EighStart start, int* sweeps_done, bool* basis_used, cudaStream_t s)
{
    // work: jacobi_work_doubles(n, start) doubles; iwork: m_pad ints
    const int m = n + (n & 1);
    if (n <= 0) return 0;
    const size_t mm = (size_t)m * m;
    double* A0 = work;
    double* A1 = A0 + mm;
    double* V = A1 + mm;
    double* part = V + mm;
    double* res = part + 512;
    double* key = res + 2;
    size_t mp = 1;
    while (mp < (size_t)m) mp <<= 1;
    double* scal = key + mp;  // two norms, then lambda
    // the FP32 start keeps A beside its products (As, X, T; G in FP32); otherwise A is read once, from A1
    bool pre = uses_basis32(n, start);
    double* As = pre ? work + jacobi_work_base(n) : A1;
    double* X = As + mm;
    double* T = X + mm;
    float* G = (float*)(T + mm);
    unsigned long long* scale = (unsigned long long*)scal;
    if (cudaMemsetAsync(scal, 0, sizeof(double) * 2, s) != cudaSuccess) return -1;
    k_pre_norms<<<n, 256, 0, s>>>(n, Ain, scale);
    k_symmetrise<<<(unsigned)(((long long)n * n + 255) / 256), 256, 0, s>>>(n, Ain, scale, As);
    double* cur = A0;
    double* nxt = A1;
    const unsigned nbm = (unsigned)((mm + 255) / 256);
    double h[2];
    auto off_norms = [&](int k, const double* M) -> int {  // h = sums of squares off the diagonal and in all
        k_offdiag<<<256, 256, 0, s>>>(k, M, part);
        k_sum2<<<1, 256, 0, s>>>(256, part, res);
        if (cudaMemcpyAsync(h, res, sizeof(h), cudaMemcpyDeviceToHost, s) != cudaSuccess) return -1;
        return cudaStreamSynchronize(s) == cudaSuccess ? 0 : -1;
    };
    // The Jacobi sweeps start from S = X^T A X (in A1) when X came out orthonormal (a matrix that is not finite, or an
    // FP32 phase that did not converge, shows here), else from A itself.
    if (pre) {
        if (pre_eigenbasis(n, As, X, T, A1, V, G, part, scal, s)) return -1;
        if (off_norms(n, V)) return -1;  // Q = X^T X: off-diagonal part and sum of squares (n for the identity)
        const double lim = 4e-16 * n;
        pre = h[0] <= lim * lim && fabs(h[1] - n) <= lim * n;
    }
    if (basis_used) *basis_used = pre;
    // padding eigenvalue: a zero-coupled padding entry only needs to be distinct and is dropped from the output.
    k_jacobi_init<<<nbm, 256, 0, s>>>(n, m, pre ? A1 : As, A0, V, 0.0);
    int sweep = 0;
    for (sweep = 0; sweep < max_sweeps; sweep++) {
        if (off_norms(m, cur)) return -1;
        // A is scaled, so its norm overflows only if an element was infinite or NaN: no eigenpairs, and no sort of NaN
        // keys, which would bring the padding's index (0x7fffffff) into the permutation
        if (!isfinite(h[1])) return 1;
        if (h[0] <= tol * tol * h[1] || h[0] == 0.0) break;
        for (int r = 0; r < m - 1; r++) {
            // every entry of Anew belongs to exactly one (row pair, column pair) block of this round
            if (launch_jacobi_round(m, r, cur, nxt, V, s)) return -1;
            std::swap(cur, nxt);
        }
        if (cudaGetLastError() != cudaSuccess) return -1;
    }
    if (sweeps_done) *sweeps_done = sweep;
    k_diag_keys<<<(unsigned)((mp + 255) / 256), 256, 0, s>>>(m, cur, key, iwork, (int)mp);
    if (bitonic_sort_desc(key, iwork, (int)mp, (int)mp, s) != 0) return -1;
    // when n is odd the padding index m-1 carries eigenvalue 0 and must be skipped: drop it from perm
    if (n != m) {
        k_drop_index<<<1, 1, 0, s>>>(m, iwork, m - 1);
    }
    const unsigned nbg = (unsigned)(((long long)n * ncols + 255) / 256);
    if (!pre) {
        k_gather_eig<<<nbg, 256, 0, s>>>(n, m, ncols, cur, V, iwork, scale, w, Vout);
    } else {
        // eigenvectors X V: with no sweep V is the identity and the sorted columns of X are the result
        double* out = sweep ? T : Vout;
        if (sweep) {
            k_gather_eig<<<nbg, 256, 0, s>>>(n, m, ncols, cur, V, iwork, scale, w, out);
            if (gemm(n, ncols, n, 1.0, X, n, false, T, ncols, false, 0.0, Vout, ncols, s)) return -1;
        } else {
            k_gather_eig<<<nbg, 256, 0, s>>>(n, m, ncols, cur, V, iwork, scale, w, As);  // As is done: only w is kept
            k_gather_cols<<<nbg, 256, 0, s>>>(n, ncols, X, iwork, out);
        }
    }
    if (cudaGetLastError() != cudaSuccess) return -1;
    return sweep >= max_sweeps ? 1 : 0;
}

// ---------------------------------------------------------------- helpers --
__global__ void k_antisym(int n, const double* __restrict__ A, double* __restrict__ E)
{
    const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (long long)n * n) return;
    const int i = (int)(e / n), j = (int)(e % n);
    E[e] = A[e] - A[(size_t)j * n + i];
}

int antisym(int n, const double* A, double* E, cudaStream_t s)
{
    k_antisym<<<(unsigned)(((long long)n * n + 255) / 256), 256, 0, s>>>(n, A, E);
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

// out[k] = <X, Y_k> for k < nk (Y_k = Ys[k]); partial sums in part[nk][256]
__global__ void k_dots(long long len, const double* __restrict__ X, const double* const* __restrict__ Ys,
                       double* __restrict__ part)
{
    __shared__ double sm[256];
    const double* Y = Ys[blockIdx.y];
    double acc = 0.0;
    for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < len; e += (long long)gridDim.x * blockDim.x)
        acc += X[e] * Y[e];
    sm[threadIdx.x] = acc;
    __syncthreads();
    for (int s = blockDim.x / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s) sm[threadIdx.x] += sm[threadIdx.x + s];
        __syncthreads();
    }
    if (threadIdx.x == 0) part[blockIdx.y * gridDim.x + blockIdx.x] = sm[0];
}

__global__ void k_dots_final(int nk, int nb, const double* __restrict__ part, double* __restrict__ out)
{
    const int k = blockIdx.x;
    __shared__ double sm[256];
    double a = 0.0;
    for (int i = threadIdx.x; i < nb; i += blockDim.x) a += part[k * nb + i];
    sm[threadIdx.x] = a;
    __syncthreads();
    for (int s = blockDim.x / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s) sm[threadIdx.x] += sm[threadIdx.x + s];
        __syncthreads();
    }
    if (threadIdx.x == 0 && k < nk) out[k] = sm[0];
}

int dots(long long len, const double* X, const double* const* Ys_dev, int nk, double* part, double* out,
         cudaStream_t s)
{
    dim3 grid(128, nk);
    k_dots<<<grid, 256, 0, s>>>(len, X, Ys_dev, part);
    k_dots_final<<<nk, 256, 0, s>>>(nk, 128, part, out);
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

// Pulay DIIS: B[m x m] (Gram of error vectors) -> solve [B -1; -1 0][c; l] = [0; -1]
// by Gaussian elimination with partial pivoting (one thread, m <= 16).
// status: 0 ok, 1 singular.
__global__ void k_diis_solve(int m, const double* __restrict__ B, double* __restrict__ coef, int* __restrict__ status)
{
    double a[17][18];
    const int n = m + 1;
    for (int i = 0; i < m; i++) {
        for (int j = 0; j < m; j++) a[i][j] = B[i * m + j];
        a[i][m] = -1.0;
        a[i][n] = 0.0;
    }
    for (int j = 0; j < m; j++) a[m][j] = -1.0;
    a[m][m] = 0.0;
    a[m][n] = -1.0;
    // scale rows of the Gram block by its largest diagonal to keep pivots moderate
    double dmax = 0.0;
    for (int i = 0; i < m; i++) dmax = fmax(dmax, fabs(a[i][i]));
    if (dmax > 0.0)
        for (int i = 0; i < m; i++)
            for (int j = 0; j < m; j++) a[i][j] /= dmax;
    for (int c = 0; c < n; c++) {
        int piv = c;
        for (int r = c + 1; r < n; r++)
            if (fabs(a[r][c]) > fabs(a[piv][c])) piv = r;
        if (fabs(a[piv][c]) < 1e-300) {
            *status = 1;
            return;
        }
        if (piv != c)
            for (int k = 0; k <= n; k++) {
                const double t = a[c][k];
                a[c][k] = a[piv][k];
                a[piv][k] = t;
            }
        for (int r = c + 1; r < n; r++) {
            const double f = a[r][c] / a[c][c];
            for (int k = c; k <= n; k++) a[r][k] -= f * a[c][k];
        }
    }
    double x[17];
    for (int r = n - 1; r >= 0; r--) {
        double v = a[r][n];
        for (int k = r + 1; k < n; k++) v -= a[r][k] * x[k];
        x[r] = v / a[r][r];
    }
    for (int i = 0; i < m; i++) coef[i] = x[i];
    *status = 0;
}

int diis_solve(int m, const double* B, double* coef, int* status, cudaStream_t s)
{
    k_diis_solve<<<1, 1, 0, s>>>(m, B, coef, status);
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

// out = sum_k coef[k] * Xs[k]
__global__ void k_lincomb(long long len, int nk, const double* const* __restrict__ Xs, const double* __restrict__ coef,
                          double* __restrict__ out)
{
    const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= len) return;
    double v = 0.0;
    for (int k = 0; k < nk; k++) v += coef[k] * Xs[k][e];
    out[e] = v;
}

int lincomb(long long len, int nk, const double* const* Xs_dev, const double* coef, double* out, cudaStream_t s)
{
    k_lincomb<<<(unsigned)((len + 255) / 256), 256, 0, s>>>(len, nk, Xs_dev, coef, out);
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

// RMS of A - B into out[0] (partials in part[256])
__global__ void k_sqdiff(long long len, const double* __restrict__ A, const double* __restrict__ B,
                         double* __restrict__ part)
{
    __shared__ double sm[256];
    double acc = 0.0;
    for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < len; e += (long long)gridDim.x * blockDim.x) {
        const double d = A[e] - B[e];
        acc += d * d;
    }
    sm[threadIdx.x] = acc;
    __syncthreads();
    for (int s = blockDim.x / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s) sm[threadIdx.x] += sm[threadIdx.x + s];
        __syncthreads();
    }
    if (threadIdx.x == 0) part[blockIdx.x] = sm[0];
}

__global__ void k_rms_final(long long len, const double* __restrict__ part, double* __restrict__ out)
{
    __shared__ double sm[256];
    sm[threadIdx.x] = part[threadIdx.x];
    __syncthreads();
    for (int s = blockDim.x / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s) sm[threadIdx.x] += sm[threadIdx.x + s];
        __syncthreads();
    }
    if (threadIdx.x == 0) *out = sqrt(sm[0] / (double)len);
}

int rms_diff(long long len, const double* A, const double* B, double* part, double* out, cudaStream_t s)
{
    k_sqdiff<<<256, 256, 0, s>>>(len, A, B, part);
    k_rms_final<<<1, 256, 0, s>>>(len, part, out);
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

// X = U diag(f(s)) U^T helper: Us[:, j] = U[:, j] * scale(s_j), zero for dropped vectors
__global__ void k_scale_cols(int n, int ncols, const double* __restrict__ U, const double* __restrict__ s,
                             double power, double drop_below, double* __restrict__ out)
{
    const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (long long)n * ncols) return;
    const int j = (int)(e % ncols);
    const double sj = s[j];
    out[e] = sj > drop_below ? U[e] * pow(sj, power) : 0.0;
}

int scale_cols(int n, int ncols, const double* U, const double* s, double power, double drop_below, double* out,
               cudaStream_t st)
{
    k_scale_cols<<<(unsigned)(((long long)n * ncols + 255) / 256), 256, 0, st>>>(n, ncols, U, s, power, drop_below, out);
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

}  // namespace hf

namespace hf {
size_t jacobi_work_doubles(int n, EighStart start)
{
    const size_t m = (size_t)(n + (n & 1));
    return jacobi_work_base(n) + (uses_basis32(n, start) ? 3 * m * m + (m * m + 1) / 2 : 0);  // As, X, T; G in FP32
}
size_t jacobi_work_ints(int n)
{
    const size_t m = (size_t)(n + (n & 1));
    size_t mp = 1;
    while (mp < m) mp <<= 1;
    return mp;
}
}  // namespace hf
