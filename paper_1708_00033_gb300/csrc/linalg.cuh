// Dense FP64 linear-algebra launchers used by the SCF driver.
#pragma once
#include <cuda_runtime.h>

namespace hf {

int gemm(int M, int N, int K, double alpha, const double* A, int lda, bool ta, const double* B, int ldb, bool tb,
         double beta, double* C, int ldc, cudaStream_t s);
// Eigen-decomposition of a symmetric n x n matrix by parallel cyclic Jacobi.
// w[ncols]: lowest ncols eigenvalues ascending; Vout[n x ncols] the matching
// eigenvectors as columns.  work: jacobi_work_doubles(n, start) doubles, iwork: jacobi_work_ints(n) ints.
// start: where the FP64 sweeps start, the matrix itself or an FP32 eigenbasis refined in FP64 (fewer or no sweeps
// left; the eigenvectors' signs then follow that basis).
// basis_used (nullable): whether the sweeps started from that basis (false where it does not apply or was rejected).
// Returns 0 converged, 1 not converged within max_sweeps or A not finite (w and Vout are then not written),
// -1 CUDA error.
enum class EighStart { kMatrix, kBasis32 };
int jacobi_eigh(int n, const double* A, double* w, double* Vout, int ncols, double* work, int* iwork, int max_sweeps,
                double tol, EighStart start, int* sweeps_done, bool* basis_used, cudaStream_t s);
size_t jacobi_work_doubles(int n, EighStart start);
size_t jacobi_work_ints(int n);
int antisym(int n, const double* A, double* E, cudaStream_t s);
int dots(long long len, const double* X, const double* const* Ys_dev, int nk, double* part, double* out,
         cudaStream_t s);
int diis_solve(int m, const double* B, double* coef, int* status, cudaStream_t s);
int lincomb(long long len, int nk, const double* const* Xs_dev, const double* coef, double* out, cudaStream_t s);
int rms_diff(long long len, const double* A, const double* B, double* part, double* out, cudaStream_t s);
int scale_cols(int n, int ncols, const double* U, const double* s, double power, double drop_below, double* out,
               cudaStream_t st);

}  // namespace hf
