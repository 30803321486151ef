// Nuclear repulsion energy (Section 3: the one-electron part is computed once per geometry; S, T and V are in
// onee_herm.cuh).
#include <math.h>

#include "setup.cuh"

namespace hf {

__global__ void k_nuclear_repulsion(int n_atoms, const double* __restrict__ xyz, const double* __restrict__ Z,
                                    double* __restrict__ out)
{
    // single block, fixed-order reduction
    __shared__ double sm[256];
    double e = 0.0;
    for (int a = threadIdx.x / 32; a < n_atoms; a += blockDim.x / 32)
        for (int b = threadIdx.x % 32; b < a; b += 32) {
            const double dx = xyz[3 * a] - xyz[3 * b], dy = xyz[3 * a + 1] - xyz[3 * b + 1],
                         dz = xyz[3 * a + 2] - xyz[3 * b + 2];
            e += Z[a] * Z[b] / sqrt(dx * dx + dy * dy + dz * dz);
        }
    sm[threadIdx.x] = e;
    __syncthreads();
    for (int s = blockDim.x / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s) sm[threadIdx.x] += sm[threadIdx.x + s];
        __syncthreads();
    }
    if (threadIdx.x == 0) *out = sm[0];
}

int launch_nuclear_repulsion(int n_atoms, const double* xyz, const double* Z, double* out, cudaStream_t s)
{
    k_nuclear_repulsion<<<1, 256, 0, s>>>(n_atoms, xyz, Z, out);
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

}  // namespace hf
