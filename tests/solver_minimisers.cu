// The element minimisers that the solve kernels inline, as kernels over
// arrays: quartic_min32x2 (column pairs of the mixed kernels) and
// elem_min64_seeded / elem_min64_linear (columns of the FP64 kernel).  The
// quartic benchmark's entry points run variants of their own, so the tests
// reach these through a small library compiled from the same headers.
#include <cuda_runtime.h>

#include "quartic32.cuh"

using namespace admm_impl;

namespace {

__global__ void pairs_kernel(const float2 *A, const float2 *B, const float2 *C, const float2 *D, const float2 *lo,
                             const float2 *hi, int pairs, int mode, bool tiny, float2 *x)
{
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    unsigned esc = 0;
    if (t < pairs) x[t] = quartic_min32x2(A[t], B[t], C[t], D[t], lo[t], hi[t], mode, esc, tiny);
}

// the choice of column64: no losses where b2 = b1 = 0
__global__ void elements_kernel(const double *b2, const double *b1, const double *u, const double *C, const double *Dh,
                                const double *hr1, const double *lo, const double *hi, int n, int mode, double *x)
{
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n) return;
    if (b2[t] == 0.0 && b1[t] == 0.0) x[t] = elem_min64_linear(C[t], Dh[t], lo[t], hi[t]);
    else x[t] = elem_min64_seeded({b2[t], b1[t], u[t], C[t], Dh[t], hr1[t]}, (float)hr1[t], lo[t], hi[t], mode);
}

} // namespace

extern "C" {

// Device pointers; return a cudaError_t.
int solver_pairs(const float *A, const float *B, const float *C, const float *D, const float *lo, const float *hi,
                 int pairs, int mode, int tiny_c, float *x)
{
    pairs_kernel<<<(pairs + 127) / 128, 128>>>((const float2 *)A, (const float2 *)B, (const float2 *)C,
                                               (const float2 *)D, (const float2 *)lo, (const float2 *)hi, pairs, mode,
                                               tiny_c != 0, (float2 *)x);
    const cudaError_t e = cudaGetLastError();
    return e != cudaSuccess ? e : cudaDeviceSynchronize();
}

int solver_elements(const double *b2, const double *b1, const double *u, const double *C, const double *Dh,
                    const double *hr1, const double *lo, const double *hi, int n, int mode, double *x)
{
    elements_kernel<<<(n + 127) / 128, 128>>>(b2, b1, u, C, Dh, hr1, lo, hi, n, mode, x);
    const cudaError_t e = cudaGetLastError();
    return e != cudaSuccess ? e : cudaDeviceSynchronize();
}

} // extern "C"
