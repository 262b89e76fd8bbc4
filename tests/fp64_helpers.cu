// the square root and the division of the FP64 pair sums, element by element
#include "sph_pairmath.cuh"

__global__ void k_helpers(int64_t n, const double* x, const double* num, double* root, double* quot, double* ref_root,
                          double* ref_quot)
{
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        root[i] = sphg::sqrt_fp64(x[i]);
        quot[i] = sphg::div_fp64(num[i], x[i]);
        ref_root[i] = sqrt(x[i]);
        ref_quot[i] = num[i] / x[i];
    }
}

extern "C" int helpers(int64_t n, const double* x, const double* num, double* root, double* quot, double* ref_root, double* ref_quot)
{
    k_helpers<<<256, 256>>>(n, x, num, root, quot, ref_root, ref_quot);
    return (int)cudaDeviceSynchronize();
}
