// Entry points of the debug library (libuncomp_debug.so) only: parts of the product that have no entry of their own, for tests.
#ifdef UNCOMP_DEBUG
#include "newton.cuh"
#include "wide_krylov.cuh"

namespace uncomp {
namespace {
template <typename T> __global__ void newton_kernel(const T *x, T *recip, T *root, int n) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        recip[i] = recip_newton(x[i]);
        root[i] = sqrt_newton(x[i]);
    }
}
}  // namespace
}  // namespace uncomp

extern "C" {

// reciprocals and square roots of n numbers, fp32 or fp64; the CUDA error of the launch
int uncomp_debug_newton(const void *d_x, void *d_recip, void *d_root, int n, int fp64, void *stream) {
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (fp64)
        uncomp::newton_kernel<double><<<256, 256, 0, st>>>(static_cast<const double *>(d_x), static_cast<double *>(d_recip),
                                                          static_cast<double *>(d_root), n);
    else
        uncomp::newton_kernel<float><<<256, 256, 0, st>>>(static_cast<const float *>(d_x), static_cast<float *>(d_recip),
                                                         static_cast<float *>(d_root), n);
    return (int)cudaGetLastError();
}

// 1 when the wide entropy of an n x n matrix starts with block Lanczos on a device that holds `ctas` of its CTAs at once
int uncomp_debug_krylov_applies(int n, int k, int ctas) { return uncomp::krylov_applies(n, k, ctas) ? 1 : 0; }

}  // extern "C"
#endif
