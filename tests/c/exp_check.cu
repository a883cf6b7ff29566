// exp_rounded and exp_cr of lb_fp64.cu over arrays in host memory (built as the library builds
// that unit, without multiply-add contraction). Returns the cudaError_t.
#include "lb_fp64.cu"

namespace lbsc {
namespace {

__global__ void k_exp(const double* __restrict__ x, double* __restrict__ y, double* __restrict__ z,
                      int n)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        y[i] = exp_rounded(x[i]);
        z[i] = exp_cr(x[i]);
    }
}

}  // namespace
}  // namespace lbsc

extern "C" int exp_check(const double* x, double* rounded, double* cr, int n)
{
    double* d = nullptr;
    const size_t bytes = sizeof(double) * (size_t)n;
    cudaError_t e = cudaMalloc((void**)&d, 3 * bytes);
    if (e != cudaSuccess) return (int)e;
    e = cudaMemcpy(d, x, bytes, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) {
        lbsc::k_exp<<<256, 128>>>(d, d + n, d + 2 * (size_t)n, n);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpy(rounded, d + n, bytes, cudaMemcpyDeviceToHost);
    if (e == cudaSuccess) e = cudaMemcpy(cr, d + 2 * (size_t)n, bytes, cudaMemcpyDeviceToHost);
    cudaFree(d);
    return (int)e;
}
