// Kernels that run single device functions of the library on given values
// (compiled and loaded by the tests that include them by name).
#include "lbmp_common.cuh"

using namespace lbmp;

// every thread of one block takes the same n cells through obs_cell; the block's four sums
static __global__ void obs_kernel(int n, const float2* phi, const float* rho, const float* u, const float* ph, double* out)
{
    __shared__ double sm[4 * 4];
    ObsAcc acc = {};
    for (int i = 0; i < n; ++i) obs_cell(acc, phi[i], rho[i], u + 3 * i, ph[i]);
    obs_block(acc, sm, out);
}

template <class T>
static cudaError_t to_device(T** dst, const T* src, size_t n)
{
    cudaError_t e = cudaMalloc(dst, n * sizeof(T));
    return e == cudaSuccess ? cudaMemcpy(*dst, src, n * sizeof(T), cudaMemcpyHostToDevice) : e;
}

extern "C" int obs_sums(int n, const float* phi, const float* rho, const float* u, const float* ph, double* out)
{
    float2* dphi = nullptr;
    float *drho = nullptr, *du = nullptr, *dph = nullptr;
    double* dout = nullptr;
    cudaError_t e = to_device(&dphi, (const float2*)phi, n);
    if (e == cudaSuccess) e = to_device(&drho, rho, n);
    if (e == cudaSuccess) e = to_device(&du, u, 3 * (size_t)n);
    if (e == cudaSuccess) e = to_device(&dph, ph, n);
    if (e == cudaSuccess) e = cudaMalloc(&dout, 4 * sizeof(double));
    if (e == cudaSuccess) {
        obs_kernel<<<1, 128>>>(n, dphi, drho, du, dph, dout);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpy(out, dout, 4 * sizeof(double), cudaMemcpyDeviceToHost);
    cudaFree(dphi), cudaFree(drho), cudaFree(du), cudaFree(dph), cudaFree(dout);
    return (int)e;
}
