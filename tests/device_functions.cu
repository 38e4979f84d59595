// Kernels that run single device functions of the library on given values
// (compiled and loaded by the tests that include them by name).
#include "lbmp_common.cuh"

using namespace lbmp;

// every thread of one block takes the same n cells through obs_cell; the block's four sums
static __global__ void obs_kernel(int n, const float2* phi, const float* rho, const float* u, const float* ph, double* out)
{
    __shared__ ObsShared<128> sm;
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

// all 2^23 significands at the exponents e0, e0 + 1, ...: how many results of
// recip (fn 0), root (1) and third (2) differ from the rounded quotient or root
static __global__ void scan_kernel(int fn, int e0, bool negative, unsigned* bad)
{
    const unsigned bits = (unsigned)(e0 + (int)blockIdx.y + 127) << 23 | (negative ? 0x80000000u : 0u);
    unsigned n = 0;
    for (unsigned m = blockIdx.x * blockDim.x + threadIdx.x; m < (1u << 23); m += gridDim.x * blockDim.x) {
        const float x = __uint_as_float(bits | m);
        const float got = fn == 0 ? recip(x) : (fn == 1 ? root(x) : third(x));
        const float want = fn == 0 ? __frcp_rn(x) : (fn == 1 ? __fsqrt_rn(x) : __fdiv_rn(x, 3.0f));
        n += __float_as_uint(got) != __float_as_uint(want);
    }
    if (n) atomicAdd(bad + blockIdx.y, n);
}

extern "C" int scan_rounded(int fn, int e0, int n, int negative, unsigned* bad)
{
    unsigned* d = nullptr;
    cudaError_t e = cudaMalloc(&d, n * sizeof(unsigned));
    if (e == cudaSuccess) e = cudaMemset(d, 0, n * sizeof(unsigned));
    if (e == cudaSuccess) {
        scan_kernel<<<dim3(64, n), 256>>>(fn, e0, negative != 0, d);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpy(bad, d, n * sizeof(unsigned), cudaMemcpyDeviceToHost);
    cudaFree(d);
    return (int)e;
}

// the largest relative error of recip_sqrt (out[0]) and of the rounded
// reciprocal of the rounded root (out[1]) over all significands at the exponents
// e0 .. e0 + n - 1, in units of 2^-24
static __global__ void scan_recip_sqrt_kernel(int e0, int* worst)
{
    const unsigned bits = (unsigned)(e0 + (int)blockIdx.y + 127) << 23;
    float w[2] = {0.f, 0.f};
    for (unsigned m = blockIdx.x * blockDim.x + threadIdx.x; m < (1u << 23); m += gridDim.x * blockDim.x) {
        const float x = __uint_as_float(bits | m);
        const double s = sqrt((double)x);
        const float got[2] = {recip_sqrt(x), __frcp_rn(__fsqrt_rn(x))};
        for (int k = 0; k < 2; ++k) w[k] = fmaxf(w[k], (float)(fabs((double)got[k] * s - 1.0) * 16777216.0));
    }
    for (int k = 0; k < 2; ++k) atomicMax(worst + k, __float_as_int(w[k]));  // positive: ordered as integers
}

extern "C" int scan_recip_sqrt(int e0, int n, float* out)
{
    int* d = nullptr;
    cudaError_t e = cudaMalloc(&d, 2 * sizeof(int));
    if (e == cudaSuccess) e = cudaMemset(d, 0, 2 * sizeof(int));
    if (e == cudaSuccess) {
        scan_recip_sqrt_kernel<<<dim3(64, n), 256>>>(e0, d);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpy(out, d, 2 * sizeof(int), cudaMemcpyDeviceToHost);
    cudaFree(d);
    return (int)e;
}
