// The interpolation weights of csrc/coef.cuh, evaluated on arrays: tests/test_gpu_coef.py
// compares them with multi-digit decimal arithmetic.
#include <cuda_runtime.h>
#include <stdint.h>

#include "coef.cuh"

namespace {

// form 0: Coef64, 1: Coef64Series (E, alpha, beta, gamma); 2: Coef64D (these four and their derivatives
// E_x, alpha_x, beta_x, gamma_x, alpha_p, beta_p, gamma_p); 3: rcp64(x), 1 / x, div64(p, x), p / x
__global__ void k_eval(int form, int n, const double *x, const double *p, const int *para, double *out)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        double *o = out + 11 * (int64_t)i;
        if (form == 0) rtk::Coef64::eval(x[i], p[i], para[i] != 0, o[0], o[1], o[2], o[3]);
        if (form == 1) rtk::Coef64Series::eval(x[i], p[i], para[i] != 0, o[0], o[1], o[2], o[3]);
        if (form == 2)
            rtk::Coef64D::eval(x[i], p[i], para[i] != 0, o[0], o[1], o[2], o[3], o[4], o[5], o[6], o[7], o[8], o[9], o[10]);
        if (form == 3) {
            o[0] = rtk::rcp64(x[i]);
            o[1] = 1.0 / x[i];
            o[2] = rtk::div64(p[i], x[i]);
            o[3] = p[i] / x[i];
        }
    }
}

}  // namespace

// Host arrays; out holds 11 values a point.  Returns the CUDA error.
extern "C" int coef_eval(int form, int n, const double *x, const double *p, const int *para, double *out)
{
    double *dx = nullptr, *dp = nullptr, *dout = nullptr;
    int *dpara = nullptr;
    cudaError_t e = cudaMalloc(&dx, sizeof(double) * (size_t)n);
    if (e == cudaSuccess) e = cudaMalloc(&dp, sizeof(double) * (size_t)n);
    if (e == cudaSuccess) e = cudaMalloc(&dout, 11 * sizeof(double) * (size_t)n);
    if (e == cudaSuccess) e = cudaMalloc(&dpara, sizeof(int) * (size_t)n);
    if (e == cudaSuccess) e = cudaMemcpy(dx, x, sizeof(double) * (size_t)n, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(dp, p, sizeof(double) * (size_t)n, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(dpara, para, sizeof(int) * (size_t)n, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemset(dout, 0, 11 * sizeof(double) * (size_t)n);
    if (e == cudaSuccess) {
        k_eval<<<256, 128>>>(form, n, dx, dp, dpara, dout);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpy(out, dout, 11 * sizeof(double) * (size_t)n, cudaMemcpyDeviceToHost);
    cudaFree(dx);
    cudaFree(dp);
    cudaFree(dout);
    cudaFree(dpara);
    return (int)e;
}
