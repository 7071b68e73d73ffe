// gks_probe.cu -- probes of the device: the FMA-chain throughput that the sweep
// kernels are compared against, and device arithmetic that differs from its
// host replica.  Compiled with the float32 kernels' arithmetic flags.
#include <cuda_runtime.h>

#include "../../include/gks.h"
#include "gks_device.cuh"

namespace {

constexpr int CHAINS = 16;  // independent FMA chains per thread (covers the pipeline latency)

template <typename T>
__global__ void __launch_bounds__(256) k_fma_chains(T* out, int iters, T b, T c)
{
    T a[CHAINS];
#pragma unroll
    for (int k = 0; k < CHAINS; ++k) a[k] = T(threadIdx.x + k) * T(1e-3);
    for (int i = 0; i < iters; ++i) {
#pragma unroll
        for (int k = 0; k < CHAINS; ++k) a[k] = fma(a[k], b, c);
    }
    T s = T(0);
#pragma unroll
    for (int k = 0; k < CHAINS; ++k) s += a[k];
    out[blockIdx.x * blockDim.x + threadIdx.x] = s;
}

template <typename T>
gks_status probe(double target_ms, double* tflops)
{
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return GKS_ECUDA;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return GKS_ECUDA;
    const int blocks = sms * 8, threads = 256;
    T* out = nullptr;
    if (cudaMalloc(&out, sizeof(T) * blocks * threads) != cudaSuccess) return GKS_ENOMEM;
    cudaEvent_t e0, e1;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    int iters = 256;
    double ms = 0.0;
    gks_status st = GKS_OK;
    for (int round = 0; round < 12; ++round) {  // grow until one launch takes target_ms
        cudaEventRecord(e0);
        k_fma_chains<T><<<blocks, threads>>>(out, iters, T(0.999999), T(1e-7));
        cudaEventRecord(e1);
        if (cudaEventSynchronize(e1) != cudaSuccess) { st = GKS_ECUDA; break; }
        float f = 0.f;
        cudaEventElapsedTime(&f, e0, e1);
        ms = f;
        if (ms >= target_ms || round == 11) break;
        iters = (int)(iters * (ms > 0.05 ? target_ms / ms * 1.05 : 8.0));
    }
    if (st == GKS_OK) {
        const double flops = 2.0 * CHAINS * (double)iters * blocks * threads;
        *tflops = flops / (ms * 1e-3) / 1e12;
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    cudaFree(out);
    return st;
}

template <typename T>
__global__ void k_half_space(const double* z, int n, double* half, double* gauss)
{
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    T h, g;
    gks::half_space_start<T>((T)z[i], T(1), h, g);
    half[i] = (double)h;
    gauss[i] = (double)g;
}

}  // namespace

extern "C" gks_status gks_eval_half_space(int precision, const double* z, int n, double* half, double* gauss)
{
    if (!z || !half || !gauss || n < 1) return GKS_EINVAL;
    const size_t bytes = sizeof(double) * (size_t)n;
    double* d = nullptr;  // z, then both results
    if (cudaMalloc(&d, 3 * bytes) != cudaSuccess) {
        cudaGetLastError();
        return GKS_ENOMEM;
    }
    cudaError_t e = cudaMemcpy(d, z, bytes, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) {
        const int blocks = (n - 1) / 256 + 1;
        if (precision == GKS_FP32_FLUX) k_half_space<float><<<blocks, 256>>>(d, n, d + n, d + 2 * (size_t)n);
        else k_half_space<double><<<blocks, 256>>>(d, n, d + n, d + 2 * (size_t)n);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpy(half, d + n, bytes, cudaMemcpyDeviceToHost);
    if (e == cudaSuccess) e = cudaMemcpy(gauss, d + 2 * (size_t)n, bytes, cudaMemcpyDeviceToHost);
    cudaFree(d);
    return e == cudaSuccess ? GKS_OK : GKS_ECUDA;
}

extern "C" gks_status gks_alu_peak(int precision, double target_ms, double* tflops)
{
    if (!tflops || !(target_ms > 0.0)) return GKS_EINVAL;
    return precision == GKS_FP32_FLUX ? probe<float>(target_ms, tflops) : probe<double>(target_ms, tflops);
}
