// Arithmetic throughput probe: the FP32, FP64 and 64-bit integer rates of the
// device, measured the way the step kernels use them (independent dependency
// chains per thread, every SM filled).  It corroborates the peaks that the
// benchmark derives from unit counts and clocks; it is not part of the method.
//
//   int alu_fma_rate(int fp64, int iters, double* flops_per_s, double* ms)
//   int alu_int_rate(int what, int iters, double* ops_per_s, double* ms)
//
// Launches 8 x (SM count) CTAs of 256 threads; each thread runs 8 chains of
// 4 x `iters` FMAs (2 flops each), or of mad.wide.s32 (what = 0: 32 x 32 -> 64
// bit multiply-adds), of 64-bit additions (what = 1) or of both in turn (what =
// 2).  Returns 0, or the CUDA error code.
#include <cuda_runtime.h>

namespace {

template <typename T>
__global__ void __launch_bounds__(256) fma_chains(T* out, int iters, T b, T c) {
    T a0 = (T)threadIdx.x, a1 = a0 + (T)1, a2 = a0 + (T)2, a3 = a0 + (T)3;
    T a4 = a0 + (T)4, a5 = a0 + (T)5, a6 = a0 + (T)6, a7 = a0 + (T)7;
    for (int i = 0; i < iters; ++i) {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            a0 = a0 * b + c; a1 = a1 * b + c; a2 = a2 * b + c; a3 = a3 * b + c;
            a4 = a4 * b + c; a5 = a5 * b + c; a6 = a6 * b + c; a7 = a7 * b + c;
        }
    }
    const T s = ((a0 + a1) + (a2 + a3)) + ((a4 + a5) + (a6 + a7));
    if (s == (T)-12345.0) out[blockIdx.x * blockDim.x + threadIdx.x] = s;   // keeps the chains live
}

// a + x y, or a + c (in PTX: the compiler folds a sum with a constant)
template <int WHAT>
__device__ __forceinline__ long long int_op(long long a, int x, int y, long long c) {
    long long r;
    if constexpr (WHAT == 0) asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(x), "r"(y), "l"(a));
    else asm("add.s64 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(c));
    return r;
}
template <int WHAT>
__global__ void __launch_bounds__(256) int_chains(long long* out, int iters, int b, long long c) {
    long long a[8], d[8];
    int x[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        a[k] = (long long)threadIdx.x * c + k;
        d[k] = a[k] * 77 + c;
        x[k] = (int)threadIdx.x * b + k;
    }
    for (int i = 0; i < iters; ++i) {
#pragma unroll
        for (int k = 0; k < 32; ++k) {
            const bool add = WHAT == 1 || (WHAT == 2 && (k & 1));
            a[k & 7] = add ? int_op<1>(a[k & 7], 0, 0, d[k & 7]) : int_op<0>(a[k & 7], x[k & 7], x[(k + 1) & 7], 0);
        }
    }
    long long s = 0;
#pragma unroll
    for (int k = 0; k < 8; ++k) s ^= a[k];
    if (s == 0x123456789abcdefLL) out[blockIdx.x * blockDim.x + threadIdx.x] = s;   // keeps the chains live
}

// five timed launches of k(out, iters) after a warm-up; ops: operations per thread and iteration
template <typename T, class K>
int run(K launch, int iters, double ops, double* rate, double* ms_out) {
    int dev = 0, nsm = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return (int)e;
    const int blocks = 8 * nsm, threads = 256;
    T* out = nullptr;
    if ((e = cudaMalloc(&out, sizeof(T) * blocks * threads)) != cudaSuccess) return (int)e;
    cudaEvent_t e0, e1;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    launch(blocks, threads, out, iters / 8);
    cudaEventRecord(e0);
    for (int r = 0; r < 5; ++r) launch(blocks, threads, out, iters);
    cudaEventRecord(e1);
    e = cudaEventSynchronize(e1);
    float ms = 0;
    if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, e0, e1);
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    cudaFree(out);
    if (e != cudaSuccess) return (int)e;
    *rate = 5.0 * ops * (double)iters * blocks * threads / (ms * 1e-3);
    *ms_out = ms / 5.0;
    return 0;
}
template <typename T>
int run_fma(int iters, double* flops, double* ms) {
    const T b = (T)0.999999, c = (T)1e-7;
    return run<T>([=](int g, int t, T* out, int it) { fma_chains<T><<<g, t>>>(out, it, b, c); }, iters, 2.0 * 32, flops, ms);
}
template <int WHAT>
int run_int(int iters, double* ops, double* ms) {
    return run<long long>([](int g, int t, long long* out, int it) { int_chains<WHAT><<<g, t>>>(out, it, 1234567, 987654321LL); },
                          iters, 32.0, ops, ms);
}

}  // namespace

extern "C" int alu_fma_rate(int fp64, int iters, double* flops_per_s, double* ms) {
    if (!flops_per_s || !ms || iters <= 0) return -1;
    return fp64 ? run_fma<double>(iters, flops_per_s, ms) : run_fma<float>(iters, flops_per_s, ms);
}
extern "C" int alu_int_rate(int what, int iters, double* ops_per_s, double* ms) {
    if (!ops_per_s || !ms || iters <= 0) return -1;
    return what == 0 ? run_int<0>(iters, ops_per_s, ms) : what == 1 ? run_int<1>(iters, ops_per_s, ms)
                                                                    : run_int<2>(iters, ops_per_s, ms);
}
