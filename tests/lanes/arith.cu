// The number helpers of fx.cuh over arrays: as host code (g++, the emulation's
// compat.cuh) and, compiled by nvcc, as a kernel per helper.
#include "fft.cuh"

using namespace pagd;

namespace {
struct ToF32 { __device__ float operator()(double x) const { return to_f32(x); } };
struct ToF64 { __device__ double operator()(float x) const { return to_f64(x); } };

#ifdef __CUDACC__
template <class F, class A, class B> __global__ void each(F f, const A* a, B* b, long long n) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) b[i] = f(a[i]);
}
template <class F, class A, class B> int apply(F f, const A* a, B* b, long long n) {
    if (n > 0) each<<<(unsigned)((n + 255) / 256), 256>>>(f, a, b, n);
    return (int)cudaDeviceSynchronize();
}
#else
template <class F, class A, class B> int apply(F f, const A* a, B* b, long long n) {
    for (long long i = 0; i < n; i++) b[i] = f(a[i]);
    return 0;
}
#endif
}  // namespace

extern "C" {
int arith_f32(const double* a, float* b, long long n) { return apply(ToF32{}, a, b, n); }
int arith_f64(const float* a, double* b, long long n) { return apply(ToF64{}, a, b, n); }
}
