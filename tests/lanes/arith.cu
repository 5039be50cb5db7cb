// The number helpers of fx.cuh and solver.cuh over arrays: as host code (g++, the emulation's
// compat.cuh) and, compiled by nvcc, as a kernel per helper.
#include "solver.cuh"

using namespace pagd;

namespace {
struct ToF32 { __device__ float operator()(double x) const { return to_f32(x); } };
struct ToF64 { __device__ double operator()(float x) const { return to_f64(x); } };
struct Rcp { __device__ double operator()(double x) const { return rcp64(x); } };
struct Div { __device__ double2 operator()(double2 n) const { return div64(double2{n.x, 1.0}, n.y); } };  // n.x / n.y, 1 / n.y
// kappa, a / M = 4 / M -> 1 / (M kappa), L
struct Pre {
    double M, b0, b2, b4;
    __device__ double2 operator()(double kap) const {
        const Precond p = precond64(4.0, M, Beta{4.0 / M, b0, b2, b4}, kap);
        return double2{p.ik, p.L};
    }
};
// the sum of m FP32 values of each of the threads of a warp
struct Sum {
    const float* a;
    int m;
    __device__ double operator()(int i) const {
        Sum3 s;
        for (int q = 0; q < m; q++) s.add(a[(long long)i * m + q]);
        return s.warp_total();
    }
};

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
int arith_rcp(const double* a, double* b, long long n) { return apply(Rcp{}, a, b, n); }
int arith_div(const double2* a, double2* b, long long n) { return apply(Div{}, a, b, n / 2); }
int arith_sum(const float* a, const int* i, double* b, long long n, int m) { return apply(Sum{a, m}, i, b, n); }
int arith_pre(const double* a, double2* b, long long n) { return apply(Pre{1.3, 0.7, -2.0, 1.0}, a, b, n / 2); }
}
