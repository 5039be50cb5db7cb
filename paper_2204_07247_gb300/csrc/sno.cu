// sno.cu -- a small spectral neural operator that proposes the initial iterate
// of an implicit time step (the learned-guess form of the solver): forward,
// backward and Adam kernels, FP32, for sm_103a.
//
// The paper starts PAGD from the extrapolation u^n + rho (u^n - u^{n-1})
// (Sec. 3.4.2); the network learns the remaining correction
// r = u^{n+1} - (u^n + rho (u^n - u^{n-1})) from (u^n, u^{n-1}), and
// pagd_step_with_guess keeps its proposal only when its first PAGD direction
// is smaller than the extrapolation's.
//
// Network, per sample on an n0 x n1 periodic grid (np = n0 n1 points):
//   a    = [u^n, s_in (u^n - u^{n-1})]                     (2 channels)
//   v_0  = P a + b_P                                        (C channels)
//   z_l  = W_l v_l + b_l + K_l v_l,  v_{l+1} = GELU(z_l),   l = 0 .. L-1
//   out  = Q v_L + b_Q,   guess = extrapolation + s_out out
// with the spectral convolution
//   (K v)[o](x) = sum over kept modes m of w_m Re( sum_c R[o][c][m] F[c][m] e^{i k_m.x} ) / np,
//   F[c][m] = sum_x v[c](x) e^{-i k_m.x},
// kept modes k0 in [-M0/2, M0/2), k1 in [0, M1), w_m = 1 for k1 = 0 and 2
// otherwise (the omitted k1 < 0 half of a real field's spectrum).
//
// Parameters are one flat FP32 array in this order: P [C][2], b_P [C]; for
// each layer W [C][C] (W[o][c]), b [C], R [C][C][M0 M1][2] (R[o][c][m], re, im);
// Q [C], b_Q.  Only the kept modes of the DFTs are computed, one axis after the
// other; a layer is one pass over its activations (k_tile).
#include "../../include/pagd_sno.h"
#include "fft.cuh"

#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <new>
#include <string>

namespace {

constexpr int kThr = 256;
constexpr int kTile = 512;       // points of a tile (k_tile)
constexpr int kPitch = kTile + 4;  // of a channel's points in shared memory: rows 16 bytes apart in the banks

// A tile is kTile points: R = 16 / QC rows of the last axis (or 1 / JB of one), whose
// points x1 = j + J q (q < QC, J = n1 / QC) go one j to a lane, so that a lane
// holds a QC-point subsequence and the 32 lanes of a warp a whole row (J <= 32)
// or 32 of its residues.
struct SnoDims {
    int n0, n1, np, C, L, M0, M1, M;
    int QC, J, JB, R, NT;  // NT: tiles of a sample
    int ljb;               // log2 JB
};

// tanh form of GELU (Hendrycks and Gimpel, 2016), x s with s = (1 + tanh u) / 2.
// (As the logistic function of 2 u, by expf and a division, the errors of the
// proposals over 87 drawn networks were 6% larger, and inference of 8 states of
// 512^2 took 762 us instead of 751.)
__device__ __forceinline__ float gelu_s(float x) {
    const float k = 0.7978845608028654f;  // sqrt(2 / pi)
    return 0.5f * (1.f + tanhf(k * (x + 0.044715f * x * x * x)));
}
__device__ __forceinline__ float gelu_f(float x) { return x * gelu_s(x); }
// its derivative at x, s = gelu_s(x)
__device__ __forceinline__ float gelu_grad(float x, float s) {
    const float k = 1.5957691216057308f;
    return s + x * s * (1.f - s) * k * (1.f + 3.f * 0.044715f * x * x);
}

__device__ __forceinline__ int k0_of(int m0, int M0, int n0) { return m0 < M0 / 2 ? m0 : n0 - M0 + m0; }

// exp(-2 pi i j / n), j < n, from sincospif, for both axes: written by every
// call in one small launch, so that nothing in the workspace has to be kept
__global__ void k_tables(float2* t0, int n0, float2* t1, int n1) {
    int j = blockIdx.x * blockDim.x + threadIdx.x;
    const bool first = j < n0;
    if (!first) j -= n0;
    const int n = first ? n0 : n1;
    if (j >= n) return;
    float sn, cs;
    sincospif(-2.f * (float)j / (float)n, &sn, &cs);
    (first ? t0 : t1)[j] = float2{cs, sn};
}

// cos(2 pi k / 16)
__host__ __device__ constexpr float cos16(int k) {
    const float c[16] = {1.f, 0.92387953251128674f, 0.70710678118654752f, 0.38268343236508977f,
                         0.f, -0.38268343236508977f, -0.70710678118654752f, -0.92387953251128674f,
                         -1.f, -0.92387953251128674f, -0.70710678118654752f, -0.38268343236508977f,
                         0.f, 0.38268343236508977f, 0.70710678118654752f, 0.92387953251128674f};
    return c[k & 15];
}
__host__ __device__ constexpr float sin16(int k) { return cos16(k - 4 + 16); }

// Y[c] = sum_q x[q] exp(-2 pi i c q / QC), c = 0 .. QC / 2, of real x, from the
// even and odd parts of x
template <int QC> __device__ __forceinline__ void rdft(const float* x, float2* Y) {
    constexpr int h = QC / 2, st = 16 / QC;
    if constexpr (QC == 1) {
        Y[0] = make_float2(x[0], 0.f);
    } else {
        float S[h > 1 ? h : 1], D[h > 1 ? h : 1];
#pragma unroll
        for (int q = 1; q < h; q++) {
            S[q] = x[q] + x[QC - q];
            D[q] = x[q] - x[QC - q];
        }
#pragma unroll
        for (int c = 0; c <= h; c++) {
            float re = (c & 1) ? x[0] - x[h] : x[0] + x[h], im = 0.f;
#pragma unroll
            for (int q = 1; q < h; q++) {
                re = fmaf(S[q], cos16(c * q * st), re);
                if (c > 0 && c < h) im = fmaf(D[q], -sin16(c * q * st), im);
            }
            Y[c] = make_float2(re, im);
        }
    }
}
// y[q] = Re sum_c Z[c] exp(+2 pi i c q / QC), c < QC
template <int QC> __device__ __forceinline__ void irdft(const float2* Z, float* y) {
    constexpr int h = QC / 2, st = 16 / QC;
    if constexpr (QC == 1) {
        y[0] = Z[0].x;
    } else {
        float A[h > 1 ? h : 1], B[h > 1 ? h : 1];
#pragma unroll
        for (int c = 1; c < h; c++) {
            A[c] = Z[c].x + Z[QC - c].x;
            B[c] = Z[c].y - Z[QC - c].y;
        }
#pragma unroll
        for (int q = 0; q <= h; q++) {
            float e = (q & 1) ? Z[0].x - Z[h].x : Z[0].x + Z[h].x, o = 0.f;
#pragma unroll
            for (int c = 1; c < h; c++) {
                e = fmaf(A[c], cos16(c * q * st), e);
                if (q > 0 && q < h) o = fmaf(B[c], sin16(c * q * st), o);
            }
            y[q] = e - o;
            if (q > 0 && q < h) y[QC - q] = e + o;
        }
    }
}

// Sums of V = 2 MM values over the lanes of a warp, dealt to the lanes: each
// exchange halves the values a lane still holds.  On return lane l holds values
// l V / 32 .. (V = 32 or 64).
template <int V> __device__ __forceinline__ void reduce_deal(float* v, int lane) {
    int cnt = V;
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) {
        const bool up = (lane & s) != 0;
        const int hf = cnt / 2;
#pragma unroll
        for (int i = 0; i < V / 2; i++) {
            if (i < hf) {
                const float give = up ? v[i] : v[i + hf], keep = up ? v[i + hf] : v[i];
                v[i] = keep + __shfl_xor_sync(0xffffffffu, give, s);
            }
        }
        cnt = hf;
    }
}

// The same with the rounding errors beside the sums (two-sum): on return v holds
// the sums and e the errors.
template <int V> __device__ __forceinline__ void reduce_deal2(float* v, float* e, int lane) {
    int cnt = V;
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) {
        const bool up = (lane & s) != 0;
        const int hf = cnt / 2;
#pragma unroll
        for (int i = 0; i < V / 2; i++) {
            if (i < hf) {
                const float got = __shfl_xor_sync(0xffffffffu, up ? v[i] : v[i + hf], s);
                const float gotE = s < 16 ? __shfl_xor_sync(0xffffffffu, up ? e[i] : e[i + hf], s) : 0.f;
                const float keepE = s < 16 ? (up ? e[i + hf] : e[i]) : 0.f;
                v[i] = up ? v[i + hf] : v[i];
                e[i] = pagd::Sum3::two_sum(v[i], got) + (keepE + gotE);
            }
        }
        cnt = hf;
    }
}

// What a tile kernel does at its points (k_tile)
enum { T_LIFT, T_LAYER, T_GUESS, T_LOSS, T_BACK, T_BACK0 };

struct TileArgs {
    const float* prm;     // P, b_P (T_LIFT)
    const double *un, *unm1, *target;
    float s_in;
    double rho, s_out, inv_s_out, dscale;  // dscale = 2 / (np B)
    const float* W;       // the layer's W [C][C] and bias
    const float* bias;
    const float* Q;       // Q [C], b_Q
    const float2* G;      // modes [B][C][M] of the spectral part
    const float* vin;     // [B][C][np]: v_l, or dz_l
    const float* zprev;   // z_{l-1} (T_BACK)
    float* vout;          // v_{l+1}, or dz_{l-1}; nullable
    float* z;             // nullable
    float2* T;            // row transforms [B][C][n0 JB][M1] of the tile's output
    const float2 *tw0, *tw1;
    double* guess;
    double* loss;
    float* part;          // per-block sums: T_LOSS [C + 1][2], T_BACK0 [C][3]
};

// One tile of every channel, in one block:
//   the spectral part at the tile's points from its modes (first axis by a
//   direct sum over the M0 kept modes, last axis by twiddles and a QC-point
//   real transform per lane), the channel mixing W v, the pointwise function,
//   and the tile's part of the last-axis transform of the result, whose first-
//   axis sums k_cols takes.
// The activations are read and written once per layer; per point and channel
// the transforms cost 2 x 15 multiply-adds and the mixing C.  FP32 throughout.
// CT: channels rounded up to 16 or 32; MM: kept modes of the last axis to 16
// or 32.  Dynamic shared memory: tile_smem().
template <int MODE, int QC, int CT, int MM>
__global__ void __launch_bounds__(kThr, CT <= 16 ? 3 : 1) k_tile(SnoDims d, TileArgs a) {
    constexpr int R = 16 / QC;
    extern __shared__ __align__(16) float sm[];
    float* y = sm;                                  // [C][kPitch]
    float* sw = y + d.C * kPitch;                   // [CT][CT] row = output channel, [CT] bias
    float2* tj = (float2*)(sw + CT * CT + CT);      // [M1][32] exp(-2 pi i m1 j / n1)
    float2* U = tj + d.M1 * 32;                     // [R][C][M1]
    float2* e0 = U + R * d.C * d.M1;                // [R][M0] exp(-2 pi i k0 x0 / n0)
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, b = blockIdx.y;
    const int rg = blockIdx.x >> d.ljb, jb = blockIdx.x & (d.JB - 1), x00 = rg * R, j = jb * 32 + lane;
    const size_t bc = (size_t)b * d.C;
    for (int i = tid; i < d.M1 * 32; i += kThr) tj[i] = a.tw1[((i >> 5) * (jb * 32 + (i & 31))) & (d.n1 - 1)];
    if constexpr (MODE != T_LIFT) {
        for (int i = tid; i < CT * CT; i += kThr) {
            const int o = i / CT, c = i % CT;
            const bool in = o < d.C && c < d.C;
            sw[i] = !in ? 0.f : (MODE == T_BACK || MODE == T_BACK0) ? a.W[c * d.C + o] : a.W[o * d.C + c];
        }
        for (int i = tid; i < CT; i += kThr)
            sw[CT * CT + i] = (i < d.C && MODE != T_BACK && MODE != T_BACK0) ? a.bias[i] : 0.f;
        for (int i = tid; i < R * d.M0; i += kThr) {
            const int rr = i / d.M0, m0 = i - rr * d.M0;
            e0[i] = a.tw0[(k0_of(m0, d.M0, d.n0) * (x00 + rr)) & (d.n0 - 1)];
        }
        __syncthreads();
        // first axis: U[rr][o][m1] = w sum_m0 G[o][m0][m1] exp(+2 pi i k0 x0 / n0)
        const bool back = MODE == T_BACK || MODE == T_BACK0;
        const float inv = 1.f / (float)d.np;
        for (int i = tid; i < d.C * d.M1; i += kThr) {
            const int o = i / d.M1, m1 = i - o * d.M1;
            const float2* g = a.G + (bc + o) * d.M + m1;
            float2 s[R];
#pragma unroll
            for (int rr = 0; rr < R; rr++) s[rr] = make_float2(0.f, 0.f);
#pragma unroll 4
            for (int m0 = 0; m0 < d.M0; m0++) {
                const float2 v = g[m0 * d.M1];
#pragma unroll
                for (int rr = 0; rr < R; rr++) {
                    const float2 e = e0[rr * d.M0 + m0];  // conjugated
                    s[rr].x += v.x * e.x + v.y * e.y;
                    s[rr].y += v.y * e.x - v.x * e.y;
                }
            }
            const float w = back ? 1.f : (m1 == 0 ? inv : 2.f * inv);
#pragma unroll
            for (int rr = 0; rr < R; rr++) U[(rr * d.C + o) * d.M1 + m1] = make_float2(w * s[rr].x, w * s[rr].y);
        }
        __syncthreads();
        // last axis: a lane's QC points of row rr, channel o
        for (int p = warp; p < R * d.C; p += kThr / 32) {
            const int rr = p / d.C, o = p - rr * d.C;
            float2 Z[QC];
#pragma unroll
            for (int c = 0; c < QC; c++) Z[c] = make_float2(0.f, 0.f);
#pragma unroll
            for (int m = 0; m < MM; m++) {
                if (m < d.M1) {
                    const float2 u = U[p * d.M1 + m], e = tj[m * 32 + lane];  // conjugated
                    Z[m % QC].x += u.x * e.x + u.y * e.y;
                    Z[m % QC].y += u.y * e.x - u.x * e.y;
                }
            }
            float v[QC];
            irdft<QC>(Z, v);
#pragma unroll
            for (int q = 0; q < QC; q++) y[o * kPitch + (rr * QC + q) * 32 + lane] = v[q];
        }
    }
    __syncthreads();
    // pointwise
    double lacc = 0.0;
    float qacc[CT + 1];   // T_LOSS: sums of dout v_L, dout
    float pacc[3][MODE == T_BACK0 ? CT : 1];
    if constexpr (MODE == T_LOSS)
        for (int c = 0; c <= CT; c++) qacc[c] = 0.f;
    if constexpr (MODE == T_BACK0)
        for (int c = 0; c < CT; c++) pacc[0][c] = pacc[1][c] = pacc[2][c] = 0.f;
    // PT points of a thread go together where few registers are live (in the
    // other modes two were slower: layer 150 -> 190 us for 8 states of 512^2)
    constexpr int PT = MODE == T_LIFT || MODE == T_BACK0 ? 2 : 1;
#pragma unroll 1
    for (int s0 = tid; s0 < kTile; s0 += kThr * PT) {
        bool in[PT];
        size_t pp[PT];
#pragma unroll
        for (int t = 0; t < PT; t++) {
            const int s = s0 + kThr * t, x0 = x00 + s / (QC * 32), q = (s >> 5) % QC, x1 = j + d.J * q;
            in[t] = x0 < d.n0 && j < d.J;
            pp[t] = in[t] ? (size_t)x0 * d.n1 + x1 : 0;
        }
        if constexpr (MODE == T_LIFT) {
            float a0[PT], a1[PT];
#pragma unroll
            for (int t = 0; t < PT; t++) {
                const size_t ip = (size_t)b * d.np + pp[t];
                const double u = in[t] ? a.un[ip] : 0.0, um = in[t] ? a.unm1[ip] : 0.0;
                a0[t] = pagd::to_f32(u);
                a1[t] = pagd::to_f32(a.s_in * (u - um));
            }
            for (int c = 0; c < d.C; c++) {
                const float p0 = a.prm[2 * c], p1 = a.prm[2 * c + 1], p2 = a.prm[2 * d.C + c];
#pragma unroll
                for (int t = 0; t < PT; t++) {
                    const float v = in[t] ? p0 * a0[t] + p1 * a1[t] + p2 : 0.f;
                    if (in[t]) a.vout[(bc + c) * d.np + pp[t]] = v;
                    y[c * kPitch + s0 + kThr * t] = v;
                }
            }
        } else {
            float vin[PT][CT];
#pragma unroll
            for (int t = 0; t < PT; t++)
#pragma unroll
                for (int c = 0; c < CT; c++) vin[t][c] = (c < d.C && in[t]) ? a.vin[(bc + c) * d.np + pp[t]] : 0.f;
            // (z_{l-1} with the other loads, not one by one in the loop below)
            float zp[PT][MODE == T_BACK ? CT : 1];
            if constexpr (MODE == T_BACK) {
#pragma unroll
                for (int t = 0; t < PT; t++)
#pragma unroll
                    for (int c = 0; c < CT; c++)
                        zp[t][c] = (c < d.C && in[t]) ? a.zprev[(bc + c) * d.np + pp[t]] : 0.f;
            }
            float out[PT];
            float sg[MODE == T_LOSS ? CT : 1], zz[MODE == T_LOSS ? CT : 1];
#pragma unroll
            for (int t = 0; t < PT; t++) out[t] = 0.f;
#pragma unroll
            for (int o = 0; o < CT; o++) {
                if (o < d.C) {
                    float f[PT];
#pragma unroll
                    for (int t = 0; t < PT; t++) f[t] = sw[CT * CT + o] + y[o * kPitch + s0 + kThr * t];
#pragma unroll
                    for (int c = 0; c < CT; c += 4) {
                        const float4 w = *(const float4*)&sw[o * CT + c];
#pragma unroll
                        for (int t = 0; t < PT; t++)
                            f[t] = fmaf(w.x, vin[t][c],
                                        fmaf(w.y, vin[t][c + 1], fmaf(w.z, vin[t][c + 2], fmaf(w.w, vin[t][c + 3], f[t]))));
                    }
#pragma unroll
                    for (int t = 0; t < PT; t++) {
                        const size_t i = (bc + o) * d.np + pp[t];
                        float* ys = &y[o * kPitch + s0 + kThr * t];
                        if constexpr (MODE == T_LAYER) {
                            const float v = gelu_f(f[t]);
                            if (in[t]) {
                                if (a.z) a.z[i] = f[t];
                                a.vout[i] = v;
                            }
                            *ys = in[t] ? v : 0.f;
                        } else if constexpr (MODE == T_GUESS) {
                            out[t] = fmaf(a.Q[o], gelu_f(f[t]), out[t]);
                        } else if constexpr (MODE == T_LOSS) {
                            sg[o] = gelu_s(f[t]);
                            zz[o] = f[t];
                            out[t] = fmaf(a.Q[o], f[t] * sg[o], out[t]);
                        } else if constexpr (MODE == T_BACK) {
                            const float z = zp[t][o];
                            const float g = f[t] * gelu_grad(z, gelu_s(z));
                            if (in[t]) a.vout[i] = g;
                            *ys = in[t] ? g : 0.f;
                        } else {
                            *ys = in[t] ? f[t] : 0.f;  // dv_0
                        }
                    }
                }
            }
            if constexpr (MODE == T_GUESS || MODE == T_LOSS) {
#pragma unroll
                for (int t = 0; t < PT; t++) {
                    const float o = out[t] + a.Q[d.C];
                    const size_t ip = (size_t)b * d.np + pp[t];
                    const double u = in[t] ? a.un[ip] : 0.0, um = in[t] ? a.unm1[ip] : 0.0, ext = fma(a.rho, u - um, u);
                    if constexpr (MODE == T_GUESS) {
                        if (in[t]) a.guess[ip] = fma(a.s_out, pagd::to_f64(o), ext);
                    } else {
                        const double e = in[t] ? pagd::to_f64(o) - (a.target[ip] - ext) * a.inv_s_out : 0.0;
                        lacc = fma(e, e, lacc);
                        const float g = pagd::to_f32(a.dscale * e);
#pragma unroll
                        for (int c = 0; c < CT; c++) {
                            if (c < d.C) {
                                qacc[c] = fmaf(g, zz[c] * sg[c], qacc[c]);
                                const float dz = a.Q[c] * g * gelu_grad(zz[c], sg[c]);
                                if (in[t]) a.vout[(bc + c) * d.np + pp[t]] = dz;
                                y[c * kPitch + s0 + kThr * t] = in[t] ? dz : 0.f;
                            }
                        }
                        qacc[CT] += g;
                    }
                }
            }
            if constexpr (MODE == T_BACK0) {
#pragma unroll
                for (int t = 0; t < PT; t++) {
                    const size_t ip = (size_t)b * d.np + pp[t];
                    const double u = in[t] ? a.un[ip] : 0.0, um = in[t] ? a.unm1[ip] : 0.0;
                    const float a0 = pagd::to_f32(u), a1 = pagd::to_f32(a.s_in * (u - um));
#pragma unroll
                    for (int c = 0; c < CT; c++) {
                        if (c < d.C) {
                            const float g = y[c * kPitch + s0 + kThr * t];
                            pacc[0][c] = fmaf(g, a0, pacc[0][c]);
                            pacc[1][c] = fmaf(g, a1, pacc[1][c]);
                            pacc[2][c] += g;
                        }
                    }
                }
            }
        }
    }
    float* red = (float*)U;  // the spectral part's buffers are free
    if constexpr (MODE == T_LOSS) {
        // block sums of the per-thread accumulators -> one row of part, two words
        // each: they nearly cancel over the grid (error of dQ, db_Q over 93 drawn
        // networks 2.7e-7 with one word, 3.0e-8 with two; gradient of 4 states of
        // 512^2 1317 -> 1353 us)
        constexpr int NV = CT + 1, V = CT <= 16 ? 32 : 64, PL = V / 32;
        float v[V], e[V];
#pragma unroll
        for (int c = 0; c < V; c++) {
            v[c] = c < NV ? qacc[c] : 0.f;
            e[c] = 0.f;
        }
        reduce_deal2<V>(v, e, lane);
#pragma unroll
        for (int q = 0; q < PL; q++) {
            const int c = lane * PL + q;
            if (c < NV) {
                red[(warp * NV + c) * 2] = v[q];
                red[(warp * NV + c) * 2 + 1] = e[q];
            }
        }
        for (int o = 16; o > 0; o >>= 1) lacc += __shfl_xor_sync(0xffffffffu, lacc, o);
        if (lane == 0) atomicAdd(a.loss, lacc * (0.5 * a.dscale));
        __syncthreads();
        const int nv = d.C + 1;
        for (int i = tid; i < nv; i += kThr) {
            const int c = i == d.C ? CT : i;
            pagd::Sum3 t;
            for (int w = 0; w < kThr / 32; w++) {
                t.add(red[(w * NV + c) * 2]);
                t.add(red[(w * NV + c) * 2 + 1]);
            }
            float* row = a.part + (((size_t)b * gridDim.x + blockIdx.x) * nv + i) * 2;
            row[0] = t.h;
            row[1] = t.m;
        }
    }
    if constexpr (MODE == T_BACK0) {
        constexpr int NV = 3 * CT;
        const int nv = 3 * d.C;
#pragma unroll
        for (int c = 0; c < NV; c++) {
            float v = pacc[c % 3][c / 3];
            for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
            if (lane == 0) red[warp * NV + c] = v;
        }
        __syncthreads();
        for (int i = tid; i < nv; i += kThr) {
            float v = 0.f;
            for (int w = 0; w < kThr / 32; w++) v += red[w * NV + i];
            a.part[((size_t)b * gridDim.x + blockIdx.x) * nv + i] = v;
        }
    }
    if constexpr (MODE == T_LIFT || MODE == T_LAYER || MODE == T_LOSS || MODE == T_BACK) {
        __syncthreads();
        // last-axis transform of the tile's rows
        for (int pq = warp; pq < R * d.C; pq += kThr / 32) {
            const int rr = pq / d.C, o = pq - rr * d.C, x0 = x00 + rr;
            float v[QC];
            float2 Y[QC / 2 + 1];
#pragma unroll
            for (int q = 0; q < QC; q++) v[q] = y[o * kPitch + (rr * QC + q) * 32 + lane];
            rdft<QC>(v, Y);
            float acc[2 * MM];
#pragma unroll
            for (int m = 0; m < MM; m++) {
                constexpr int h = QC / 2;
                const int c = m % QC;
                float2 w = c <= h ? Y[c] : make_float2(Y[QC - c].x, -Y[QC - c].y);
                const float2 e = m < d.M1 ? tj[m * 32 + lane] : make_float2(0.f, 0.f);
                acc[2 * m] = w.x * e.x - w.y * e.y;
                acc[2 * m + 1] = w.x * e.y + w.y * e.x;
            }
            reduce_deal<2 * MM>(acc, lane);
            if (x0 < d.n0) {
                float* t = (float*)(a.T + ((bc + o) * (size_t)(d.n0 * d.JB) + (size_t)x0 * d.JB + jb) * d.M1);
                if constexpr (MM == 32) {
                    if (lane < d.M1) *(float2*)&t[2 * lane] = make_float2(acc[0], acc[1]);
                } else {
                    if (lane < 2 * d.M1) t[lane] = acc[0];
                }
            }
        }
    }
}

static size_t tile_smem(const SnoDims& d, int CT) {
    const size_t red = (size_t)(kThr / 32) * 3 * CT * sizeof(float);
    size_t spec = sizeof(float2) * ((size_t)d.R * d.C * d.M1 + (size_t)d.R * d.M0);
    if (spec < red) spec = red;
    return sizeof(float) * ((size_t)d.C * kPitch + CT * CT + CT) + sizeof(float2) * (size_t)d.M1 * 32 + spec;
}

// First axis: F[g][m0][m1] = sum over the rows r of T[g][r][m1] exp(-2 pi i k0 x0(r) / n0), one
// block per channel g, a thread per mode and share of the rows; the rows go
// through shared memory, kColRows at a time, loaded together
constexpr int kColThr = 1024, kColRows = 512;
__global__ void __launch_bounds__(kColThr) k_cols(SnoDims d, const float2* T, const float2* tw0, float2* F) {
    extern __shared__ __align__(16) float2 cs[];  // n0 twiddles, the rows, the shares' sums
    float2* rw = cs + d.n0;
    float2* part = rw + kColRows * d.M1;
    for (int i = threadIdx.x; i < d.n0; i += kColThr) cs[i] = tw0[i];
    int mp = 32;
    while (mp < d.M) mp <<= 1;
    const int g = blockIdx.x, m = threadIdx.x & (mp - 1), q = threadIdx.x / mp, nq = kColThr / mp, nr = d.n0 * d.JB;
    const int m0 = m / d.M1, m1 = m - m0 * d.M1, k0 = k0_of(m0, d.M0, d.n0);
    float2 s = make_float2(0.f, 0.f);
    for (int c0 = 0; c0 < nr; c0 += kColRows) {
        const int cr = nr - c0 < kColRows ? nr - c0 : kColRows;
        const float2* t = T + ((size_t)g * nr + c0) * d.M1;
        __syncthreads();
#pragma unroll 4
        for (int i = threadIdx.x; i < cr * d.M1; i += kColThr) rw[i] = t[i];
        __syncthreads();
        if (m < d.M) {
#pragma unroll 4
            for (int r = q; r < cr; r += nq) {
                const float2 v = rw[r * d.M1 + m1], e = cs[(k0 * ((c0 + r) >> d.ljb)) & (d.n0 - 1)];
                s.x += v.x * e.x - v.y * e.y;
                s.y += v.x * e.y + v.y * e.x;
            }
        }
    }
    if (m < d.M) part[q * mp + m] = s;
    __syncthreads();
    for (int i = threadIdx.x; i < d.M; i += kColThr) {
        float2 f = part[i];
        for (int k = 1; k < nq; k++) {
            f.x += part[k * mp + i].x;
            f.y += part[k * mp + i].y;
        }
        F[(size_t)g * d.M + i] = f;
    }
}

// ---------------------------------------------------------------- mixing
// G[b][o][m] = sum_c R[o][c][m] F[b][c][m]
__global__ void k_mix(SnoDims d, const float* R, const float2* F, float2* G) {
    const int b = blockIdx.y;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;  // o * M + m
    if (i >= d.C * d.M) return;
    const int o = i / d.M, m = i % d.M;
    float2 s = make_float2(0.f, 0.f);
#pragma unroll 4
    for (int c = 0; c < d.C; c++) {
        const float* rp = R + (((size_t)o * d.C + c) * d.M + m) * 2;  // may start at an odd float
        const float2 r = make_float2(rp[0], rp[1]);
        const float2 f = F[((size_t)b * d.C + c) * d.M + m];
        s.x += r.x * f.x - r.y * f.y;
        s.y += r.x * f.y + r.y * f.x;
    }
    G[((size_t)b * d.C + o) * d.M + m] = s;
}

// spectral part of the backward pass: dG[b][o][m] = (w_m / np) DFT(dz)[b][o][m];
// dR[o][c][m] = sum_b dG conj(F), dF[b][c][m] = sum_o conj(R) dG.  One block per
// channel c and 32 modes, the o split over its warps.
__global__ void __launch_bounds__(kThr) k_mix_back(SnoDims d, const float* R, const float2* F, const float2* dZ, float* dR,
                                                   float2* dF, int B) {
    __shared__ float2 red[kThr / 32][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, c = blockIdx.y, m = blockIdx.x * 32 + lane;
    const bool in = m < d.M;
    const int mm = in ? m : 0;
    const float wm = (mm % d.M1 == 0 ? 1.f : 2.f) / (float)d.np;
    float2 acc[4], r[4];
#pragma unroll
    for (int k = 0; k < 4; k++) {
        const int o = w + 8 * k;
        acc[k] = r[k] = make_float2(0.f, 0.f);
        if (o < d.C) {
            const float* rp = R + (((size_t)o * d.C + c) * d.M + mm) * 2;  // may start at an odd float
            r[k] = make_float2(rp[0], rp[1]);
        }
    }
    for (int b = 0; b < B; b++) {
        const float2 f = F[((size_t)b * d.C + c) * d.M + mm];
        float2 s = make_float2(0.f, 0.f);
#pragma unroll
        for (int k = 0; k < 4; k++) {
            const int o = w + 8 * k;
            if (o < d.C) {
                float2 g = dZ[((size_t)b * d.C + o) * d.M + mm];
                g.x *= wm;
                g.y *= wm;
                acc[k].x += g.x * f.x + g.y * f.y;  // dG conj(F)
                acc[k].y += g.y * f.x - g.x * f.y;
                s.x += r[k].x * g.x + r[k].y * g.y;  // conj(R) dG
                s.y += r[k].x * g.y - r[k].y * g.x;
            }
        }
        __syncthreads();
        red[w][lane] = s;
        __syncthreads();
        if (w == 0 && in) {
            for (int q = 1; q < kThr / 32; q++) {
                s.x += red[q][lane].x;
                s.y += red[q][lane].y;
            }
            dF[((size_t)b * d.C + c) * d.M + m] = s;
        }
    }
#pragma unroll
    for (int k = 0; k < 4; k++) {
        const int o = w + 8 * k;
        if (o < d.C && in) {
            float* dr = dR + (((size_t)o * d.C + c) * d.M + m) * 2;
            dr[0] = acc[k].x;
            dr[1] = acc[k].y;
        }
    }
}

// Partial sums over kTile consecutive points dW[o][c] = sum dz[o] v[c] and
// db[o] = sum dz[o] -> row of part.  Both channels sets are staged in shared
// memory; a warp takes kTile / 8 of the points, a lane a (CT / 4) x (CT / 8)
// block of the products, four points per shared load.
template <int CT>
__global__ void __launch_bounds__(kThr) k_wgrad(SnoDims d, const float* dz, const float* v, float* part) {
    extern __shared__ __align__(16) float sm[];
    float *sd = sm, *sv = sm + CT * kPitch;
    constexpr int NO = CT / 4, NC = CT / 8;  // lanes: 4 x 8
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5, b = blockIdx.y, p0 = blockIdx.x * kTile;
    for (int i = tid; i < CT * (kTile / 4); i += kThr) {
        const int ch = i / (kTile / 4), x = 4 * (i % (kTile / 4));
        float4 g = make_float4(0.f, 0.f, 0.f, 0.f), u = g;
        if (ch < d.C && p0 + x < d.np) {  // np is a multiple of 4
            g = *(const float4*)&dz[((size_t)b * d.C + ch) * d.np + p0 + x];
            u = *(const float4*)&v[((size_t)b * d.C + ch) * d.np + p0 + x];
        }
        *(float4*)&sd[ch * kPitch + x] = g;
        *(float4*)&sv[ch * kPitch + x] = u;
    }
    __syncthreads();
    const int o0 = lane >> 3, c0 = lane & 7;
    float acc[NO][NC], bs[NO];
#pragma unroll
    for (int i = 0; i < NO; i++) {
        bs[i] = 0.f;
#pragma unroll
        for (int k = 0; k < NC; k++) acc[i][k] = 0.f;
    }
#pragma unroll 2
    for (int x = w * (kTile / 8); x < (w + 1) * (kTile / 8); x += 4) {
        float4 g[NO], u[NC];
#pragma unroll
        for (int i = 0; i < NO; i++) g[i] = *(const float4*)&sd[(o0 + 4 * i) * kPitch + x];
#pragma unroll
        for (int k = 0; k < NC; k++) u[k] = *(const float4*)&sv[(c0 + 8 * k) * kPitch + x];
#pragma unroll
        for (int i = 0; i < NO; i++) {
            bs[i] += (g[i].x + g[i].y) + (g[i].z + g[i].w);
#pragma unroll
            for (int k = 0; k < NC; k++)
                acc[i][k] = fmaf(g[i].x, u[k].x, fmaf(g[i].y, u[k].y, fmaf(g[i].z, u[k].z, fmaf(g[i].w, u[k].w, acc[i][k]))));
        }
    }
    __syncthreads();
    float* red = sm;  // [8 warps][CT][CT + 1]
#pragma unroll
    for (int i = 0; i < NO; i++) {
        const int o = o0 + 4 * i;
#pragma unroll
        for (int k = 0; k < NC; k++) red[(w * CT + o) * (CT + 1) + c0 + 8 * k] = acc[i][k];
        if (c0 == 0) red[(w * CT + o) * (CT + 1) + CT] = bs[i];
    }
    __syncthreads();
    const int nrow = d.C * d.C + d.C;
    for (int i = tid; i < nrow; i += kThr) {
        const int o = i < d.C * d.C ? i / d.C : i - d.C * d.C, c = i < d.C * d.C ? i % d.C : CT;
        float s = 0.f;
        for (int q = 0; q < 8; q++) s += red[(q * CT + o) * (CT + 1) + c];
        part[((size_t)blockIdx.y * gridDim.x + blockIdx.x) * nrow + i] = s;
    }
}

// out[col(j)] = sum over rows of part[row][j], without loss (Sum3), of `words`
// words each; lift: the partials [C][3] = (dP0, dP1, db) go to the layout P [C][2], b_P [C]
constexpr int kSumThr = 1024;
__global__ void __launch_bounds__(kSumThr) k_sum_rows(const float* part, int rows, int cols, int words, float* out, int lift) {
    __shared__ float red[3][kSumThr / 32][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, j = blockIdx.x * 32 + lane;
    pagd::Sum3 s;
    if (j < cols)
        for (int r = w; r < rows; r += kSumThr / 32) {
            const float* p = part + ((size_t)r * cols + j) * words;
            s.add(p[0]);
            if (words > 1) s.add(p[1]);
        }
    red[0][w][lane] = s.h;
    red[1][w][lane] = s.m;
    red[2][w][lane] = s.l;
    __syncthreads();
    if (w == 0 && j < cols) {
        for (int q = 1; q < kSumThr / 32; q++) s.add(pagd::Sum3{red[0][q][lane], red[1][q][lane], red[2][q][lane]});
        const int o = !lift ? j : (j % 3 < 2 ? 2 * (j / 3) + j % 3 : 2 * lift + j / 3);
        out[o] = pagd::to_f32(s.value());
    }
}

// Adam (Kingma and Ba, 2015) with bias correction
// the weights as BF16 numbers (round to nearest even), kept in FP32 storage:
// the network computes with them and accumulates in FP32, Adam updates the
// FP32 master copy they are rounded from
__global__ void k_round_bf16(const float* src, float* dst, long long n) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) dst[i] = __bfloat162float(__float2bfloat16_rn(src[i]));
}

__global__ void k_adam(float* p, const float* g, float* m, float* v, long long n, float lr, float b1, float b2,
                       float eps, float c1, float c2) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

}  // namespace

struct sno_net {
    SnoDims d;
    int batch;
    void* stream;
    char* ws;
    size_t ws_bytes;
    size_t off_v, off_z, off_F, off_G, off_T, off_dz, off_dz2, off_part, off_dF, off_loss, off_tw0, off_tw1;
    std::string err;
};

static size_t param_count(const SnoDims& d) {
    return (size_t)3 * d.C + (size_t)d.L * ((size_t)d.C * d.C + d.C + (size_t)2 * d.C * d.C * d.M) + d.C + 1;
}
static size_t off_layer(const SnoDims& d, int l) {
    return (size_t)3 * d.C + (size_t)l * ((size_t)d.C * d.C + d.C + (size_t)2 * d.C * d.C * d.M);
}
static size_t off_Q(const SnoDims& d) { return off_layer(d, d.L); }

static pagd_status sno_fail(sno_net* s, pagd_status st, const char* m) {
    if (s) s->err = m;
    return st;
}

static void plan(sno_net* s) {
    const SnoDims& d = s->d;
    const size_t B = (size_t)s->batch, np = (size_t)d.np;
    size_t o = 0;
    auto take = [&](size_t bytes) {
        const size_t at = o;
        o += (bytes + 255) & ~(size_t)255;
        return at;
    };
    s->off_v = take(sizeof(float) * B * d.C * np * d.L);
    s->off_z = take(sizeof(float) * B * d.C * np * (d.L > 1 ? d.L - 1 : 0));
    s->off_F = take(sizeof(float2) * B * d.C * d.M * d.L);
    s->off_G = take(sizeof(float2) * B * d.C * d.M);
    s->off_T = take(sizeof(float2) * B * d.C * d.n0 * d.JB * d.M1);
    s->off_dz = take(sizeof(float) * B * d.C * np);
    s->off_dz2 = take(sizeof(float) * B * d.C * np);
    const size_t rows = B * std::max<size_t>((size_t)d.NT, (np + kTile - 1) / kTile);
    s->off_part = take(sizeof(float) * rows * std::max<size_t>({(size_t)d.C * d.C + d.C, (size_t)3 * d.C, (size_t)2 * (d.C + 1)}));
    s->off_dF = take(sizeof(float2) * B * d.C * d.M);
    s->off_loss = take(sizeof(double));
    s->off_tw0 = take(sizeof(float2) * d.n0);
    s->off_tw1 = take(sizeof(float2) * d.n1);
    s->ws_bytes = o;
}

#define CK(x)                                                                       \
    do {                                                                            \
        cudaError_t e_ = (x);                                                       \
        if (e_ != cudaSuccess) return sno_fail(s, PAGD_ECUDA, cudaGetErrorString(e_)); \
    } while (0)

// A kernel may take all of an SM's shared memory, whatever this call needs: the
// attribute is the process's, and a call that lowered it to its own size would
// fail another thread's launch.
constexpr int kMaxSmem = 227 * 1024;
template <class K> static cudaError_t allow_smem(K* kern) {
    return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem);
}

template <int MODE, int QC, int CT, int MM>
static cudaError_t launch_tile(const SnoDims& d, const TileArgs& a, int B, cudaStream_t st) {
    const size_t smem = tile_smem(d, CT);
    if (smem > 48 * 1024) {
        const cudaError_t e = allow_smem(k_tile<MODE, QC, CT, MM>);
        if (e != cudaSuccess) return e;
    }
    k_tile<MODE, QC, CT, MM><<<dim3(d.NT, B), kThr, smem, st>>>(d, a);
    return cudaGetLastError();
}
template <int MODE, int QC> static cudaError_t tile_qc(const SnoDims& d, const TileArgs& a, int B, cudaStream_t st) {
    if (d.C <= 16) return d.M1 <= 16 ? launch_tile<MODE, QC, 16, 16>(d, a, B, st) : launch_tile<MODE, QC, 16, 32>(d, a, B, st);
    return d.M1 <= 16 ? launch_tile<MODE, QC, 32, 16>(d, a, B, st) : launch_tile<MODE, QC, 32, 32>(d, a, B, st);
}
template <int MODE> static cudaError_t tile(const SnoDims& d, const TileArgs& a, int B, cudaStream_t st) {
    if (d.QC == 16) return tile_qc<MODE, 16>(d, a, B, st);
    if (d.QC == 4) return tile_qc<MODE, 4>(d, a, B, st);
    return tile_qc<MODE, 1>(d, a, B, st);
}
template <int CT> static cudaError_t launch_wgrad(const SnoDims& d, const float* dz, const float* v, float* part, int B,
                                                  cudaStream_t st) {
    const size_t smem = std::max<size_t>((size_t)2 * CT * kPitch, (size_t)8 * CT * (CT + 1)) * sizeof(float);
    const cudaError_t e = allow_smem(k_wgrad<CT>);
    if (e != cudaSuccess) return e;
    k_wgrad<CT><<<dim3((d.np + kTile - 1) / kTile, B), kThr, smem, st>>>(d, dz, v, part);
    return cudaGetLastError();
}

static TileArgs tile_args(const sno_net* s, const float* prm, const double* un, const double* unm1, float s_in) {
    TileArgs a = {};
    a.prm = prm;
    a.un = un;
    a.unm1 = unm1;
    a.s_in = s_in;
    a.Q = prm + off_Q(s->d);
    a.G = (const float2*)(s->ws + s->off_G);
    a.T = (float2*)(s->ws + s->off_T);
    a.tw0 = (const float2*)(s->ws + s->off_tw0);
    a.tw1 = (const float2*)(s->ws + s->off_tw1);
    return a;
}
static void set_layer(TileArgs& a, const SnoDims& d, int l) {
    a.W = a.prm + off_layer(d, l);
    a.bias = a.W + d.C * d.C;
}

// T -> the modes F
static cudaError_t launch_cols(const sno_net* s, int G, const float2* T, float2* F) {
    const SnoDims& d = s->d;
    const size_t smem = sizeof(float2) * (d.n0 + (size_t)kColRows * d.M1 + kColThr);
    const cudaError_t e = allow_smem(k_cols);
    if (e != cudaSuccess) return e;
    k_cols<<<G, kColThr, smem, (cudaStream_t)s->stream>>>(d, T, (const float2*)(s->ws + s->off_tw0), F);
    return cudaGetLastError();
}

// The forward pass for B samples up to the modes of the last layer; v_l (and,
// with train, z_l) stay in the workspace.  The last layer's pass is the caller's.
static pagd_status forward(sno_net* s, TileArgs& a, int B, bool train) {
    const SnoDims& d = s->d;
    cudaStream_t st = (cudaStream_t)s->stream;
    char* w = s->ws;
    float* v = (float*)(w + s->off_v);
    float* z = (float*)(w + s->off_z);
    float2* F = (float2*)(w + s->off_F);
    float2* G = (float2*)(w + s->off_G);
    const size_t vs = (size_t)B * d.C * d.np;  // one layer of activations
    k_tables<<<(d.n0 + d.n1 + kThr - 1) / kThr, kThr, 0, st>>>((float2*)(w + s->off_tw0), d.n0,
                                                                (float2*)(w + s->off_tw1), d.n1);
    CK(cudaGetLastError());
    a.vout = v;
    CK(tile<T_LIFT>(d, a, B, st));
    for (int l = 0; l < d.L; l++) {
        float2* Fl = F + (size_t)l * B * d.C * d.M;
        set_layer(a, d, l);
        CK(launch_cols(s, B * d.C, a.T, Fl));
        k_mix<<<dim3((d.C * d.M + kThr - 1) / kThr, B), kThr, 0, st>>>(d, a.bias + d.C, Fl, G);
        a.vin = v + l * vs;
        if (l + 1 < d.L) {
            a.vout = v + (l + 1) * vs;
            a.z = train ? z + l * vs : nullptr;
            CK(tile<T_LAYER>(d, a, B, st));
        }
    }
    CK(cudaGetLastError());
    return PAGD_OK;
}

extern "C" {

pagd_status sno_create(sno_net** out, int n0, int n1, int channels, int layers, int modes0, int modes1, int batch,
                       void* stream) {
    if (!out) return PAGD_EINVAL;
    *out = nullptr;
    auto pow2 = [](int v) { return v >= 8 && v <= 4096 && (v & (v - 1)) == 0; };
    if (!pow2(n0) || !pow2(n1) || channels < 1 || channels > 32 || layers < 1 || layers > 16 || modes0 < 2 ||
        (modes0 & 1) || modes0 > n0 || modes1 < 1 || modes1 > 32 || modes1 > n1 / 2 || modes0 * modes1 > 1024 ||
        batch < 1)
        return PAGD_EINVAL;
    sno_net* s = new (std::nothrow) sno_net();
    if (!s) return PAGD_ENOMEM;
    SnoDims& d = s->d;
    d = SnoDims{n0, n1, n0 * n1, channels, layers, modes0, modes1, modes0 * modes1, 0, 0, 0, 0, 0, 0};
    // QC points of a row per lane: more points share the twiddle sums of their
    // residue, but fewer than 32 residues leave lanes idle.  Inference / gradient in
    // us, 16 channels, 4 layers, 16 x 16 modes, QC = 1, 4, 16: 64 samples of 32^2
    // 263 / 706, 300 / 807, 451 / 1191; 64 of 64^2 554 / 1395, 417 / 1147, 757 /
    // 1971; 8 of 256^2 904 / 2050, 400 / 1007, 431 / 1121; 4 of 512^2 2164 / 4678,
    // 814 / 1972, 476 / 1322.
    d.QC = n1 >= 512 ? 16 : n1 >= 64 ? 4 : 1;
    d.J = n1 / d.QC;
    d.JB = d.J > 32 ? d.J / 32 : 1;
    while ((1 << d.ljb) < d.JB) d.ljb++;
    d.R = 16 / d.QC;
    d.NT = (n0 + d.R - 1) / d.R * d.JB;
    s->batch = batch;
    s->stream = stream;
    s->ws = nullptr;
    plan(s);
    *out = s;
    return PAGD_OK;
}

pagd_status sno_param_count(const sno_net* s, size_t* n) {
    if (!s || !n) return PAGD_EINVAL;
    *n = param_count(s->d);
    return PAGD_OK;
}

pagd_status sno_workspace_size(const sno_net* s, size_t* bytes) {
    if (!s || !bytes) return PAGD_EINVAL;
    *bytes = s->ws_bytes;
    return PAGD_OK;
}

pagd_status sno_set_workspace(sno_net* s, void* dev, size_t bytes) {
    if (!s || !dev) return PAGD_EINVAL;
    if (((uintptr_t)dev & 255) != 0) return sno_fail(s, PAGD_EINVAL, "workspace not 256-byte aligned");
    if (bytes < s->ws_bytes) return sno_fail(s, PAGD_ENOMEM, "workspace too small");
    s->ws = (char*)dev;
    return PAGD_OK;
}

pagd_status sno_predict(sno_net* s, const float* params, const double* un, const double* unm1, double rho,
                        double s_in, double s_out, int nsamples, double* guess) {
    if (!s || !params || !un || !unm1 || !guess) return PAGD_EINVAL;
    if (!s->ws) return sno_fail(s, PAGD_ESTATE, "no workspace");
    if (nsamples < 1 || nsamples > s->batch) return sno_fail(s, PAGD_EINVAL, "bad sample count");
    TileArgs a = tile_args(s, params, un, unm1, (float)s_in);
    a.rho = rho;
    a.s_out = s_out;
    a.guess = guess;
    const pagd_status r = forward(s, a, nsamples, false);
    if (r != PAGD_OK) return r;
    CK(tile<T_GUESS>(s->d, a, nsamples, (cudaStream_t)s->stream));
    CK(cudaStreamSynchronize((cudaStream_t)s->stream));
    return PAGD_OK;
}

pagd_status sno_loss_grad(sno_net* s, const float* params, const double* un, const double* unm1,
                          const double* target, double rho, double s_in, double s_out, int nsamples, float* grad,
                          double* loss) {
    if (!s || !params || !un || !unm1 || !target || !grad) return PAGD_EINVAL;
    if (!s->ws) return sno_fail(s, PAGD_ESTATE, "no workspace");
    if (nsamples < 1 || nsamples > s->batch) return sno_fail(s, PAGD_EINVAL, "bad sample count");
    const SnoDims& d = s->d;
    const int B = nsamples;
    cudaStream_t st = (cudaStream_t)s->stream;
    char* w = s->ws;
    float* v = (float*)(w + s->off_v);
    float* z = (float*)(w + s->off_z);
    float2* F = (float2*)(w + s->off_F);
    float2* dZ = (float2*)(w + s->off_G);
    float2* dF = (float2*)(w + s->off_dF);
    float* dz = (float*)(w + s->off_dz);
    float* dz2 = (float*)(w + s->off_dz2);
    float* part = (float*)(w + s->off_part);
    double* dloss = (double*)(w + s->off_loss);
    const size_t vs = (size_t)B * d.C * d.np;
    const int nrow = d.C * d.C + d.C, tiles = d.NT * B, wrows = (d.np + kTile - 1) / kTile * B;
    CK(cudaMemsetAsync(dloss, 0, sizeof(double), st));
    TileArgs a = tile_args(s, params, un, unm1, (float)s_in);
    a.target = target;
    a.rho = rho;
    a.inv_s_out = 1.0 / s_out;
    a.dscale = 2.0 / ((double)d.np * B);
    a.loss = dloss;
    a.part = part;
    const pagd_status r = forward(s, a, B, true);
    if (r != PAGD_OK) return r;
    // last layer, projection, loss, and the way back to dz of the last layer
    a.vout = dz;
    CK(tile<T_LOSS>(d, a, B, st));
    auto sum_rows = [&](int rows, int cols, int words, float* out, int lift) {
        k_sum_rows<<<(cols + 31) / 32, kSumThr, 0, st>>>(part, rows, cols, words, out, lift);
    };
    sum_rows(tiles, d.C + 1, 2, grad + off_Q(d), 0);
    a.G = dF;
    for (int l = d.L - 1; l >= 0; l--) {
        float* gL = grad + off_layer(d, l);
        set_layer(a, d, l);
        CK(launch_cols(s, B * d.C, a.T, dZ));
        k_mix_back<<<dim3((d.M + 31) / 32, d.C), kThr, 0, st>>>(d, a.bias + d.C, F + (size_t)l * B * d.C * d.M, dZ,
                                                              gL + nrow, dF, B);
        if (d.C <= 16) CK(launch_wgrad<16>(d, dz, v + (size_t)l * vs, part, B, st));
        else CK(launch_wgrad<32>(d, dz, v + (size_t)l * vs, part, B, st));
        sum_rows(wrows, nrow, 1, gL, 0);
        a.vin = dz;
        a.vout = dz2;
        if (l > 0) {
            a.zprev = z + (size_t)(l - 1) * vs;
            CK(tile<T_BACK>(d, a, B, st));
        } else {
            CK(tile<T_BACK0>(d, a, B, st));
        }
        std::swap(dz, dz2);
    }
    sum_rows(tiles, 3 * d.C, 1, grad, d.C);
    CK(cudaGetLastError());
    if (loss) CK(cudaMemcpyAsync(loss, dloss, sizeof(double), cudaMemcpyDeviceToHost, st));
    CK(cudaStreamSynchronize(st));
    return PAGD_OK;
}

pagd_status sno_adam_step(sno_net* s, float* params, const float* grad, float* m, float* v, int t, double lr) {
    if (!s || !params || !grad || !m || !v || t < 1 || !(lr > 0.0)) return PAGD_EINVAL;
    const long long n = (long long)param_count(s->d);
    const float b1 = 0.9f, b2 = 0.999f;
    const float c1 = 1.f - powf(b1, (float)t), c2 = 1.f - powf(b2, (float)t);
    k_adam<<<(unsigned)((n + kThr - 1) / kThr), kThr, 0, (cudaStream_t)s->stream>>>(params, grad, m, v, n, (float)lr,
                                                                                   b1, b2, 1e-8f, c1, c2);
    CK(cudaGetLastError());
    return PAGD_OK;
}

pagd_status sno_round_bf16(sno_net* s, const float* master, float* weights) {
    if (!s || !master || !weights) return PAGD_EINVAL;
    const long long n = (long long)param_count(s->d);
    k_round_bf16<<<(unsigned)((n + kThr - 1) / kThr), kThr, 0, (cudaStream_t)s->stream>>>(master, weights, n);
    CK(cudaGetLastError());
    return PAGD_OK;
}

const char* sno_last_error(const sno_net* s) { return s ? s->err.c_str() : "null network"; }

void sno_destroy(sno_net* s) { delete s; }

}  // extern "C"
