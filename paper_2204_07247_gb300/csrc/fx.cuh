// fx.cuh -- FP64 line transforms in 64-bit block fixed point.
//
// GB300 issues an FP64 instruction (FMA, add or conversion alike) at 1/64 of
// the FP32 rate: measured 64 cycles per warp instruction on one SM
// sub-partition whatever the active lanes, 19 cycles per SM with all four busy.
// A 64-bit integer add costs 0.4 cycles per SM and warp, the fixed-point
// product below 6.5.  A transform is mostly additions, so the lines of every
// FP64 pass are transformed as 64-bit integers with one exponent per line: a
// 256-point line takes about 390 SM cycles of arithmetic against 3700 in FP64.
//
// The values enter and leave as doubles.  A line is converted at the scale of
// its largest element (no bit of any value above 2^-8 of it is lost), the sum of the
// moduli of its points then fixes how far it has to be shifted so that no
// partial sum of the transform can overflow, and the result is rounded once
// to double.  The error against a transform in extended precision is no
// larger than that of the FP64 one it replaces (tests/test_fx_host.py
// measures both): about a third of it for lines of up to 256 points and for
// any line whose energy sits in few points, the same for 512 points of noise.
// Every partial sum of a radix stage is bounded by the sum of the moduli, so
// the bound holds for any input; a line with a NaN or an infinity comes out NaN.
//
// Layout: 16-byte slots, point i of a line at slot i ^ ((i >> 3) & 7), which
// spreads the strided stores of the first stages over all bank groups.
#pragma once
#include "compat.cuh"

namespace pagd {

template <> struct V2<long long> { using type = longlong2; };

// twiddle tables hold cos and sin in units of 2^-61 (FxTw)
constexpr int kFxTw = 61;
constexpr int kFxNaN = 1 << 28;  // exponent of a line that holds a NaN or an infinity

__host__ __device__ __forceinline__ int fxs(int i) { return i ^ ((i >> 3) & 7); }

// A factor w, |w| <= sqrt(2) in units of 2^-61, as h 2^31 + l with 0 <= l < 2^31
struct FxW {
    int h, l;
};
__host__ __device__ constexpr FxW fx_split(long long w) { return FxW{(int)(w >> 31), (int)(w & 0x7fffffff)}; }
// A twiddle c + i s: the factors c, c + s, s - c of fx_cmul, split when the
// table is made (six integer instructions less per complex product)
struct alignas(8) FxTw {
    FxW c, p, q;
};
__host__ __device__ constexpr FxTw fx_tw(long long c, long long s) { return FxTw{fx_split(c), fx_split(c + s), fx_split(s - c)}; }

// a w 2^-61 rounded, |a| < 2^62: a split like w; the product of the low parts
// enters with its leading bits
__device__ __forceinline__ long long fx_mul(long long a, FxW w) {
    const int ah = (int)(a >> 31), al = (int)a & 0x7fffffff;
    long long m = (long long)ah * w.l + (1ll << 29);
    m += (long long)w.h * al;
    m += (al >> 16) * (w.l >> 15);
    return (((long long)ah * w.h) << 1) + (m >> 30);
}
// a w (S < 0) or a conj(w) (S > 0) in three real products
template <int S> __device__ __forceinline__ longlong2 fx_cmul(longlong2 a, const FxTw& w) {
    const long long k1 = fx_mul(a.x + a.y, w.c);
    if (S < 0) return longlong2{k1 - fx_mul(a.y, w.p), k1 + fx_mul(a.x, w.q)};
    return longlong2{k1 + fx_mul(a.y, w.q), k1 - fx_mul(a.x, w.p)};
}

template <int S> __device__ __forceinline__ void fx_dft8(longlong2* v) {
    constexpr FxW c = fx_split(1630477228166597777ll);  // cos(pi / 4) 2^61
    longlong2 e0 = v[0], e1 = v[2], e2 = v[4], e3 = v[6];
    longlong2 o0 = v[1], o1 = v[3], o2 = v[5], o3 = v[7];
    dft4<S>(e0, e1, e2, e3);
    dft4<S>(o0, o1, o2, o3);
    const longlong2 w1{fx_mul(S < 0 ? o1.x + o1.y : o1.x - o1.y, c), fx_mul(S < 0 ? o1.y - o1.x : o1.y + o1.x, c)};
    const longlong2 w2 = mul_si<S>(o2);
    const longlong2 w3{fx_mul(S < 0 ? o3.y - o3.x : -o3.x - o3.y, c), fx_mul(S < 0 ? -o3.x - o3.y : o3.x - o3.y, c)};
    v[0] = cadd(e0, o0);
    v[4] = csub(e0, o0);
    v[1] = cadd(e1, w1);
    v[5] = csub(e1, w1);
    v[2] = cadd(e2, w2);
    v[6] = csub(e2, w2);
    v[3] = cadd(e3, w3);
    v[7] = csub(e3, w3);
}
template <int R, int S> __device__ __forceinline__ void fx_dft(longlong2* v) {
    if constexpr (R == 2) dft2<S>(v);
    else if constexpr (R == 4) dft4<S>(v[0], v[1], v[2], v[3]);
    else fx_dft8<S>(v);
}

// ------------------------------------------------------------- conversions

__device__ __forceinline__ unsigned fx_hi(double x) { return (unsigned)(dbl_bits(x) >> 32) & 0x7fffffffu; }
// exponent field of a line from the largest fx_hi of its values
__device__ __forceinline__ int fx_emax(unsigned hi) { return (int)(hi >> 20); }

// x in units of 2^(emax - 1083): |result| < 2^61.  (Subnormal numbers count, in
// lines of values below 2^-960; the select for them is 1% of a transform.  A
// branch for such lines, per value or per line, cost 2 to 6%.)
__device__ __forceinline__ long long fx_from(double x, int emax) {
    const unsigned long long b = dbl_bits(x), f = b & 0xfffffffffffffull;
    const int e = (int)(b >> 52) & 0x7ff;
    const unsigned long long m = e == 0 ? f << 9 : (f | 0x10000000000000ull) << 8;
    int r = emax - e;
    if (r > 63) r = 63;  // below 2^-62 of the largest: zero
    const long long v = (long long)(m >> r);
    return (long long)b < 0 ? -v : v;
}
// upper bound of a point's modulus, in units of 2^41
__device__ __forceinline__ unsigned fx_mag(longlong2 z) {
    const int x = (int)(z.x >> 41), y = (int)(z.y >> 41);
    const unsigned ax = (unsigned)(x < 0 ? -x : x) + 1u, ay = (unsigned)(y < 0 ? -y : y) + 1u;
    const unsigned M = ax > ay ? ax : ay, m = ax > ay ? ay : ax;
    return M + ((m * 27u) >> 6) + 1u;
}
// right shift that brings a line whose moduli sum to less than s 2^41 below 2^61.5
__device__ __forceinline__ int fx_shift(unsigned s) {
    const int lz = clz32(s);
    const int k = 31 - lz + ((s << lz) > 0xb504f333u ? 1 : 0);
    return k > 20 ? k - 20 : 0;
}
__device__ __forceinline__ long long fx_shr(long long a, int sh, long long half) { return (a + half) >> sh; }
__device__ __forceinline__ long long fx_half(int sh) { return (1ll << sh) >> 1; }

// a 2^-S as a double (round half away), |a| < 2^63.  FAST: S in [kFxLo, kFxUp], where
// no value overflows or falls below 2^-1022 (else to an infinity, to a subnormal
// number or zero; NaN for a line marked kFxNaN).
constexpr int kFxLo = -900, kFxUp = 1000;
template <bool FAST> __device__ __forceinline__ double fx_to_t(long long a, int S) {
    const unsigned long long sgn = (unsigned long long)a & 0x8000000000000000ull;
    const unsigned long long u = a < 0 ? (unsigned long long)-a : (unsigned long long)a;
    const int lz = clz64(u);  // at least 1
    const unsigned long long n = u << ((lz - 1) & 63);
    const int E = 1085 - lz - S;
    unsigned long long t = ((n + 0x200ull) >> 10) + ((unsigned long long)(unsigned)E << 52);
    if (!FAST && E < 0) t = E < -53 ? 0ull : (n + (0x200ull << -E)) >> (10 - E);
    if (u == 0) t = 0;
    if (!FAST) {
        if (E >= 2046) t = 0x7ff0000000000000ull;
        if (S > kFxNaN / 2) t = 0x7ff8000000000000ull;
    }
    return bits_dbl(t | sgn);
}
__device__ __forceinline__ bool fx_fast(int S) { return S >= kFxLo && S <= kFxUp; }
__device__ __forceinline__ double fx_to(long long a, int S) { return fx_to_t<false>(a, S); }
// the exponent S of a converted line: 2^-S is its unit after the shift sh
__device__ __forceinline__ int fx_scale(int emax, int sh) { return emax == 0x7ff ? kFxNaN : 1083 - emax - sh; }

// FP64 <-> FP32 conversions with integer instructions: the hardware's issue
// at the FP64 rate (64 cycles per warp and sub-partition), these are about
// twelve instructions each.  The same values, rounded to nearest even; subnormal
// FP32 numbers go through a normal one 2^64 times as large, so that a result
// among them is rounded twice (within 0.5 + 2^-24 of its last place).  A branch to the
// hardware's conversion for them cost the FP32-mixed runs 5 to 9%.
__device__ __forceinline__ float to_f32(double x) {
    const unsigned long long b = dbl_bits(x), m = b & 0x7fffffffffffffffull;
    const unsigned hi = (unsigned)(m >> 32);
    const bool sub = hi < 0x38100000u;  // below 2^-126
    const unsigned long long t = m - ((unsigned long long)(sub ? 832u << 20 : 896u << 20) << 32);
    unsigned r = (unsigned)((t + 0x0fffffffull + ((t >> 29) & 1ull)) >> 29);
    if (hi < 0x34100000u) r = 0u;                                   // below 2^-190
    if (hi >= 0x47f00000u) r = m > 0x7ff0000000000000ull ? 0x7fc00000u : 0x7f800000u;  // 2^128 and above, inf, NaN
    if (sub) r = flt_bits(bits_flt(r) * 0x1p-64f);
    return bits_flt(r | ((unsigned)(b >> 32) & 0x80000000u));
}
__device__ __forceinline__ double to_f64(float x) {
    const unsigned b = flt_bits(x), m = b & 0x7fffffffu;
    const bool sub = m < 0x00800000u;
    const unsigned n = sub ? flt_bits(bits_flt(m) * 0x1p64f) : m;
    unsigned hi = (n >> 3) + (sub ? 832u << 20 : 896u << 20);
    const unsigned lo = n << 29;
    if (m == 0u) hi = 0u;
    if (m >= 0x7f800000u) hi += 896u << 20;  // inf, NaN
    hi |= b & 0x80000000u;
    return bits_dbl(((unsigned long long)hi << 32) | lo);
}
// 1 / x for a positive normal x in three FP64 instructions (the compiled
// division takes 364 cycles, six times one): an FP32 reciprocal of the
// significand, then one step of Newton's iteration for 1 / x with its next
// term, x0 (1 + e + e^2) with e = 1 - m x0 (|e| <= 2^-21, so e^3 is below the
// rounding), and the exponent by integer arithmetic: within 0.501 ulp, the
// division 0.5.  Other x (rcp_plain): the division.
__device__ __forceinline__ bool rcp_plain(double x) { return (unsigned)(dbl_bits(x) >> 32) - 0x00100000u >= 0x7fa00000u; }
__device__ __forceinline__ double rcp64(double x) {
    if (rcp_plain(x)) return 1.0 / x;
    const unsigned long long b = dbl_bits(x);
    const unsigned hi = (unsigned)(b >> 32), lo = (unsigned)b;
    const float m = bits_flt(0x3f800000u | ((hi & 0xfffffu) << 3) | (lo >> 29));
    const double x0 = to_f64(1.0f / m), md = bits_dbl((b & 0xfffffffffffffull) | 0x3ff0000000000000ull);
    const double e = fma(-md, x0, 1.0), y = fma(x0, fma(e, e, e), x0);
    return bits_dbl(dbl_bits(y) + ((unsigned long long)(1023u - (hi >> 20)) << 52));
}
__device__ __forceinline__ float rcp64(float x) { return 1.0f / x; }
// a / x and b / x: the product with the reciprocal, corrected by its remainder
// (Markstein 1990), within 0.501 ulp where the plain product has 1
__device__ __forceinline__ double2 div64(double2 n, double x) {
    if (rcp_plain(x)) return double2{n.x / x, n.y / x};
    const double r = rcp64(x);
    const double2 q{n.x * r, n.y * r};
    return double2{fma(fma(-x, q.x, n.x), r, q.x), fma(fma(-x, q.y, n.y), r, q.y)};
}
template <class T> __device__ __forceinline__ T cvt(double x) {
    if constexpr (sizeof(T) == 8) return x;
    else return to_f32(x);
}
__device__ __forceinline__ double wide(double x) { return x; }
__device__ __forceinline__ double wide(float x) { return to_f64(x); }

// Sum of FP32 values without FP64 instructions, to the last place of an FP64
// one and better: three words, the rounding error of each word's additions
// (Knuth's two-sum) going into the next (Ogita, Rump and Oishi 2005, SumK), so
// that 2^-70 of the sum of the magnitudes is left.  Thirteen FP32 additions a
// value; an FP64 addition with its conversion takes 128 cycles.  Two words (seven
// additions) left 2^-48, more than the 2^-53 per addition of an FP64 sum.
// A partial sum above 3.4e38 becomes an infinity, as in FP32.
struct Sum3 {
    float h = 0.f, m = 0.f, l = 0.f;
    // a + b -> a, returns the rounding error
    static __device__ __forceinline__ float two_sum(float& a, float b) {
        const float s = fadd(a, b), v = fadd(s, -a), e = fadd(fadd(a, -fadd(s, -v)), fadd(b, -v));
        a = s;
        return e;
    }
    __device__ __forceinline__ void add(float x) { l = fadd(l, two_sum(m, two_sum(h, x))); }
    __device__ __forceinline__ void add(const Sum3& o) {
        add(o.h);
        l = fadd(l, fadd(two_sum(m, o.m), o.l));
    }
    __device__ __forceinline__ double value() const {
        if ((flt_bits(h) & 0x7f800000u) == 0x7f800000u) return to_f64(h);  // (the errors are NaN)
        return to_f64(h) + (to_f64(m) + to_f64(l));
    }
    __device__ __forceinline__ double warp_total() const {
        Sum3 t = *this;
#pragma unroll
        for (int o = kWarp / 2; o > 0; o >>= 1) {
            Sum3 u;
            u.h = warp_xor(t.h, o);
            u.m = warp_xor(t.m, o);
            u.l = warp_xor(t.l, o);
            t.add(u);
        }
        return t.value();
    }
};

// ---------------------------------------------------------- warp-owned line

// radix of the stage that starts at LOGNS: as stage_radix, but 4 (and one 2) up
// to 128 points, where a warp has fewer butterflies of radix 8 than lanes.  128
// points go 2, 4, 4, 4: their first and last butterflies then cover all lanes.
// PFC FP64, two steps, radix 8 / 4: 64^3 1701 / 1452 us, 32 x 16 x 64 1094 / 1002,
// a batch of 32 members of 128^2 1964 / 1616, of 4 987 / 904.
__host__ __device__ constexpr int fx_radix(int logn, int logns) {
    if (logn == 7) return logns == 0 ? 2 : 4;
    return logn < 7 ? (logn - logns >= 2 ? 4 : 2) : stage_radix(logn, logns);
}

template <int R, int S, int LOGN, int LOGNS, bool FIRST>
__device__ __forceinline__ void fx_stage(longlong2* b, int sh, const FxTw* tw, int logTw, int lane) {
    constexpr int LR = (R == 2) ? 1 : (R == 4) ? 2 : 3;
    constexpr int NB = 1 << (LOGN - LR), NS = 1 << LOGNS;
    constexpr int PER = (NB + kWarp - 1) / kWarp;
    const int twshift = logTw - (LOGNS + LR);
    longlong2 v[PER * R];
    const long long half = fx_half(sh);
#pragma unroll
    for (int i = 0; i < PER; i++) {
        const int j = lane + kWarp * i;
        if (NB % kWarp == 0 || j < NB) {
            const int jm = j & (NS - 1);
            longlong2* u = v + i * R;
#pragma unroll
            for (int r = 0; r < R; r++) {
                u[r] = b[fxs(j + r * NB)];
                if (FIRST) u[r] = longlong2{fx_shr(u[r].x, sh, half), fx_shr(u[r].y, sh, half)};
                if (LOGNS > 0 && r > 0) u[r] = fx_cmul<S>(u[r], tw[(jm * r) << twshift]);
            }
            fx_dft<R, S>(u);
        }
    }
    warp_sync();
#pragma unroll
    for (int i = 0; i < PER; i++) {
        const int j = lane + kWarp * i;
        if (NB % kWarp == 0 || j < NB) {
            const int jm = j & (NS - 1), d = ((j - jm) << LR) + jm;
#pragma unroll
            for (int r = 0; r < R; r++) b[fxs(d + r * NS)] = v[i * R + r];
        }
    }
    warp_sync();
}
template <int S, int LOGN, int LOGNS>
__device__ __forceinline__ void fx_stages(longlong2* b, int sh, const FxTw* tw, int logTw, int lane) {
    if constexpr (LOGNS < LOGN) {
        constexpr int R = fx_radix(LOGN, LOGNS);
        fx_stage<R, S, LOGN, LOGNS, LOGNS == 0>(b, sh, tw, logTw, lane);
        fx_stages<S, LOGN, LOGNS + radix_log(R)>(b, sh, tw, logTw, lane);
    }
}

// One line of 1 << LOGN points (slot layout, converted, to be shifted by sh)
// transformed in place by one warp.  A function of its own: every pass of a
// kernel shares its code, and its registers do not add to theirs.  Data
// written before the call and read after it by any lane.
template <int S, int LOGN>
static __device__ __noinline__ void fx_line_n(longlong2* b, int sh, const FxTw* tw, int logTw, int lane) {
    warp_sync();
    fx_stages<S, LOGN, 0>(b, sh, tw, logTw, lane);
}
// NF: the line length, or 0 for the runtime length 1 << logn (8 .. 512)
template <int S, int NF>
__device__ __forceinline__ void fx_line(longlong2* b, int logn, int sh, const FxTw* tw, int logTw, int lane) {
    if constexpr (NF > 0) {
        fx_line_n<S, ilog2c(NF)>(b, sh, tw, logTw, lane);
    } else {
        switch (logn) {
            case 3: fx_line_n<S, 3>(b, sh, tw, logTw, lane); break;
            case 4: fx_line_n<S, 4>(b, sh, tw, logTw, lane); break;
            case 5: fx_line_n<S, 5>(b, sh, tw, logTw, lane); break;
            case 6: fx_line_n<S, 6>(b, sh, tw, logTw, lane); break;
            case 7: fx_line_n<S, 7>(b, sh, tw, logTw, lane); break;
            case 8: fx_line_n<S, 8>(b, sh, tw, logTw, lane); break;
            default: fx_line_n<S, 9>(b, sh, tw, logTw, lane); break;
        }
    }
}

// the doubles in one slot -> fixed point in place; returns the point's fx_mag
__device__ __forceinline__ unsigned fx_point(longlong2* slot, int emax) {
    const double2 z = *(const double2*)slot;
    const longlong2 f{fx_from(z.x, emax), fx_from(z.y, emax)};
    *slot = f;
    return fx_mag(f);
}
// Coefficient k < n / 2 of two rows' half spectra, A[k] in slot k and B[k] in
// slot n - k (k = 0: the real parts of A[0], B[0] in slot 0, of A[n / 2],
// B[n / 2] in slot n / 2), -> points k and n - k (n / 2) of the packed complex
// line A + i B in fixed point
__device__ __forceinline__ unsigned fx_pair_rows(longlong2* b, int k, int n, int emax) {
    const int k2 = k == 0 ? n >> 1 : n - k;
    const double2 a = *(const double2*)&b[fxs(k)], c = *(const double2*)&b[fxs(k2)];
    longlong2 A{fx_from(a.x, emax), fx_from(a.y, emax)}, B{fx_from(c.x, emax), fx_from(c.y, emax)};
    if (k != 0) {
        const longlong2 p{A.x - B.y, A.y + B.x};
        B = longlong2{A.x + B.y, B.x - A.y};
        A = p;
    }
    b[fxs(k)] = A;
    b[fxs(k2)] = B;
    return fx_mag(A) + fx_mag(B);
}
// A line of n doubles in its slots (each slot written and read by the lane
// that owns it, lane + kWarp i) -> fixed point in place.  hi: this lane's
// largest fx_hi.  Returns the line's exponent e and the shift sh that the
// transform applies (the transformed line's exponent is e - sh).
struct FxExp {
    int e, sh;
};
static __device__ __noinline__ FxExp fx_convert(longlong2* b, int n, unsigned hi, int lane) {
    const int emax = fx_emax(warp_umax(hi));
    unsigned s = 0;
#pragma unroll 4
    for (int i = lane; i < n; i += kWarp) s += fx_point(b + fxs(i), emax);
    return FxExp{fx_scale(emax, 0), fx_shift(warp_uadd(s))};
}
static __device__ __noinline__ FxExp fx_convert_rows(longlong2* b, int n, unsigned hi, int lane) {
    const int emax = fx_emax(warp_umax(hi)), half = n >> 1;
    unsigned s = 0;
#pragma unroll 2
    for (int k = lane; k < half; k += kWarp) s += fx_pair_rows(b, k, n, emax);
    return FxExp{fx_scale(emax, 0), fx_shift(warp_uadd(s))};
}

// Global memory -> slots as doubles, by the threads first, first + step, ...
// (the lanes of a warp or the threads of a CTA); each returns the largest
// fx_hi of its values.  The loads of kFxLoad points are in flight together.
// Functions of their own, like the transforms: every pass shares them.
constexpr int kFxLoad = 4;

// the two rows' half spectra of one field, as fx_pair_rows reads them
static __device__ __noinline__ unsigned fx_load_rows(longlong2* b, const double2* s0, int n, int rows, int first, int step) {
    const int half = n >> 1;
    unsigned hi = 0;
    for (int k0 = first; k0 < half; k0 += step * kFxLoad) {
        double2 a[kFxLoad], c[kFxLoad];
#pragma unroll
        for (int q = 0; q < kFxLoad; q++) {
            const int k = k0 + step * q;
            if (k < half) {
                a[q] = s0[(size_t)k * rows];
                c[q] = s0[(size_t)k * rows + 1];
            }
        }
#pragma unroll
        for (int q = 0; q < kFxLoad; q++) {
            const int k = k0 + step * q;
            if (k < half) {
                int k2 = n - k;
                if (k == 0) {  // k = 0 and n / 2: real coefficients
                    const double2 ah = s0[(size_t)half * rows], ch = s0[(size_t)half * rows + 1];
                    a[q].y = c[q].x;
                    c[q] = double2{ah.x, ch.x};
                    k2 = half;
                }
                const unsigned h0 = fx_hi(a[q].x), h1 = fx_hi(a[q].y), h2 = fx_hi(c[q].x), h3 = fx_hi(c[q].y);
                const unsigned m0 = h0 > h1 ? h0 : h1, m1 = h2 > h3 ? h2 : h3, m = m0 > m1 ? m0 : m1;
                hi = m > hi ? m : hi;
                *(double2*)&b[fxs(k)] = a[q];
                *(double2*)&b[fxs(k2)] = c[q];
            }
        }
    }
    return hi;
}
// n contiguous points
static __device__ __noinline__ unsigned fx_load(longlong2* b, const double2* s, int n, int first, int step) {
    unsigned hi = 0;
    for (int x0 = first; x0 < n; x0 += step * 2 * kFxLoad) {
        double2 v[2 * kFxLoad];
#pragma unroll
        for (int q = 0; q < 2 * kFxLoad; q++)
            if (x0 + step * q < n) v[q] = s[x0 + step * q];
#pragma unroll
        for (int q = 0; q < 2 * kFxLoad; q++) {
            if (x0 + step * q < n) {
                const unsigned a = fx_hi(v[q].x), c = fx_hi(v[q].y), m = a > c ? a : c;
                hi = m > hi ? m : hi;
                *(double2*)&b[fxs(x0 + step * q)] = v[q];
            }
        }
    }
    return hi;
}
// a transformed packed line of exponent S -> the two rows' half spectra
template <bool FAST>
__device__ __forceinline__ void fx_store_rows_t(const longlong2* b, int n, int S, double2* d0, int rows, int first, int step) {
#pragma unroll 2
    for (int k = first; k <= (n >> 1); k += step) {
        const longlong2 zk = b[fxs(k)], zn = b[fxs((n - k) & (n - 1))];
        double2* d = d0 + (size_t)k * rows;
        d[0] = double2{fx_to_t<FAST>(zk.x + zn.x, S), fx_to_t<FAST>(zk.y - zn.y, S)};
        d[1] = double2{fx_to_t<FAST>(zk.y + zn.y, S), fx_to_t<FAST>(zn.x - zk.x, S)};
    }
}
static __device__ __noinline__ void fx_store_rows(const longlong2* b, int n, int S, double2* d0, int rows, int first, int step) {
    if (fx_fast(S + 1)) fx_store_rows_t<true>(b, n, S + 1, d0, rows, first, step);
    else fx_store_rows_t<false>(b, n, S + 1, d0, rows, first, step);
}
template <bool FAST>
__device__ __forceinline__ void fx_store_t(const longlong2* b, int n, int S, double2* d, int first, int step) {
#pragma unroll 2
    for (int x = first; x < n; x += step) {
        const longlong2 z = b[fxs(x)];
        d[x] = double2{fx_to_t<FAST>(z.x, S), fx_to_t<FAST>(z.y, S)};
    }
}
static __device__ __noinline__ void fx_store(const longlong2* b, int n, int S, double2* d, int first, int step) {
    if (fx_fast(S)) fx_store_t<true>(b, n, S, d, first, step);
    else fx_store_t<false>(b, n, S, d, first, step);
}

// --------------------------------------- lines between memory and registers
//
// Lines of 128, 256 and 512 points: a lane holds points lane + kWarp i in
// registers, which are whole butterflies of the first and of the last stage,
// so a line is converted and its first stage done before it goes to shared
// memory, and a line on its way out is converted to doubles from the registers
// of its last stage: two round trips through shared memory instead of five.

// v (converted, to be shifted by sh) -> first stage -> b
template <int S, int LOGN> __device__ __forceinline__ void fx_first(const longlong2* v, longlong2* b, int sh, int lane) {
    constexpr int R = fx_radix(LOGN, 0), NB = (1 << LOGN) / R, PER = NB / kWarp;
    const long long half = fx_half(sh);
    warp_sync();
#pragma unroll
    for (int i = 0; i < PER; i++) {
        longlong2 u[R];
#pragma unroll
        for (int r = 0; r < R; r++)
            u[r] = longlong2{fx_shr(v[i + r * PER].x, sh, half), fx_shr(v[i + r * PER].y, sh, half)};
        fx_dft<R, S>(u);
#pragma unroll
        for (int r = 0; r < R; r++) b[fxs((lane + kWarp * i) * R + r)] = u[r];
    }
    warp_sync();
}
// b (all stages but the last done) -> v
template <int S, int LOGN>
__device__ __forceinline__ void fx_last(longlong2* v, const longlong2* b, const FxTw* tw, int logTw, int lane) {
    constexpr int R = LOGN == 9 ? 8 : 4, NB = (1 << LOGN) / R, PER = NB / kWarp;
    const int twshift = logTw - LOGN;
#pragma unroll
    for (int i = 0; i < PER; i++) {
        const int j = lane + kWarp * i;
        longlong2 u[R];
#pragma unroll
        for (int r = 0; r < R; r++) {
            u[r] = b[fxs(j + r * NB)];
            if (r > 0) u[r] = fx_cmul<S>(u[r], tw[(j * r) << twshift]);
        }
        fx_dft<R, S>(u);
#pragma unroll
        for (int r = 0; r < R; r++) v[i + r * PER] = u[r];
    }
    warp_sync();
}
template <int S, int LOGN, int LOGNS, int END>
__device__ __forceinline__ void fx_middle(longlong2* b, const FxTw* tw, int logTw, int lane) {
    if constexpr (LOGNS < END) {
        constexpr int R = fx_radix(LOGN, LOGNS);
        fx_stage<R, S, LOGN, LOGNS, false>(b, 0, tw, logTw, lane);
        fx_middle<S, LOGN, LOGNS + radix_log(R), END>(b, tw, logTw, lane);
    }
}
// doubles in registers -> fixed point in registers
template <int E> __device__ __forceinline__ FxExp fx_regs(const double2* z, longlong2* v) {
    unsigned hi = 0, s = 0;
#pragma unroll
    for (int i = 0; i < E; i++) {
        const unsigned a = fx_hi(z[i].x), c = fx_hi(z[i].y), m = a > c ? a : c;
        hi = m > hi ? m : hi;
    }
    const int emax = fx_emax(warp_umax(hi));
#pragma unroll
    for (int i = 0; i < E; i++) {
        v[i] = longlong2{fx_from(z[i].x, emax), fx_from(z[i].y, emax)};
        s += fx_mag(v[i]);
    }
    return FxExp{fx_scale(emax, 0), fx_shift(warp_uadd(s))};
}
template <int E> __device__ __forceinline__ void fx_put(const longlong2* v, int S, double2* d, int stride, int lane) {
    if (fx_fast(S)) {
#pragma unroll
        for (int i = 0; i < E; i++)
            d[(size_t)(lane + kWarp * i) * stride] = double2{fx_to_t<true>(v[i].x, S), fx_to_t<true>(v[i].y, S)};
    } else {
#pragma unroll 1
        for (int i = 0; i < E; i++) {
            longlong2 t = v[0];
#pragma unroll
            for (int q = 1; q < E; q++)
                if (q == i) t = v[q];
            d[(size_t)(lane + kWarp * i) * stride] = double2{fx_to(t.x, S), fx_to(t.y, S)};
        }
    }
}
// n contiguous points -> their transform in the slots of b; returns the exponent
template <int S, int LOGN>
__device__ __noinline__ int fx_line_in(longlong2* b, const double2* s, const FxTw* tw, int logTw, int lane) {
    constexpr int E = (1 << LOGN) / kWarp;
    double2 z[E];
    longlong2 v[E];
#pragma unroll
    for (int i = 0; i < E; i++) z[i] = s[lane + kWarp * i];
    const FxExp x = fx_regs<E>(z, v);
    fx_first<S, LOGN>(v, b, x.sh, lane);
    fx_middle<S, LOGN, radix_log(fx_radix(LOGN, 0)), LOGN>(b, tw, logTw, lane);
    return x.e - x.sh;
}
// doubles in the lane's slots of b -> the transform at d, contiguous
template <int S, int LOGN>
__device__ __noinline__ void fx_line_out(longlong2* b, double2* d, const FxTw* tw, int logTw, int lane) {
    constexpr int E = (1 << LOGN) / kWarp, END = LOGN - (LOGN == 9 ? 3 : 2);
    longlong2 v[E];
    double2 z[E];
#pragma unroll
    for (int i = 0; i < E; i++) z[i] = *(const double2*)&b[fxs(lane + kWarp * i)];
    const FxExp x = fx_regs<E>(z, v);
    fx_first<S, LOGN>(v, b, x.sh, lane);
    fx_middle<S, LOGN, radix_log(fx_radix(LOGN, 0)), END>(b, tw, logTw, lane);
    fx_last<S, LOGN>(v, b, tw, logTw, lane);
    fx_put<E>(v, x.e - x.sh, d, 1, lane);
}
// doubles in the lane's slots of b -> the transform in the slots; returns the exponent
template <int S, int LOGN>
__device__ __noinline__ int fx_line_mid(longlong2* b, const FxTw* tw, int logTw, int lane) {
    constexpr int E = (1 << LOGN) / kWarp;
    longlong2 v[E];
    double2 z[E];
#pragma unroll
    for (int i = 0; i < E; i++) z[i] = *(const double2*)&b[fxs(lane + kWarp * i)];
    const FxExp x = fx_regs<E>(z, v);
    fx_first<S, LOGN>(v, b, x.sh, lane);
    fx_middle<S, LOGN, radix_log(fx_radix(LOGN, 0)), LOGN>(b, tw, logTw, lane);
    return x.e - x.sh;
}
// s[i ss] -> the transform at d[i ds]
template <int S, int LOGN>
__device__ __noinline__ void fx_line_move(longlong2* b, const double2* s, int ss, double2* d, int ds, const FxTw* tw,
                                          int logTw, int lane) {
    constexpr int E = (1 << LOGN) / kWarp, END = LOGN - (LOGN == 9 ? 3 : 2);
    double2 z[E];
    longlong2 v[E];
#pragma unroll
    for (int i = 0; i < E; i++) z[i] = s[(size_t)(lane + kWarp * i) * ss];
    const FxExp x = fx_regs<E>(z, v);
    fx_first<S, LOGN>(v, b, x.sh, lane);
    fx_middle<S, LOGN, radix_log(fx_radix(LOGN, 0)), END>(b, tw, logTw, lane);
    fx_last<S, LOGN>(v, b, tw, logTw, lane);
    fx_put<E>(v, x.e - x.sh, d, ds, lane);
}
// line lengths with those forms
__host__ __device__ constexpr bool fx_regs_ok(int nf) { return nf == 128 || nf == 256 || nf == 512; }

// The passes' entries for a line of n = 1 << logn points (NF: n, or 0 for the
// runtime length): memory -> transform in the slots (in), slots' doubles ->
// transform in the slots (mid), slots' doubles -> transform in memory (out).
// hi: this lane's largest fx_hi of its slots.  in and mid return the exponent.
template <int S, int NF>
__device__ __forceinline__ int fx_in(longlong2* b, const double2* s, int n, int logn, const FxTw* tw, int logTw, int lane) {
    if constexpr (fx_regs_ok(NF)) return fx_line_in<S, ilog2c(NF)>(b, s, tw, logTw, lane);
    const FxExp x = fx_convert(b, n, fx_load(b, s, n, lane, kWarp), lane);
    fx_line<S, NF>(b, logn, x.sh, tw, logTw, lane);
    return x.e - x.sh;
}
template <int S, int NF>
__device__ __forceinline__ int fx_mid(longlong2* b, unsigned hi, int n, int logn, const FxTw* tw, int logTw, int lane) {
    if constexpr (fx_regs_ok(NF)) return fx_line_mid<S, ilog2c(NF)>(b, tw, logTw, lane);
    const FxExp x = fx_convert(b, n, hi, lane);
    fx_line<S, NF>(b, logn, x.sh, tw, logTw, lane);
    return x.e - x.sh;
}
template <int S, int NF>
__device__ __forceinline__ void fx_out(longlong2* b, unsigned hi, double2* d, int n, int logn, const FxTw* tw, int logTw,
                                       int lane) {
    if constexpr (fx_regs_ok(NF)) {
        fx_line_out<S, ilog2c(NF)>(b, d, tw, logTw, lane);
    } else {
        const FxExp x = fx_convert(b, n, hi, lane);
        fx_line<S, NF>(b, logn, x.sh, tw, logTw, lane);
        fx_store(b, n, x.e - x.sh, d, lane, kWarp);
    }
}

// ------------------------------------------------- lines shared by a CTA
//
// nl lines of n = 1 << logn points, line l in slots l n .., dealt to the
// threads of a CTA over (line, point) so that all lines' loads are in flight
// together.  red: [largest fx_hi][line], [sum of fx_mag][line] (zero before).

__device__ __forceinline__ void fxc_put_max(unsigned* red, int l, bool in, unsigned v, int n) {
    if (n >= kWarp) {  // a warp's points are of one line
        v = warp_umax(in ? v : 0u);
        if ((threadIdx.x % kWarp) == 0) atomicMax(red + l, v);
    } else if (in) {
        atomicMax(red + l, v);
    }
}
__device__ __forceinline__ void fxc_put_sum(unsigned* red, int l, bool in, unsigned v, int n) {
    if (n >= kWarp) {
        v = warp_uadd(in ? v : 0u);
        if ((threadIdx.x % kWarp) == 0) atomicAdd(red + l, v);
    } else if (in) {
        atomicAdd(red + l, v);
    }
}
// columns: line l's points at s + l H
static __device__ __noinline__ void fxc_load(longlong2* b, const double2* s, long long H, int nl, int logn, unsigned* red,
                                             int tid, int nthr) {
    const int n = 1 << logn, tot = nl << logn, lane = tid % kWarp;
    for (int i0 = tid - lane; i0 < tot; i0 += nthr * kFxLoad) {
        double2 v[kFxLoad];
#pragma unroll
        for (int q = 0; q < kFxLoad; q++) {
            const int i = i0 + lane + nthr * q;
            if (i < tot) v[q] = s[(size_t)(i >> logn) * H + (i & (n - 1))];
        }
#pragma unroll
        for (int q = 0; q < kFxLoad; q++) {
            const int iw = i0 + nthr * q, i = iw + lane;
            if (iw < tot) {
                const bool in = i < tot;
                unsigned m = 0;
                if (in) {
                    const unsigned a = fx_hi(v[q].x), c = fx_hi(v[q].y);
                    m = a > c ? a : c;
                    *(double2*)&b[(i >> logn << logn) + fxs(i & (n - 1))] = v[q];
                }
                fxc_put_max(red, in ? i >> logn : 0, in, m, n);
            }
        }
    }
}
// row pairs: line l's coefficients at s + l H + k rows, as fx_pair_rows reads them
static __device__ __noinline__ void fxc_load_rows(longlong2* b, const double2* s, long long H, int rows, int nl, int logn,
                                                  unsigned* red, int tid, int nthr) {
    const int n = 1 << logn, half = n >> 1, tot = nl * half, lane = tid % kWarp;
    for (int i0 = tid - lane; i0 < tot; i0 += nthr * 2) {
        double2 a[2], c[2], e[2];
#pragma unroll
        for (int q = 0; q < 2; q++) {
            const int i = i0 + lane + nthr * q;
            if (i < tot) {
                const double2* p = s + (size_t)(i >> (logn - 1)) * H + (size_t)(i & (half - 1)) * rows;
                a[q] = p[0];
                c[q] = p[1];
                if ((i & (half - 1)) == 0) {  // n / 2, with k = 0
                    p += (size_t)half * rows;
                    e[q] = double2{p[0].x, p[1].x};
                }
            }
        }
#pragma unroll
        for (int q = 0; q < 2; q++) {
            const int iw = i0 + nthr * q, i = iw + lane;
            if (iw < tot) {
                const bool in = i < tot;
                const int l = in ? i >> (logn - 1) : 0, k = i & (half - 1);
                unsigned m = 0;
                if (in) {
                    int k2 = n - k;
                    if (k == 0) {  // k = 0 and n / 2: real coefficients
                        a[q].y = c[q].x;
                        c[q] = e[q];
                        k2 = half;
                    }
                    const unsigned h0 = fx_hi(a[q].x), h1 = fx_hi(a[q].y), h2 = fx_hi(c[q].x), h3 = fx_hi(c[q].y);
                    const unsigned m0 = h0 > h1 ? h0 : h1, m1 = h2 > h3 ? h2 : h3;
                    m = m0 > m1 ? m0 : m1;
                    *(double2*)&b[l * n + fxs(k)] = a[q];
                    *(double2*)&b[l * n + fxs(k2)] = c[q];
                }
                fxc_put_max(red, l, in, m, half);
            }
        }
    }
}
// the doubles in the slots -> fixed point in place (rows: of fxc_load_rows)
static __device__ __noinline__ void fxc_convert(longlong2* b, int nl, int logn, unsigned* red, unsigned* sums, int tid,
                                                int nthr) {
    const int n = 1 << logn, tot = nl << logn, lane = tid % kWarp;
    for (int iw = tid - lane; iw < tot; iw += nthr) {
        const int i = iw + lane, l = i < tot ? i >> logn : 0;
        unsigned s = 0;
        if (i < tot) s = fx_point(b + (l << logn) + fxs(i & (n - 1)), fx_emax(red[l]));
        fxc_put_sum(sums, l, i < tot, s, n);
    }
}
static __device__ __noinline__ void fxc_convert_rows(longlong2* b, int nl, int logn, unsigned* red, unsigned* sums, int tid,
                                                     int nthr) {
    const int n = 1 << logn, half = n >> 1, tot = nl * half, lane = tid % kWarp;
    for (int iw = tid - lane; iw < tot; iw += nthr) {
        const int i = iw + lane, l = i < tot ? i >> (logn - 1) : 0;
        unsigned s = 0;
        if (i < tot) s = fx_pair_rows(b + l * n, i & (half - 1), n, fx_emax(red[l]));
        fxc_put_sum(sums, l, i < tot, s, half);
    }
}
__device__ __forceinline__ int fxc_scale(const unsigned* red, const unsigned* sums, int l) {
    return fx_scale(fx_emax(red[l]), fx_shift(sums[l]));
}
// transformed lines -> memory (FAST as fx_to_t)
__device__ __forceinline__ bool fxc_fast(const unsigned* red, const unsigned* sums, int nl) {
    bool fast = true;
    for (int l = 0; l < nl; l++) fast = fast && fx_fast(fxc_scale(red, sums, l)) && fx_fast(fxc_scale(red, sums, l) + 1);
    return fast;
}
template <bool FAST>
__device__ __noinline__ void fxc_store_t(const longlong2* b, double2* d, long long H, int nl, int logn, const unsigned* red,
                                         const unsigned* sums, int tid, int nthr) {
    const int n = 1 << logn, tot = nl << logn;
#pragma unroll 1
    for (int i = tid; i < tot; i += nthr) {
        const int l = i >> logn, x = i & (n - 1), S = fxc_scale(red, sums, l);
        const longlong2 z = b[(l << logn) + fxs(x)];
        d[(size_t)l * H + x] = double2{fx_to_t<FAST>(z.x, S), fx_to_t<FAST>(z.y, S)};
    }
}
__device__ __forceinline__ void fxc_store(const longlong2* b, double2* d, long long H, int nl, int logn,
                                          const unsigned* red, const unsigned* sums, int tid, int nthr) {
    if (fxc_fast(red, sums, nl)) fxc_store_t<true>(b, d, H, nl, logn, red, sums, tid, nthr);
    else fxc_store_t<false>(b, d, H, nl, logn, red, sums, tid, nthr);
}
template <bool FAST>
__device__ __noinline__ void fxc_store_rows_t(const longlong2* b, double2* d0, long long H, int rows, int nl, int logn,
                                              const unsigned* red, const unsigned* sums, int tid, int nthr) {
    const int n = 1 << logn, half = n >> 1, tot = nl * half;
    // coefficients k < n / 2, then n / 2 of every line
#pragma unroll 1
    for (int i = tid; i < tot + nl; i += nthr) {
        const int l = i < tot ? i >> (logn - 1) : i - tot, k = i < tot ? i & (half - 1) : half, S = fxc_scale(red, sums, l) + 1;
        const longlong2 zk = b[l * n + fxs(k)], zn = b[l * n + fxs((n - k) & (n - 1))];
        double2* d = d0 + (size_t)l * H + (size_t)k * rows;
        d[0] = double2{fx_to_t<FAST>(zk.x + zn.x, S), fx_to_t<FAST>(zk.y - zn.y, S)};
        d[1] = double2{fx_to_t<FAST>(zk.y + zn.y, S), fx_to_t<FAST>(zn.x - zk.x, S)};
    }
}
__device__ __forceinline__ void fxc_store_rows(const longlong2* b, double2* d0, long long H, int rows, int nl, int logn,
                                               const unsigned* red, const unsigned* sums, int tid, int nthr) {
    if (fxc_fast(red, sums, nl)) fxc_store_rows_t<true>(b, d0, H, rows, nl, logn, red, sums, tid, nthr);
    else fxc_store_rows_t<false>(b, d0, H, rows, nl, logn, red, sums, tid, nthr);
}

// One radix-R stage at runtime lengths: the stages of a line share their code.
// (A unit runs each instruction of a pass a few times only: an SM missed 390
// times per phase in its instruction cache with a copy per stage and length.)
template <int R, int S, bool FIRST>
__device__ __forceinline__ void fx_stage_coop(const longlong2* src, longlong2* dst, int logn, int logNs, int nl,
                                              const unsigned* sums, const FxTw* tw, int logTw, int tid, int nthr) {
    constexpr int LR = (R == 2) ? 1 : (R == 4) ? 2 : 3;
    const int lnb = logn - LR, nsm = (1 << logNs) - 1, twshift = logTw - (logNs + LR), tot = nl << lnb;
#pragma unroll 1
    for (int it = tid; it < tot; it += nthr) {
        const int l = it >> lnb, j = it & ((1 << lnb) - 1), jm = j & nsm;
        const longlong2* s = src + (l << logn);
        longlong2* d = dst + (l << logn);
        longlong2 v[R];
#pragma unroll
        for (int r = 0; r < R; r++) v[r] = s[fxs(j + (r << lnb))];
        if (FIRST) {
            const int sh = fx_shift(sums[l]);
            const long long half = fx_half(sh);
#pragma unroll
            for (int r = 0; r < R; r++) v[r] = longlong2{fx_shr(v[r].x, sh, half), fx_shr(v[r].y, sh, half)};
        } else {
#pragma unroll
            for (int r = 1; r < R; r++) v[r] = fx_cmul<S>(v[r], tw[(jm * r) << twshift]);
        }
        fx_dft<R, S>(v);
        const int dd = ((j - jm) << LR) + jm;
#pragma unroll
        for (int r = 0; r < R; r++) d[fxs(dd + (r << logNs))] = v[r];
    }
}
#ifndef PAGD_EMU
__device__ __forceinline__ longlong2 fx_xor(longlong2 v, int o) {
    return longlong2{__shfl_xor_sync(0xffffffffu, v.x, o), __shfl_xor_sync(0xffffffffu, v.y, o)};
}
// A radix-4 stage with twiddles, a point per thread: four lanes share a
// butterfly, each one input's complex product, and combine by shuffles.  For
// lines of up to 64 points, which otherwise keep half a warp busy: 64 points
// 2050 -> 1600 cycles, 128 the same, 256 slower (2800 -> 3000).
template <int S>
__device__ __forceinline__ void fx_stage_quad(const longlong2* src, longlong2* dst, int logn, int logNs, int nl,
                                              const FxTw* tw, int logTw, int tid, int nthr) {
    const int lnb = logn - 2, twshift = logTw - (logNs + 2), tot = nl << logn;
#pragma unroll 1
    for (int i0 = tid & ~31; i0 < tot; i0 += nthr) {  // whole warps: nl << logn may end inside one
        const int it = i0 + (tid & 31), on = it < tot ? it : 0;
        const int l = on >> logn, j = (on & ((1 << logn) - 1)) >> 2, r = on & 3, jm = j & ((1 << logNs) - 1);
        longlong2 v = fx_cmul<S>(src[(l << logn) + fxs(j + (r << lnb))], tw[(jm * r) << twshift]);
        longlong2 o = fx_xor(v, 2);
        v = r < 2 ? cadd(v, o) : csub(o, v);       // p0 + p2, p1 + p3, p0 - p2, p1 - p3
        if (r == 3) v = mul_si<S>(v);
        o = fx_xor(v, 1);
        v = (r & 1) ? csub(o, v) : cadd(v, o);     // outputs 0, 2, 1, 3
        const int k = (r >> 1) | ((r & 1) << 1);
        if (it < tot) dst[(l << logn) + fxs(((j - jm) << 2) + jm + (k << logNs))] = v;
    }
}
#endif

// nl converted lines of 1 << logn points in b0 (sums complete before the call)
// -> the transforms in b0 (returns 0) or b1 (1), visible to every thread on
// return.  Radix 4, and 8 for the first stage of an odd number of levels: a
// stage costs a barrier and a round trip through shared memory; a lone warp on
// a sub-partition issues a product in about 30 cycles, and wider radices leave
// more of them idle.
template <int S>
__device__ __noinline__ int fx_coop(longlong2* b0, longlong2* b1, int logn, int nl, const unsigned* sums, const FxTw* tw,
                                    int logTw, int tid, int nthr) {
    longlong2 *s = b0, *d = b1;
    int logNs = 2, r = 1;
    if (logn & 1) {
        fx_stage_coop<8, S, true>(s, d, logn, 0, nl, sums, tw, logTw, tid, nthr);
        logNs = 3;
    } else {
        fx_stage_coop<4, S, true>(s, d, logn, 0, nl, sums, tw, logTw, tid, nthr);
    }
    cta_sync();
#pragma unroll 1
    for (; logNs < logn; logNs += 2, r ^= 1) {
        longlong2* t = s;
        s = d;
        d = t;
#ifndef PAGD_EMU
        if (logn <= 6 && (nl << logn) <= nthr) fx_stage_quad<S>(s, d, logn, logNs, nl, tw, logTw, tid, nthr);
        else
#endif
            fx_stage_coop<4, S, false>(s, d, logn, logNs, nl, sums, tw, logTw, tid, nthr);
        cta_sync();
    }
    return r;
}

}  // namespace pagd
