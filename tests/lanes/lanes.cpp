// The passes of solver.cuh on the lane emulation (compat.cuh beside this file),
// with a pointwise step that hands its fields through.
#include "solver.cuh"

using namespace pagd;

namespace {
struct Nothing {};
template <class T> std::vector<cx<T>> table() {
    std::vector<cx<T>> t(512);
    for (int m = 0; m < 512; m++) {
        const double a = -2.0 * 3.14159265358979323846 * m / 512;
        t[m] = cx<T>{(T)cos(a), (T)sin(a)};
    }
    return t;
}
struct Setup {
    std::vector<FxTw> fx;
    std::vector<float2> t32 = table<float>();
    std::vector<double> sq;
    std::vector<char> smem;
    Params P;
    Setup(int n0, int nm, int n1, int warps) : fx(512), sq(kSq), smem(256 * 1024 * 2) {
        for (int m = 0; m < 512; m++) {
            const long double a = -2.0L * 3.141592653589793238462643383279502884L * m / 512, o = (long double)(1ull << kFxTw);
            fx[m] = fx_tw(llroundl(cosl(a) * o), llroundl(sinl(a) * o));
        }
        for (int m = 0; m < kSq; m++) sq[m] = (double)(m * m);
        std::memset((void*)&P, 0, sizeof(P));
        P.n0 = n0; P.nm = nm; P.n1 = n1;
        P.logn0 = ilog2c(n0); P.logm = ilog2c(nm); P.logn1 = ilog2c(n1);
        P.h1 = n1 / 2 + 1;
        P.rows = n0 * nm;
        P.ncols = P.h1 * nm;
        P.H = (long long)P.h1 * P.rows;
        P.npts = (long long)P.rows * n1;
        P.inv_npts = 1.0 / (double)P.npts;
        P.warp_bytes = (long long)(smem.size() / warps) & ~127ll;
        P.k0sq = P.k1sq = P.kmsq = 1.0;
        P.k0sqf = P.k1sqf = P.kmsqf = 1.f;
    }
    char* mem() { return (char*)(((uintptr_t)smem.data() + 127) & ~(uintptr_t)127); }
    Tw tw(int warps) {
        const int w = threadIdx.x / kWarp;
        return Tw{fx.data(), t32.data(), sq.data(), 9, w, warps, 0, -1, w, warps, nullptr};
    }
};
auto ld_row = [](long long, int, int) { return Nothing{}; };
auto ld_col = [](const Line&, int) { return Nothing{}; };

// state: scale of the pointwise state that the staged passes add to every field (0: none)
template <int NF> bool run(const char* pass, int n, int k, bool up, float state, const double* src, double* dst) {
    auto is = [&](const char* s) { return std::strcmp(pass, s) == 0; };
    const bool row = pass[0] == 'r', mid = pass[0] == 'm';
    const int other = 8, warps = (std::strstr(pass, "coop") || std::strstr(pass, "pair")) ? 4 : 2;
    Setup S(mid ? other : row ? other : n, mid ? n : 1, row ? n : other, std::strstr(pass, "pair") ? 2 : warps);
    Params& P = S.P;
    if (std::strstr(pass, "pair")) P.warp_bytes /= 2;  // a pair's unit lies in its first warp's slice, two slices apart
    const size_t H = (size_t)P.H;
    const double2* s64 = (const double2*)src;
    double2* d64 = (double2*)dst;
    std::vector<float2> s32(H * 3), d32(H * 3);
    for (size_t i = 0; i < H * k; i++) s32[i] = float2{(float)s64[i].x, (float)s64[i].y};
    gridDim.x = 1;
    char* mem = S.mem();
    bool f32 = true;
    auto rf = [&](long long, int, int, const Nothing&, const auto* in, auto* out) { for (int f = 0; f < k; f++) out[f] = in[f]; };
    auto cf = [&](const Line&, int, const Nothing&, const auto* in, auto* out) { for (int f = 0; f < k; f++) out[f] = in[f]; };
    // as phase C: three FP64 fields in, one FP32 out
    auto csum = [&](const Line&, int, const Nothing&, const double2* in, float2* out) {
        double2 t{0.0, 0.0};
        for (int f = 0; f < k; f++) t = cadd(t, in[f]);
        out[0] = float2{(float)t.x, (float)t.y};
    };
    auto rs = [&](long long p, int row, int x, const float* sv, const float* in, float* out) {
        const float bad = p == (long long)row * P.n1 + x ? 0.f : NAN;
        for (int f = 0; f < k; f++) out[f] = in[f] + sv[f] + bad;
    };
    auto cs = [&](const Line& l, int k0, const float2* sv, const float2* in, float2* out) {
        for (int f = 0; f < k; f++) out[f] = float2{in[f].x + sv[f].x, in[f].y + sv[f].y * (float)(l.l + k0 != 3)};
    };
    std::vector<float> st[2];
    std::vector<float2> sl[2];
    for (int a = 0; a < 2; a++) {
        for (long long i = 0; i < P.npts; i++) st[a].push_back(state * (float)((i * 37 + a * 11) % 101));
        for (size_t i = 0; i < H; i++) sl[a].push_back(float2{state * (float)(i * 41 % 103), state * (float)((i + a) * 43 % 107)});
    }
    const float* sp[2] = {st[0].data(), st[1].data()};
    const float2* sc[2] = {sl[0].data(), sl[1].data()};
    const bool ok = emu_cta(warps * 32, up, 0, [&](int) {
        const Tw t = S.tw(warps);
        if (is("row_fx")) { f32 = false; row_pass_fx<NF>(P, t, k, k, s64, d64, mem, ld_row, rf); }
        else if (is("row_coop_fx")) { f32 = false; row_pass_coop_fx<NF>(P, t, k, k, s64, d64, mem, ld_row, rf); }
        else if (is("col_fx")) { f32 = false; col_pass_fx<double, NF>(P, t, k, k, s64, d64, mem, ld_col, cf); }
        else if (is("col_coop_fx")) { f32 = false; col_pass_coop_fx<double, NF>(P, t, k, k, s64, d64, mem, ld_col, cf); }
        else if (is("col_sum_fx")) col_pass_fx<float, NF>(P, t, k, 1, s64, d32.data(), mem, ld_col, csum);
        else if (is("col_sum_coop_fx")) col_pass_coop_fx<float, NF>(P, t, k, 1, s64, d32.data(), mem, ld_col, csum);
        else if (is("row_coop")) row_pass_coop<NF>(P, t, k, k, s32.data(), d32.data(), mem, ld_row, rf);
        else if (is("col_coop")) col_pass_coop<NF>(P, t, k, k, s32.data(), d32.data(), mem, ld_col, cf);
        else if (is("mid_fx_fwd")) { f32 = false; mid_pass_fx<-1, NF>(P, t, k, s64, d64, mem); }
        else if (is("mid_fx_inv")) { f32 = false; mid_pass_fx<+1, NF>(P, t, k, s64, d64, mem); }
        else if constexpr (NF > 0) {
            if (is("row_staged")) {
                if (k == 1) row_pass_staged<NF, 1, 2>(P, t, s32.data(), d32.data(), sp, mem, rs);
                else row_pass_staged<NF, 2, 2>(P, t, s32.data(), d32.data(), sp, mem, rs);
            } else if (is("col_staged")) {
                if (k == 1) col_pass_staged<NF, 1, 2>(P, t, s32.data(), d32.data(), sc, mem, cs);
                else col_pass_staged<NF, 2, 2>(P, t, s32.data(), d32.data(), sc, mem, cs);
            } else if (is("row_pair")) row_pass_pair<NF, 2>(P, t, s32.data(), d32.data(), sp, mem, rs);
            else if (is("col_pair")) col_pass_pair<NF, 2>(P, t, s32.data(), d32.data(), sc, mem, cs);
            else if (is("mid_staged_fwd")) mid_pass_staged<NF, -1>(P, t, k, s32.data(), d32.data(), mem);
            else if (is("mid_staged_inv")) mid_pass_staged<NF, +1>(P, t, k, s32.data(), d32.data(), mem);
        }
    });
    if (f32)
        for (size_t i = 0; i < H * k; i++) d64[i] = double2{d32[i].x, d32[i].y};
    return ok;
}
}  // namespace

extern "C" {
// one pass over k fields of a grid whose transformed axis has n points and the
// others 8; 1: done
int lanes_pass(const char* pass, int n, int nf, int k, int up, double state, const double* src, double* dst) {
    switch (nf) {
        case 0: return run<0>(pass, n, k, up != 0, (float)state, src, dst);
        case 64: return run<64>(pass, n, k, up != 0, (float)state, src, dst);
        case 128: return run<128>(pass, n, k, up != 0, (float)state, src, dst);
        case 512: return run<512>(pass, n, k, up != 0, (float)state, src, dst);
    }
    return 0;
}
// publish_group by one CTA of nw warps: maximum and sums of the warps' values
int lanes_publish(int nw, int up, const unsigned long long* m, const double* v, unsigned long long* mo, double* vo) {
    gridDim.x = kFewCtas + 1;
    *mo = 0;
    for (int i = 0; i < 3; i++) vo[i] = 0.0;
    return emu_cta(nw * 32, up != 0, sizeof(CtaRed), [&](int t) {
        Tw tw{};
        tw.cr = (CtaRed*)emu_region();
        double* const a[3] = {vo, vo + 1, vo + 2};
        const int w = t / 32;
        const double x[3] = {v[3 * w], v[3 * w + 1], v[3 * w + 2]};
        publish_group<3>(tw, true, mo, m[w], a, x);
    });
}
// The short control path and the whole machine after the phase ph (0: CI, 1: RI)
// of an iteration: 0: both leave the same state, 1: the short path leaves the
// decision to the machine (and the state alone), 2: they differ.
int lanes_ctl(int t64, int ph, int ev, int best_ev, double best, double base, double nrm, double tol, int max_iter, int last) {
    Setup S(8, 1, 8, 1);
    Params& P = S.P;
    P.prog = PROG_RUN;
    P.precision = t64 ? P_FP64 : P_MIXED;
    P.tol = tol;
    P.max_iter = max_iter;
    P.max_recheck = 16;
    P.nsteps = last ? 1 : 3;
    P.nslots = 64;
    std::vector<unsigned long long> norms(2 * P.nslots, 0);
    std::vector<double> mass(3, 0.0);
    P.norms = norms.data();
    P.mass = mass.data();
    Ctl c;
    std::memset((void*)&c, 0, sizeof(c));
    c.ph = ph ? PH_RI : PH_CI;
    c.it = 3;
    c.ev = ev;
    c.best_ev = best_ev;
    c.best_nrm = best;
    c.base_nrm = base;
    c.reb_nrm = kRebaseRatio * base;
    c.exact_done = 1;
    norms[ev] = dbl_bits(nrm);
    Ctl a, b;
    std::memcpy((void*)&a, (void*)&c, sizeof(c));
    std::memcpy((void*)&b, (void*)&c, sizeof(c));
    const bool fast = t64 ? ctl_fast<double>(P, a) : ctl_fast<float>(P, a);
    if (!fast) return std::memcmp((void*)&a, (void*)&c, sizeof(c)) == 0 ? 1 : 2;
    if (t64) ctl_advance<double>(P, b);
    else ctl_advance<float>(P, b);
    return std::memcmp((void*)&a, (void*)&b, sizeof(c)) == 0 ? 0 : 2;
}
}
