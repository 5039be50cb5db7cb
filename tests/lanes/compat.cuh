// compat.cuh for the lane emulation (tests/test_lanes_host.py): stands in for
// csrc/compat.cuh and runs every thread of a CTA as a fiber with its own lane,
// so that code which relies on an order that no barrier gives shows.
//
// A fiber runs until it has to wait (for its warp, a pair of warps or the CTA);
// only then does the next one run, in ascending or descending order of the
// thread index.  What the programming model leaves open is taken the worst way:
//  - lanes do not advance together between barriers;
//  - a shuffle exchanges values and orders no memory: of the structure made
//    coherent by emu_region() every thread has a copy of its own, which only
//    its own fence or a barrier brings up to date;
//  - an asynchronous copy is done when its group is waited for.
#pragma once
#include <ucontext.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <functional>
#include <vector>

#define __device__
#define __host__
#define __global__
#define __forceinline__ inline
#define __noinline__
#define __launch_bounds__(...)

struct EmuDim3 { unsigned x, y, z; };
inline EmuDim3 threadIdx{0, 0, 0}, blockIdx{0, 0, 0}, blockDim{1, 1, 1}, gridDim{1, 1, 1};
struct alignas(8) float2 { float x, y; };
struct alignas(16) double2 { double x, y; };
struct alignas(16) float4 { float x, y, z, w; };
struct alignas(16) longlong2 { long long x, y; };

enum { EMU_RUN, EMU_DONE, EMU_WARP, EMU_SHFL, EMU_PAIR, EMU_CTA };
struct EmuCopy { void* dst; const void* src; };
struct EmuFiber {
    ucontext_t ctx;
    std::vector<char> stack;
    int state = EMU_RUN, key = 0, parity = 0;
    unsigned long long slot[2] = {0, 0};
    std::vector<std::vector<EmuCopy>> groups;  // committed
    std::vector<EmuCopy> open;
    std::vector<char> copy, base;  // this thread's view of the region
};
inline std::vector<EmuFiber> emu_f;
inline ucontext_t emu_main;
inline std::function<void(int)> emu_body;
inline std::vector<char> emu_shared;  // the region as last published
inline bool emu_stuck = false;

inline void emu_publish(EmuFiber& f) {
    for (size_t i = 0; i < f.copy.size(); i++)
        if (f.copy[i] != f.base[i]) emu_shared[i] = f.copy[i];
}
inline void emu_refresh(EmuFiber& f) {
    f.copy.assign(emu_shared.begin(), emu_shared.end());
    f.base = f.copy;
}
inline EmuFiber& emu_self() { return emu_f[threadIdx.x]; }
inline void emu_wait(int kind, int key) {
    EmuFiber& f = emu_self();
    f.state = kind;
    f.key = key;
    swapcontext(&f.ctx, &emu_main);
}
inline void emu_entry() {
    emu_body((int)threadIdx.x);
    emu_self().state = EMU_DONE;
    swapcontext(&emu_self().ctx, &emu_main);
}
// runs one CTA of n threads; false: threads wait for each other at different places
inline bool emu_cta(int n, bool ascending, size_t region, std::function<void(int)> body) {
    emu_body = body;
    blockDim = EmuDim3{(unsigned)n, 1, 1};
    emu_shared.assign(region, 0);
    emu_f.clear();
    emu_f.resize(n);
    for (auto& f : emu_f) {
        f.stack.resize(256 * 1024);
        emu_refresh(f);
        getcontext(&f.ctx);
        f.ctx.uc_stack.ss_sp = f.stack.data();
        f.ctx.uc_stack.ss_size = f.stack.size();
        f.ctx.uc_link = nullptr;
        makecontext(&f.ctx, emu_entry, 0);
    }
    auto release = [&](int lo, int hi, int kind, int key) {
        for (int i = lo; i < hi; i++)
            if (emu_f[i].state != kind || emu_f[i].key != key) return false;
        if (kind != EMU_SHFL) {
            for (int i = lo; i < hi; i++) emu_publish(emu_f[i]);
            for (int i = lo; i < hi; i++) emu_refresh(emu_f[i]);
        }
        for (int i = lo; i < hi; i++) emu_f[i].state = EMU_RUN;
        return true;
    };
    for (;;) {
        bool moved = false, done = true;
        for (int q = 0; q < n; q++) {
            const int i = ascending ? q : n - 1 - q;
            if (emu_f[i].state != EMU_RUN) continue;
            threadIdx.x = (unsigned)i;
            swapcontext(&emu_main, &emu_f[i].ctx);
            moved = true;
        }
        for (int w = 0; w < n; w += 32) {
            moved |= release(w, w + 32, EMU_WARP, w / 32) || release(w, w + 32, EMU_SHFL, w / 32);
            if (w % 64 == 0 && w + 64 <= n) moved |= release(w, w + 64, EMU_PAIR, w / 64);
        }
        moved |= release(0, n, EMU_CTA, 0);
        for (auto& f : emu_f) done = done && f.state == EMU_DONE;
        if (done) return true;
        if (!moved) return false;
    }
}
// this thread's copy of the region
inline void* emu_region() { return emu_self().copy.data(); }

inline void __syncwarp() { emu_wait(EMU_WARP, threadIdx.x / 32); }
inline void __syncthreads() { emu_wait(EMU_CTA, 0); }
inline void pair_sync(int p) { emu_wait(EMU_PAIR, p); }
inline void __threadfence_block() {
    emu_publish(emu_self());
    emu_refresh(emu_self());
}
inline void __threadfence() { __threadfence_block(); }

// every lane's value, by lane of this warp
template <class T, class F> inline T emu_all(T v, F&& f) {
    EmuFiber& s = emu_self();
    const int p = s.parity, w0 = (int)(threadIdx.x & ~31u);
    static_assert(sizeof(T) <= 8, "");
    std::memcpy(&s.slot[p], &v, sizeof(T));
    s.parity ^= 1;
    emu_wait(EMU_SHFL, threadIdx.x / 32);
    return f([&](int lane) {
        T t;
        std::memcpy(&t, &emu_f[w0 + lane].slot[p], sizeof(T));
        return t;
    });
}
template <class T> inline T __shfl_xor_sync(unsigned, T v, int o) {
    const int l = threadIdx.x & 31;
    return emu_all(v, [&](auto get) { return get(l ^ o); });
}
template <class T> inline T warp_xor(T v, int o) { return __shfl_xor_sync(0xffffffffu, v, o); }
inline unsigned warp_bcast(unsigned v) { return emu_all(v, [&](auto get) { return get(0); }); }
template <class T> inline T warp_max(T v) {
    for (int o = 16; o > 0; o >>= 1) {
        T w = warp_xor(v, o);
        v = (w > v || w != w) ? w : v;
    }
    return v;
}
template <class T> inline T warp_sum(T v) {
    for (int o = 16; o > 0; o >>= 1) v += warp_xor(v, o);
    return v;
}
inline unsigned warp_umax(unsigned v) {
    return emu_all(v, [&](auto get) { unsigned m = 0; for (int l = 0; l < 32; l++) m = std::max<unsigned>(m, get(l)); return m; });
}
inline unsigned warp_uadd(unsigned v) {
    return emu_all(v, [&](auto get) { unsigned m = 0; for (int l = 0; l < 32; l++) m += get(l); return m; });
}

// atomics act on the published region
template <class T> inline T* emu_atomic(T* p) {
    EmuFiber& s = emu_self();
    char* c = (char*)p;
    if (s.copy.empty() || c < s.copy.data() || c >= s.copy.data() + s.copy.size()) return p;
    return (T*)(emu_shared.data() + (c - s.copy.data()));
}
template <class T> inline void emu_seen(T* p, T v) {
    EmuFiber& s = emu_self();
    if (emu_atomic(p) == p) return;
    std::memcpy(p, &v, sizeof(T));
    std::memcpy(s.base.data() + ((char*)p - s.copy.data()), &v, sizeof(T));
}
template <class T, class F> inline T emu_rmw(T* p, F&& f) {
    T* g = emu_atomic(p);
    const T o = *g;
    *g = f(o);
    emu_seen(p, *g);
    return o;
}
template <class T> inline T atomicAdd(T* p, T v) { return emu_rmw(p, [&](T o) { return (T)(o + v); }); }
template <class T> inline T atomicMax(T* p, T v) { return emu_rmw(p, [&](T o) { return o > v ? o : v; }); }
inline int atomicOr(int* p, int v) { return emu_rmw(p, [&](int o) { return o | v; }); }

template <class T> inline T ldcg(const T* p) { return *p; }
template <class T> inline T ldg(const T* p) { return *p; }
inline unsigned long long dbl_bits(double d) { unsigned long long u; std::memcpy(&u, &d, 8); return u; }
inline double bits_dbl(unsigned long long u) { double d; std::memcpy(&d, &u, 8); return d; }
inline unsigned flt_bits(float f) { unsigned u; std::memcpy(&u, &f, 4); return u; }
inline float bits_flt(unsigned u) { float f; std::memcpy(&f, &u, 4); return f; }
inline float fadd(float a, float b) { return a + b; }
inline int clz32(unsigned v) { return v ? __builtin_clz(v) : 32; }
inline int clz64(unsigned long long v) { return v ? __builtin_clzll(v) : 64; }
#define PAGD_WARP 32

inline void cp_async16(void* dst, const void* src) { emu_self().open.push_back(EmuCopy{dst, src}); }
inline void cp_async_commit() {
    EmuFiber& s = emu_self();
    s.groups.push_back(s.open);
    s.open.clear();
}
template <int N> inline void cp_async_wait() {
    EmuFiber& s = emu_self();
    while ((int)s.groups.size() > N) {
        for (auto& c : s.groups.front()) std::memcpy(c.dst, c.src, 16);
        s.groups.erase(s.groups.begin());
    }
}
