// warp_fibers.h -- CUDA's device built-ins for one CTA on the CPU: every lane is
// a fiber, the lanes of a warp run one after the other from one warp collective
// to the next, and the warps take turns by a clock of their own that each fence,
// sleep and (now and then) collective moves on by a random length from a seed.
// One thread, no GPU, the same run for the same seed.
#pragma once
#include <cuda_runtime.h>
#include <setjmp.h>
#include <ucontext.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <vector>

using std::max;
using std::min;
#undef __forceinline__
#undef __noinline__
#undef __launch_bounds__
#define __forceinline__ inline
#define __noinline__
#define __launch_bounds__(...)

namespace fibers {

constexpr int kMaxWarps = 16;
struct Lane {
    ucontext_t first;
    jmp_buf at;
    bool started = false;
    unsigned parity = 0;
    std::vector<char> stack;
};
struct Warp {
    Lane lane[32];
    uint64_t slot[2][32];
    double clock = 0;
    bool done = false, waits = false;   // (waits: at the CTA's barrier)
    bool slow = false;                  // the event under way took a sine and cosine
};
inline Warp warp[kMaxWarps];
inline int warps, w, l;
inline void (*body)();
inline jmp_buf back;
inline uint64_t rng = 1, passes, limit;
inline double slow_events = 1.0;        // length of an event with a sine and cosine, against the others
inline int jitter = 64;                 // a warp also yields at every jitter-th collective or so

inline uint64_t random() { rng ^= rng << 13; rng ^= rng >> 7; rng ^= rng << 17; return rng; }

inline void entry() {
    for (;;) {
        body();
        Warp &W = warp[w];
        if (l < 31) {
            ++l;
        } else {
            W.done = true;
            l = -1;
        }
        extern void go();
        go();
    }
}
// on to lane l of warp w, or (l < 0) to the next warp
inline void enter() {
    Lane &L = warp[w].lane[l];
    if (!L.started) {
        L.started = true;
        setcontext(&L.first);
    }
    _longjmp(L.at, 1);
}
inline void pick() {
    int best = -1;
    for (int i = 0; i < warps; ++i)
        if (!warp[i].done && !warp[i].waits && (best < 0 || warp[i].clock < warp[best].clock)) best = i;
    if (best < 0) {
        bool any = false;
        for (int i = 0; i < warps; ++i) {
            any = any || warp[i].waits;
            if (warp[i].waits && !warp[i].done && best < 0) best = i;
            warp[i].waits = false;
        }
        if (!any) _longjmp(back, 1);
    }
    w = best;
    l = 0;
}
inline void go() {
    if (l < 0) pick();
    enter();
}
// the lane waits for the others of its warp; the last one may let other warps run
inline void meet(double time, bool barrier = false) {
    Warp &W = warp[w];
    if (_setjmp(W.lane[l].at)) return;
    if (l < 31) {
        ++l;
        enter();
    }
    W.waits = barrier;
    if (time > 0) W.clock += time * (0.5 + (double)(random() >> 11) * 0x1p-53);
    if (barrier || time > 0 || random() % jitter == 0) {
        if (++passes > limit) _longjmp(back, 2);
        l = -1;
    } else {
        l = 0;
    }
    go();
}
// 0: every warp has come to its end; 2: the limit of passes was reached first
inline int run(int n_warps, void (*f)(), uint64_t seed, uint64_t pass_limit) {
    warps = n_warps;
    body = f;
    rng = seed * 0x9E3779B97F4A7C15ull + 1;
    passes = 0;
    limit = pass_limit;
    for (int i = 0; i < warps; ++i) {
        warp[i].clock = 0;
        warp[i].done = warp[i].waits = false;
        for (Lane &L : warp[i].lane) {
            L.started = false;
            L.parity = 0;
            L.stack.resize(64 << 10);
            getcontext(&L.first);
            L.first.uc_stack.ss_sp = L.stack.data();
            L.first.uc_stack.ss_size = L.stack.size();
            L.first.uc_link = nullptr;
            makecontext(&L.first, entry, 0);
        }
    }
    const int r = _setjmp(back);
    if (r == 0) {
        w = l = 0;
        enter();
    }
    return r == 1 ? 0 : r;
}

struct Coord { unsigned x; };
inline Coord thread() { return {(unsigned)(w * 32 + l)}; }
template <class T>
inline const uint64_t *all(T v) {
    Warp &W = warp[w];
    const unsigned p = W.lane[l].parity++ & 1u;
    W.slot[p][l] = 0;
    std::memcpy(&W.slot[p][l], &v, sizeof(T));
    meet(0);
    return warp[w].slot[p];
}

}  // namespace fibers

#define threadIdx (fibers::thread())
#define blockIdx (fibers::Coord{0})
#define gridDim (fibers::Coord{1})
#define blockDim (fibers::Coord{(unsigned)fibers::warps * 32u})

inline void __syncwarp(unsigned = ~0u) { fibers::meet(0); }
inline void __syncthreads() { fibers::meet(1, true); }
inline unsigned __ballot_sync(unsigned, int p) {
    const uint64_t *v = fibers::all<unsigned>(p != 0);
    unsigned r = 0;
    for (int i = 0; i < 32; ++i) r |= (unsigned)v[i] << i;
    return r;
}
inline int __all_sync(unsigned m, int p) { return __ballot_sync(m, p) == ~0u; }
inline int __any_sync(unsigned m, int p) { return __ballot_sync(m, p) != 0; }
inline unsigned __reduce_add_sync(unsigned, unsigned x) {
    const uint64_t *v = fibers::all(x);
    unsigned r = 0;
    for (int i = 0; i < 32; ++i) r += (unsigned)v[i];
    return r;
}
inline unsigned __reduce_max_sync(unsigned, unsigned x) {
    const uint64_t *v = fibers::all(x);
    unsigned r = 0;
    for (int i = 0; i < 32; ++i) r = max(r, (unsigned)v[i]);
    return r;
}
template <class T>
inline T __shfl_sync(unsigned, T x, int from) {
    const uint64_t *v = fibers::all(x);
    T r;
    std::memcpy(&r, v + from, sizeof(T));
    return r;
}
inline unsigned __match_any_sync(unsigned, unsigned long long) { abort(); }   // (live launches only)
inline void __threadfence_block() {
    const bool slow = fibers::all<unsigned>(fibers::warp[fibers::w].slow)[0];
    if (fibers::l == 31) fibers::warp[fibers::w].slow = false;
    fibers::meet(slow ? fibers::slow_events : 1.0);
}
inline void __threadfence() {}
inline void __nanosleep(unsigned) { fibers::meet(0.1); }

template <class T, class U> inline T atomicAdd(T *p, U v) { T o = *p; *p = (T)(o + (T)v); return o; }
template <class T, class U> inline T atomicOr(T *p, U v) { T o = *p; *p = o | (T)v; return o; }
template <class T, class U> inline T atomicAnd(T *p, U v) { T o = *p; *p = o & (T)v; return o; }
template <class T, class U> inline T atomicMax(T *p, U v) { T o = *p; *p = max(o, (T)v); return o; }
template <class T> inline T __ldg(const T *p) { return *p; }
template <class T> inline T __ldcg(const T *p) { return *p; }
inline int __popc(unsigned v) { return __builtin_popcount(v); }
inline int __clz(int v) { return v ? __builtin_clz((unsigned)v) : 32; }
inline int __ffs(int v) { return __builtin_ffs(v); }
inline unsigned __umulhi(unsigned a, unsigned b) { return (unsigned)(((uint64_t)a * b) >> 32); }
inline uint64_t __umul64hi(uint64_t a, uint64_t b) { return (uint64_t)(((unsigned __int128)a * b) >> 64); }
inline unsigned __funnelshift_r(unsigned lo, unsigned hi, unsigned s) { return (unsigned)((((uint64_t)hi << 32) | lo) >> (s & 31)); }
inline unsigned __funnelshift_l(unsigned lo, unsigned hi, unsigned s) { return (unsigned)(((((uint64_t)hi << 32) | lo) << (s & 31)) >> 32); }
inline float __uint_as_float(unsigned u) { float f; std::memcpy(&f, &u, 4); return f; }
inline unsigned __float_as_uint(float f) { unsigned u; std::memcpy(&u, &f, 4); return u; }
inline float __logf(float x) { return std::log(x); }
inline float __fdividef(float a, float b) { return a / b; }
inline float __frcp_rn(float a) { return 1.0f / a; }
inline unsigned long long __float2ull_rn(float f) { return (unsigned long long)std::llrint(f); }
inline void sincospif(float x, float *s, float *c) {
    *s = (float)std::sin(M_PI * (double)x);
    *c = (float)std::cos(M_PI * (double)x);
    fibers::warp[fibers::w].slow = true;
}
