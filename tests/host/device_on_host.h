// Compiles the element operator's device headers for the host: the CUDA
// qualifiers expand to nothing, the intrinsics used by the headers are restated
// in plain C++, and a CTA's threads are host threads with a barrier.  The code
// under test is the headers' own.
#pragma once

#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>
#include <string.h>

#include <algorithm>
#include <barrier>
#include <functional>
#include <memory>
#include <mutex>
#include <thread>
#include <vector>

namespace host {
inline thread_local uint3 tid{0, 0, 0};
inline uint3 bid{0, 0, 0};
inline dim3 bdim(1), gdim(1);
inline std::unique_ptr<std::barrier<>> bar;
inline std::vector<std::unique_ptr<std::barrier<>>> wbar;   // one per warp
inline std::vector<unsigned> lane;                          // a value per thread
inline std::mutex mu;

// Loads through __ldcs outside [lo, hi) are counted and answered with zeros.
inline const char *lo = nullptr, *hi = nullptr;
inline long outside = 0;

// One CTA of `threads` threads.
inline void cta(int threads, const std::function<void()> &body) {
    bdim = dim3(threads);
    bar = std::make_unique<std::barrier<>>(threads);
    wbar.clear();
    for (int w = 0; w < threads; w += 32) wbar.push_back(std::make_unique<std::barrier<>>(std::min(32, threads - w)));
    lane.assign(threads, 0u);
    std::vector<std::thread> th;
    for (int t = 0; t < threads; t++)
        th.emplace_back([&, t] {
            tid.x = (unsigned)t;
            body();
        });
    for (auto &x : th) x.join();
}
}  // namespace host

#undef __noinline__
#define __noinline__
#undef __shared__
#define __shared__ static
#define threadIdx (::host::tid)
#define blockIdx (::host::bid)
#define blockDim (::host::bdim)
#define gridDim (::host::gdim)

template <typename A, typename B>
inline A bits_as(B b) {
    static_assert(sizeof(A) == sizeof(B), "");
    A a;
    memcpy(&a, &b, sizeof a);
    return a;
}
inline float __int_as_float(int x) { return bits_as<float>(x); }
inline int __float_as_int(float x) { return bits_as<int>(x); }
inline float __uint_as_float(unsigned x) { return bits_as<float>(x); }
inline unsigned __float_as_uint(float x) { return bits_as<unsigned>(x); }
inline double __longlong_as_double(long long x) { return bits_as<double>(x); }
inline long long __double_as_longlong(double x) { return bits_as<long long>(x); }
inline int __double2hiint(double x) { return (int)(bits_as<unsigned long long>(x) >> 32); }
inline float __double2float_rn(double x) { return (float)x; }
inline long long __float2ll_rn(float x) { return llrintf(x); }
inline float __fadd_rn(float a, float b) { return a + b; }
inline float __fsub_rn(float a, float b) { return a - b; }
inline float __fmul_rn(float a, float b) { return a * b; }
inline float __fmaf_rn(float a, float b, float c) { return fmaf(a, b, c); }
inline double __dadd_rn(double a, double b) { return a + b; }
inline int __popc(unsigned x) { return __builtin_popcount(x); }
inline int __clzll(long long x) { return x ? __builtin_clzll((unsigned long long)x) : 64; }
inline unsigned long long __umul64hi(unsigned long long a, unsigned long long b) {
    return (unsigned long long)(((unsigned __int128)a * b) >> 64);
}
template <typename T>
inline T __ldcs(const T *p) {
    if (host::lo && ((const char *)p < host::lo || (const char *)(p + 1) > host::hi)) {
        std::lock_guard<std::mutex> g(host::mu);
        host::outside++;
        return T{};
    }
    return *p;
}
template <typename T>
inline T __ldg(const T *p) { return *p; }
template <typename T>
inline T __ldcg(const T *p) { return *p; }
template <typename T>
inline void __stcs(T *p, T v) { *p = v; }
inline void __syncthreads() { host::bar->arrive_and_wait(); }
template <typename T>
inline T atomicAdd(T *p, T v) {
    std::lock_guard<std::mutex> g(host::mu);
    const T o = *p;
    *p = o + v;
    return o;
}
template <typename T>
inline T atomicMax(T *p, T v) {
    std::lock_guard<std::mutex> g(host::mu);
    const T o = *p;
    *p = std::max(o, v);
    return o;
}
template <typename T>
inline T atomicExch(T *p, T v) {
    std::lock_guard<std::mutex> g(host::mu);
    const T o = *p;
    *p = v;
    return o;
}
template <typename T>
inline T atomicOr(T *p, T v) {
    std::lock_guard<std::mutex> g(host::mu);
    const T o = *p;
    *p = o | v;
    return o;
}
inline unsigned __reduce_max_sync(unsigned, unsigned v) {   // all 32 lanes
    const unsigned w = host::tid.x / 32, end = std::min<unsigned>(host::lane.size(), 32 * (w + 1));
    host::lane[host::tid.x] = v;
    host::wbar[w]->arrive_and_wait();
    unsigned m = 0;
    for (unsigned t = 32 * w; t < end; t++) m = std::max(m, host::lane[t]);
    host::wbar[w]->arrive_and_wait();
    return m;
}
inline int __reduce_max_sync(unsigned mask, int v) { return (int)__reduce_max_sync(mask, (unsigned)v); }   // v >= 0
// Declared for the headers' other functions; nothing here calls it.
template <typename T>
T __shfl_down_sync(unsigned, T, int);
inline void __threadfence() {}
