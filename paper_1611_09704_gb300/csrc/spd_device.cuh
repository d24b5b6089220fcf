// spd_device.cuh -- device helpers shared by the detect kernels: packed
// (SNR, code) floats, packed f32x2 arithmetic, 1-D bulk (TMA) copies with a
// time-bounded mbarrier wait, and vector loads of stored samples.
#pragma once
#include "spd_internal.cuh"

#include <math.h>

namespace spd {

namespace {

constexpr int kWaitLimit = 1 << 22;          // polls, a backstop to the time bound
constexpr uint32_t kSuspendNs = 20000;       // suspend hint of one poll

__device__ __forceinline__ float packw(float s, uint32_t code) {
    return __uint_as_float((__float_as_uint(s) & 0xFFFFFFC0u) | code);
}
__device__ __forceinline__ float trunc17(float s) {
    return __uint_as_float(__float_as_uint(s) & 0xFFFFFFC0u);
}

__device__ __forceinline__ float fmax3(float a, float b, float c) {
    float r;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}

__device__ __forceinline__ float fmin3(float a, float b, float c) {
    float r;
    asm("min.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}

// The larger of two, NaN when either is.
__device__ __forceinline__ float fmax_nan(float a, float b) {
    float r;
    asm("max.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
    return r;
}

__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }

// ------------------------------------------------------------- bulk copies

__device__ __forceinline__ uint32_t saddr(const void *p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void mbar_init(uint64_t *bar) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(saddr(bar)) : "memory");
}
// Its words become ordinary shared memory again.
__device__ __forceinline__ void mbar_inval(uint64_t *bar) {
    asm volatile("mbarrier.inval.shared::cta.b64 [%0];" ::"r"(saddr(bar)) : "memory");
}
__device__ __forceinline__ void fence_mbar_init() {
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void fence_proxy_async() {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
// One arrival that also expects `bytes` of bulk-copy completion.
__device__ __forceinline__ void mbar_expect(uint64_t *bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(saddr(bar)),
                 "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void bulk_load(void *dst, const void *src, uint32_t bytes,
                                          uint64_t *bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
        ::"r"(saddr(dst)), "l"(src), "r"(bytes), "r"(saddr(bar))
        : "memory");
}
// One poll; the thread may be suspended (up to kSuspendNs) until the phase
// completes instead of spinning on issue slots.
__device__ __forceinline__ bool mbar_test(uint64_t *bar, uint32_t phase) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n"
        " selp.u32 %0, 1, 0, p;\n}"
        : "=r"(ok)
        : "r"(saddr(bar)), "r"(phase), "r"(kSuspendNs)
        : "memory");
    return ok != 0;
}
__device__ __forceinline__ uint64_t global_ns() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
// Bounded wait for a phase of `bar`: false if it did not complete within
// limit_ns of wall time (or kWaitLimit polls).
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t phase, uint64_t limit_ns) {
    if (mbar_test(bar, phase)) return true;
    const uint64_t t0 = global_ns();
    for (int it = 0; it < kWaitLimit; ++it) {
        if (mbar_test(bar, phase)) return true;
        if (global_ns() - t0 > limit_ns) return false;
    }
    return false;
}

template <int DT>
__device__ __forceinline__ void load4v(const typename Elem<DT>::T *p, float &a, float &b,
                                       float &c, float &d);
template <>
__device__ __forceinline__ void load4v<SPD_F32>(const float *p, float &a, float &b, float &c,
                                                float &d) {
    const float4 v = *reinterpret_cast<const float4 *>(p);
    a = v.x; b = v.y; c = v.z; d = v.w;
}
template <>
__device__ __forceinline__ void load4v<SPD_F16>(const __half *p, float &a, float &b, float &c,
                                                float &d) {
    const uint2 v = *reinterpret_cast<const uint2 *>(p);
    const float2 lo = __half22float2(*reinterpret_cast<const __half2 *>(&v.x));
    const float2 hi = __half22float2(*reinterpret_cast<const __half2 *>(&v.y));
    a = lo.x; b = lo.y; c = hi.x; d = hi.y;
}
template <>
__device__ __forceinline__ void load4v<SPD_BF16>(const __nv_bfloat16 *p, float &a, float &b,
                                                 float &c, float &d) {
    const uint2 v = *reinterpret_cast<const uint2 *>(p);
    const float2 lo = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&v.x));
    const float2 hi = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&v.y));
    a = lo.x; b = lo.y; c = hi.x; d = hi.y;
}

// ------------------------------------------------ positions of a window

// Word of position p: 16 positions take kSPad words.
__device__ __forceinline__ int sadr(int p) { return (p & 15) + kSPad * (p >> 4); }

// Centred values y = (x - mu.hi) - mu.lo of window positions p .. p+N-1
// (x = fmaf(scale, q, offset) for scaled storage), -inf at and past `have`.
// Elements below nraw come from the raw staging buffer, the rest of the row
// from global memory.
template <int DT, int N>
__device__ __forceinline__ void load_centred(float *v, const typename Elem<DT>::T *raw,
                                             const typename Elem<DT>::T *gsrc, int p, int nraw,
                                             int have, bool has_sc, float sc, float of, float2 mu) {
    const float2 mh = make_float2(-mu.x, -mu.x), ml = make_float2(-mu.y, -mu.y);
    if (p + N <= nraw) {
#pragma unroll
        for (int u = 0; u < N / 4; ++u) {
            float a, b, c, d;
            load4v<DT>(raw + p + 4 * u, a, b, c, d);
            float2 x0 = make_float2(a, b), x1 = make_float2(c, d);
            if (has_sc) {
                const float2 s2 = make_float2(sc, sc), o2 = make_float2(of, of);
                x0 = fma2(s2, x0, o2);
                x1 = fma2(s2, x1, o2);
            }
            x0 = add2(add2(x0, mh), ml);
            x1 = add2(add2(x1, mh), ml);
            v[4 * u] = x0.x; v[4 * u + 1] = x0.y; v[4 * u + 2] = x1.x; v[4 * u + 3] = x1.y;
        }
    } else {
#pragma unroll
        for (int e = 0; e < N; ++e) {
            const int q = p + e;
            float x = 0.f;
            if (q < nraw) x = Elem<DT>::cvt(raw[q]);
            else if (q < have) x = Elem<DT>::cvt(gsrc[q]);
            if (has_sc) x = fmaf(sc, x, of);
            x = __fsub_rn(__fsub_rn(x, mu.x), mu.y);
            v[e] = q < have ? x : -INFINITY;
        }
    }
}

}  // namespace

}  // namespace spd
