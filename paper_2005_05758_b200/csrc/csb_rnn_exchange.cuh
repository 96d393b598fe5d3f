// Device pieces that the resident time loops share: the exchange of vectors between CTAs, asynchronous copies,
// the gates' activations.
#pragma once

#include "csb_internal.hpp"
#include "csb_device.cuh"

namespace csb {

#ifdef CSB_PHASE_CLOCKS
#define R1_LAP(i) do { if (tid == 0) { const long long n_ = clock64(); lap[i] += n_ - lap_at; lap_at = n_; } } while (0)
#else
#define R1_LAP(i) do { } while (0)
#endif

// (value, step) pairs, 8 bytes each: one store, one indivisible part of a 16-byte load.
__device__ __forceinline__ void st_one(uint2* p, float v, uint32_t tag) {
    const unsigned long long w = (unsigned long long)__float_as_uint(v) | ((unsigned long long)tag << 32);
    asm volatile("st.relaxed.gpu.global.b64 [%0], %1;" ::"l"(p), "l"(w) : "memory");
}
__device__ __forceinline__ uint4 ld_two(const uint2* p) {
    unsigned long long x, y;
    asm volatile("ld.relaxed.gpu.global.v2.b64 {%0, %1}, [%2];" : "=l"(x), "=l"(y) : "l"(p) : "memory");
    return make_uint4((uint32_t)x, (uint32_t)(x >> 32), (uint32_t)y, (uint32_t)(y >> 32));
}
__device__ __forceinline__ uint32_t ld_relaxed(const uint32_t* p) {
    uint32_t v;
    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void cp_async4(void* dst, const void* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
    unsigned long long d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;"
        : "=l"(d)
        : "l"(*reinterpret_cast<unsigned long long*>(&a)), "l"(*reinterpret_cast<unsigned long long*>(&b)), "l"(*reinterpret_cast<unsigned long long*>(&c)));
    return *reinterpret_cast<float2*>(&d);
}
__device__ __forceinline__ float2 half2_to_float2(uint32_t w) { return __half22float2(*reinterpret_cast<const __half2*>(&w)); }
// 1 / d for 1 <= d <= 2: the approximate reciprocal and one step of Newton's iteration r (2 - d r).
__device__ __forceinline__ float reciprocal(float d) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(d));
    return fmaf(r, fmaf(-d, r, 1.f), r);
}
// tanh (th) or the logistic function of x, without a branch: the gates of a unit sit on neighbouring lanes,
// and a divergent choice would run one after the other.  Both from e = exp(-|x|) (tanh: exp(-2 |x|)):
// 1 / (1 + e), e / (1 + e), (1 - e) / (1 + e).  Near zero 1 - e is left with e's error while the result shrinks, so
// there tanh is x + x^3 q(x^2), q the least-squares polynomial of degree 4 to (tanh(x) / x - 1) / x^2 at the Chebyshev
// nodes of 0 <= x^2 <= 25/64 (tests/test_activation.py fits it again).  5/8 is as far as degree 4 goes: its own error
// stays below 0.2 units in the last place there and is seven times that at 3/4.  Measured against float64, in units in the
// last place: tanh 0.83 up to 5/8, 2.1 above (3.7 where the exponential form is used from 1/2 on), logistic 3.5;
// tanhf has 1.8, 1 / (1 + expf(-x)) 3.1 where it does not flush to zero (x > -88).
__device__ __forceinline__ float activation(float x, bool th) {
    const float ax = fabsf(x), e = expf(th ? -2.f * ax : -ax), d = reciprocal(1.f + e), s = x * x;
    float q = fmaf(s, -0.006104947999119759f, 0.021003641188144684f);
    q = fmaf(s, q, -0.05385249853134155f);
    q = fmaf(s, q, 0.13332782685756683f);
    q = fmaf(s, q, -0.333333283662796f);
    const float t = ax < 0.625f ? fmaf(x * s, q, x) : copysignf((1.f - e) * d, x);
    const float l = x >= 0.f ? d : e * d;
    return x != x ? x : th ? t : l;
}
// The slow path of a wait: asks for two pairs again until both (two) are of step `want`.
static __device__ __noinline__ uint4 wait_two(const uint2* p, uint32_t want, bool two, volatile int* s_ok, uint32_t* status, unsigned long long limit_ns) {
    unsigned long long t0 = 0;
    unsigned int spins = 0;
    for (;;) {
        const uint4 w = ld_two(p);
        if ((w.y == want && (!two || w.w == want)) || *s_ok == 0) return w;   // *s_ok == 0: another thread has given up
        if ((++spins & 63u) == 0) {
            const unsigned long long now = global_ns();
            if (t0 == 0) t0 = now;
            else if (now - t0 > limit_ns) { *(volatile uint32_t*)status = (uint32_t)kDevBarrierTimeout; *s_ok = 0; return w; }
        }
    }
}
// The same for the progress of the layer above; false = gave up.
static __device__ __noinline__ bool wait_progress(const uint32_t* p, uint32_t from, uint32_t need, volatile int* s_ok, uint32_t* status, unsigned long long limit_ns) {
    unsigned long long t0 = 0;
    unsigned int spins = 0;
    while (ld_relaxed(p) - from < need) {
        if ((++spins & 63u) == 0) {
            const unsigned long long now = global_ns();
            if (t0 == 0) t0 = now;
            else if (now - t0 > limit_ns) { *(volatile uint32_t*)status = (uint32_t)kDevBarrierTimeout; *s_ok = 0; return false; }
        }
    }
    return true;
}

}  // namespace csb
