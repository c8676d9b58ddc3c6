// Device primitives shared by the row kernels: packed fp32 arithmetic, shared-memory access by 32-bit address,
// bounded barrier waits, warp reductions.
#pragma once

#include <math.h>

#include "rdk_common.cuh"

namespace rdk {

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// ---- packed fp32 pairs ---------------------------------------------------------------------------
__device__ __forceinline__ float2 ffma2(float2 a, float2 b, float2 c) {
    float2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;"
        : "=l"(*reinterpret_cast<unsigned long long*>(&d))
        : "l"(*reinterpret_cast<unsigned long long*>(&a)), "l"(*reinterpret_cast<unsigned long long*>(&b)),
          "l"(*reinterpret_cast<unsigned long long*>(&c)));
    return d;
}
__device__ __forceinline__ float2 fadd2(float2 a, float2 b) {
    float2 d;
    asm("add.rn.f32x2 %0, %1, %2;"
        : "=l"(*reinterpret_cast<unsigned long long*>(&d))
        : "l"(*reinterpret_cast<unsigned long long*>(&a)), "l"(*reinterpret_cast<unsigned long long*>(&b)));
    return d;
}
__device__ __forceinline__ float2 fmul2(float2 a, float2 b) {
    float2 d;
    asm("mul.rn.f32x2 %0, %1, %2;"
        : "=l"(*reinterpret_cast<unsigned long long*>(&d))
        : "l"(*reinterpret_cast<unsigned long long*>(&a)), "l"(*reinterpret_cast<unsigned long long*>(&b)));
    return d;
}
__device__ __forceinline__ float2 splat(float v) { return make_float2(v, v); }
__device__ __forceinline__ float2 ex2_2(float2 x) { return make_float2(ex2(x.x), ex2(x.y)); }

// ---- shared-memory access by 32-bit shared address -----------------------------------------------
__device__ __forceinline__ uint4 lds128(uint32_t a) {
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a));
    return v;
}
__device__ __forceinline__ uint2 lds64(uint32_t a) {
    uint2 v;
    asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(a));
    return v;
}
__device__ __forceinline__ uint32_t lds32(uint32_t a) {
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(a));
    return v;
}
__device__ __forceinline__ uint32_t lds16(uint32_t a) {
    uint16_t v;
    asm volatile("ld.shared.u16 %0, [%1];" : "=h"(v) : "r"(a));
    return v;
}
__device__ __forceinline__ void sts128(uint32_t a, float x, float y, float z, float w) {
    asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(a), "f"(x), "f"(y), "f"(z), "f"(w) : "memory");
}
__device__ __forceinline__ void sts32(uint32_t a, uint32_t v) {
    asm volatile("st.shared.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}

// one target logit at shared byte address a, as fp32
template <typename TZ> __device__ __forceinline__ float lds_z(uint32_t a);
template <> __device__ __forceinline__ float lds_z<__nv_bfloat16>(uint32_t a) { return __uint_as_float(lds16(a) << 16); }
template <> __device__ __forceinline__ float lds_z<float>(uint32_t a) { return __uint_as_float(lds32(a)); }

// two consecutive drafter values at shared byte address a (aligned to the pair), as fp32
template <typename TY> __device__ __forceinline__ float2 lds_ypair(uint32_t a);
template <> __device__ __forceinline__ float2 lds_ypair<__nv_bfloat16>(uint32_t a) {
    const uint32_t w = lds32(a);
    return make_float2(bf16_lo(w), bf16_hi(w));
}
template <> __device__ __forceinline__ float2 lds_ypair<float>(uint32_t a) {
    const uint2 w = lds64(a);
    return make_float2(__uint_as_float(w.x), __uint_as_float(w.y));
}

// maximum of the 8 logits (bf16) / 4 logits (fp32) in one 16-byte vector
template <typename TZ> struct MaxAcc;
template <> struct MaxAcc<float> {
    float m = -INFINITY;
    __device__ __forceinline__ void push(uint4 q) {
        m = fmaxf(fmaxf(m, __uint_as_float(q.x)), fmaxf(__uint_as_float(q.y), fmaxf(__uint_as_float(q.z), __uint_as_float(q.w))));
    }
    __device__ __forceinline__ float result() const { return m; }
};
template <> struct MaxAcc<__nv_bfloat16> {
    __nv_bfloat162 ma = __float2bfloat162_rn(-INFINITY), mb = __float2bfloat162_rn(-INFINITY);
    __device__ __forceinline__ void push(uint4 q) {
        ma = __hmax2(ma, *reinterpret_cast<const __nv_bfloat162*>(&q.x));
        mb = __hmax2(mb, *reinterpret_cast<const __nv_bfloat162*>(&q.y));
        ma = __hmax2(ma, *reinterpret_cast<const __nv_bfloat162*>(&q.z));
        mb = __hmax2(mb, *reinterpret_cast<const __nv_bfloat162*>(&q.w));
    }
    __device__ __forceinline__ float result() const {
        const __nv_bfloat162 m2 = __hmax2(ma, mb);
        return fmaxf(__low2float(m2), __high2float(m2));
    }
};

// sum of e = 2^(z log2e + off) over the logits of one 16-byte vector, two packed accumulators.  (Evaluating a
// share of the exponentials by a polynomial on the FMA pipe relieves the special-function unit but costs issue
// slots, which are the scarcer resource in this kernel: measured, it does not pay.)
template <typename TZ> __device__ __forceinline__ void exp_sum_vec(uint4 q, float2 scale, float2 off, float2& Ea, float2& Eb);
template <> __device__ __forceinline__ void exp_sum_vec<__nv_bfloat16>(uint4 q, float2 scale, float2 off, float2& Ea, float2& Eb) {
    const float2 e0 = ex2_2(ffma2(make_float2(bf16_lo(q.x), bf16_hi(q.x)), scale, off));
    const float2 e1 = ex2_2(ffma2(make_float2(bf16_lo(q.y), bf16_hi(q.y)), scale, off));
    const float2 e2 = ex2_2(ffma2(make_float2(bf16_lo(q.z), bf16_hi(q.z)), scale, off));
    const float2 e3 = ex2_2(ffma2(make_float2(bf16_lo(q.w), bf16_hi(q.w)), scale, off));
    Ea = fadd2(Ea, e0); Eb = fadd2(Eb, e1); Ea = fadd2(Ea, e2); Eb = fadd2(Eb, e3);
}
template <> __device__ __forceinline__ void exp_sum_vec<float>(uint4 q, float2 scale, float2 off, float2& Ea, float2& Eb) {
    const float2 e0 = ex2_2(ffma2(make_float2(__uint_as_float(q.x), __uint_as_float(q.y)), scale, off));
    const float2 e1 = ex2_2(ffma2(make_float2(__uint_as_float(q.z), __uint_as_float(q.w)), scale, off));
    Ea = fadd2(Ea, e0); Eb = fadd2(Eb, e1);
}

// Wait for the phase of `bar` with the given parity.  Each try may park the warp in hardware for up to
// HINT_NS nanoseconds (it wakes as soon as the phase completes), so a waiting warp issues next to nothing;
// after `limit` failed tries the wait gives up and the host reads RDK_ERR_TIMEOUT.
template <int HINT_NS = 2000>
__device__ __forceinline__ void mbar_wait(uint32_t bar, uint32_t parity, int* fail, unsigned limit) {
    unsigned spins = 0;
    uint32_t done = 0;
    while (!done) {
        asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n selp.u32 %0, 1, 0, p;\n}"
                     : "=r"(done) : "r"(bar), "r"(parity), "r"((uint32_t)HINT_NS) : "memory");
        if (!done && (++spins > limit || *reinterpret_cast<volatile int*>(fail))) {
            atomicExch(fail, 1);
            break;
        }
    }
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.release.cta.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

// (value, tag) words in global memory: one 64-bit relaxed access each, so a reader sees a value
// together with the tag that was stored with it
__device__ __forceinline__ void st_tagged(unsigned char* p, float v, uint32_t tag) {
    const unsigned long long w = ((unsigned long long)tag << 32) | (unsigned long long)__float_as_uint(v);
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(w) : "memory");
}
__device__ __forceinline__ unsigned long long ld_tagged(const unsigned char* p) {
    unsigned long long w;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(w) : "l"(p) : "memory");
    return w;
}
__device__ __forceinline__ int ld_volatile_s32(const int* p) {
    int v;
    asm volatile("ld.volatile.shared.s32 %0, [%1];" : "=r"(v) : "r"(smem_u32(p)) : "memory");
    return v;
}

// Sums of four per-lane values over the warp with 6 shuffles: afterwards lanes 0-7 hold the total of
// v0, lanes 8-15 of v1, lanes 16-23 of v2, lanes 24-31 of v3.
__device__ __forceinline__ float warp_sum4(float v0, float v1, float v2, float v3, int lane) {
    const bool up = lane & 16;
    float a = up ? v2 : v0, b = up ? v3 : v1;
    a += __shfl_xor_sync(0xffffffffu, up ? v0 : v2, 16);
    b += __shfl_xor_sync(0xffffffffu, up ? v1 : v3, 16);
    const bool odd = lane & 8;
    float k = odd ? b : a;
    k += __shfl_xor_sync(0xffffffffu, odd ? a : b, 8);
    k += __shfl_xor_sync(0xffffffffu, k, 4);
    k += __shfl_xor_sync(0xffffffffu, k, 2);
    k += __shfl_xor_sync(0xffffffffu, k, 1);
    return k;
}
__device__ __forceinline__ float warp_max_redux(float v) {
    float m;
    asm volatile("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(m) : "f"(v));
    return m;
}

// Combine per-lane partial soft-max records (sum e, sum e_y, sum e e_y on the scales m, my) over
// the warp; lanes without a record pass m = my = -inf and zeros.
__device__ __forceinline__ void combine_records(float& E1, float& Zq, float& th, float& m, float& my, int lane) {
    const float mm = warp_max_redux(m), mmy = warp_max_redux(my);
    const float f = m > -INFINITY ? ex2((m - mm) * kLog2e) : 0.f;
    const float g = my > -INFINITY ? ex2((my - mmy) * kLog2e) : 0.f;
    const float tot = warp_sum4(E1 * f, Zq * g, th * f * g, 0.f, lane);
    E1 = __shfl_sync(0xffffffffu, tot, 0); Zq = __shfl_sync(0xffffffffu, tot, 8); th = __shfl_sync(0xffffffffu, tot, 16);
    m = mm; my = mmy;
}

// The same on scales 2^m and 2^my, with th on that of Zq alone (e_pi, which it has in place of e_z, is on one scale in all
// records); x is summed up as it is.
__device__ __forceinline__ void combine_records_prior(float& E1, float& Zq, float& th, float& m, float& my, float& x, int lane) {
    const float mm = warp_max_redux(m), mmy = warp_max_redux(my);
    const float f = m > -INFINITY ? ex2(m - mm) : 0.f;
    const float g = my > -INFINITY ? ex2(my - mmy) : 0.f;
    const float tot = warp_sum4(E1 * f, Zq * g, th * g, x, lane);
    E1 = __shfl_sync(0xffffffffu, tot, 0); Zq = __shfl_sync(0xffffffffu, tot, 8); th = __shfl_sync(0xffffffffu, tot, 16); x = __shfl_sync(0xffffffffu, tot, 24);
    m = mm; my = mmy;
}

}  // namespace rdk
