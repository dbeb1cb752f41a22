// Device arithmetic shared by the quantizer's kernels.
#pragma once
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <stdint.h>

namespace fp8attn {
namespace {

__device__ __forceinline__ uint4 ld_nc_v4(const uint4* p) {
    uint4 v;
    asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
}

// The two 16-bit input types: packed |x| / max for the reduction, and the exact
// fp32 value of the low and high half of a 32-bit word for the conversion.
template <bool kHalf> struct In16;
template <> struct In16<false> {
    using V2 = __nv_bfloat162;
    static __device__ __forceinline__ V2 as2(uint32_t u) { return *reinterpret_cast<V2*>(&u); }
    // an fp32 with the bf16 bits in its upper half is that value
    static __device__ __forceinline__ float lo(uint32_t w) { return __uint_as_float(w << 16); }
    static __device__ __forceinline__ float hi(uint32_t w) { return __uint_as_float(w & 0xffff0000u); }
    // negated (the addition flips the sign bit)
    static __device__ __forceinline__ float neg_lo(uint32_t w) { return __uint_as_float(w * 65536u + 0x80000000u); }
    static __device__ __forceinline__ float neg_hi(uint32_t w) { return __uint_as_float((w & 0xffff0000u) ^ 0x80000000u); }
};
template <> struct In16<true> {
    using V2 = __half2;
    static __device__ __forceinline__ V2 as2(uint32_t u) { return *reinterpret_cast<V2*>(&u); }
    static __device__ __forceinline__ float lo(uint32_t w) { return __low2float(as2(w)); }
    static __device__ __forceinline__ float hi(uint32_t w) { return __high2float(as2(w)); }
    static __device__ __forceinline__ float neg_lo(uint32_t w) { return -__low2float(as2(w)); }
    static __device__ __forceinline__ float neg_hi(uint32_t w) { return -__high2float(as2(w)); }
};

// max(m, |x|) over the eight 16-bit values of a vector, as a packed pair
template <bool kHalf>
__device__ __forceinline__ typename In16<kHalf>::V2 absmax8(typename In16<kHalf>::V2 m, const uint4& v) {
    using T = In16<kHalf>;
    return __hmax2(m, __hmax2(__hmax2(__habs2(T::as2(v.x)), __habs2(T::as2(v.y))),
                              __hmax2(__habs2(T::as2(v.z)), __habs2(T::as2(v.w)))));
}

// two floats -> two e4m3 codes (lo in bits 0..7, hi in bits 8..15), RNE, saturating
__device__ __forceinline__ uint32_t cvt_e4m3x2(float lo, float hi) {
    uint16_t r;
    asm("cvt.rn.satfinite.e4m3x2.f32 %0, %1, %2;" : "=h"(r) : "f"(hi), "f"(lo));
    return (uint32_t)r;
}

// scale of a head: amax / 448 by the IEEE division; 1 for an all-zero head
__device__ __forceinline__ float head_scale(float amax) { return amax == 0.0f ? 1.0f : __fdiv_rn(amax, 448.0f); }

// What a thread needs to divide by a head's scale.
struct Divisor {
    float s, r;      // scale; RN(1 / s)
    bool direct;     // outside the range in which the multiplications below are exact
};
__device__ __forceinline__ Divisor divisor(float s) {
    return Divisor{s, __frcp_rn(s), !(s >= 0x1p-60f && s <= 0x1p60f)};
}

// RN(x / s) of a pair without a division per element, by Markstein's correction (P. Markstein,
// "Computation of elementary functions on the IBM RISC System/6000 processor", 1990): with
// r = RN(1/s) and q0 = RN(x r), the remainder x - q0 s is exact in one fused multiply-add, and
// RN(q0 + remainder * r) is the correctly rounded quotient.  For the inputs here, whose
// mantissas have 8 or 11 bits, that holds for every pair of an input mantissa and an fp32 scale
// mantissa (checked exhaustively, 2^23 * 2^10 pairs); the scale range of `Divisor` keeps the
// remainder clear of the subnormal numbers wherever the code is not zero.  Written in y = -x, which
// costs nothing to unpack and keeps the sign of a zero: q0 = RN(y * -r), remainder' = q0 s + y,
// RN(remainder' * -r + q0).  (A table of the quotients of all mantissas in shared memory, one lookup
// per element, spent its time on bank conflicts: 654 MB in and out took 189 us, 182 us this way.)
template <bool kHalf, bool kClamp>
__device__ __forceinline__ uint32_t quant2(uint32_t w, uint64_t ss, uint64_t neg_rr, float lim) {
    float lo = In16<kHalf>::neg_lo(w), hi = In16<kHalf>::neg_hi(w);
    if (kClamp) {   // values far outside the scale's range: the quotient must not overflow
        lo = fminf(fmaxf(lo, -lim), lim);
        hi = fminf(fmaxf(hi, -lim), lim);
    }
    uint64_t y, q, e;
    asm("mov.b64 %0, {%1, %2};" : "=l"(y) : "f"(lo), "f"(hi));
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(q) : "l"(y), "l"(neg_rr));
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(e) : "l"(q), "l"(ss), "l"(y));
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(q) : "l"(e), "l"(neg_rr), "l"(q));
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(q));
    return cvt_e4m3x2(lo, hi);
}
// eight 16-bit values -> eight codes, by the IEEE division (for any scale) ...
template <bool kHalf>
__device__ __forceinline__ uint2 quant8_direct(const uint4& v, const Divisor& dv) {
    using T = In16<kHalf>;
    auto d2 = [&](uint32_t w) { return cvt_e4m3x2(__fdiv_rn(T::lo(w), dv.s), __fdiv_rn(T::hi(w), dv.s)); };
    return make_uint2(d2(v.x) | d2(v.y) << 16, d2(v.z) | d2(v.w) << 16);
}
// ... and for a scale in range (kClamp: values may lie outside the scale's range)
template <bool kHalf, bool kClamp>
__device__ __forceinline__ uint2 quant8(const uint4& v, const Divisor& dv) {
    uint64_t ss, neg_rr;
    asm("mov.b64 %0, {%1, %1};" : "=l"(ss) : "f"(dv.s));
    asm("mov.b64 %0, {%1, %1};" : "=l"(neg_rr) : "f"(-dv.r));
    const float lim = 512.0f * dv.s;
    auto q2 = [&](uint32_t w) { return quant2<kHalf, kClamp>(w, ss, neg_rr, lim); };
    return make_uint2(q2(v.x) | q2(v.y) << 16, q2(v.z) | q2(v.w) << 16);
}

}  // namespace
}  // namespace fp8attn
