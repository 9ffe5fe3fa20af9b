// Arithmetic on unevaluated pairs of floats (about 47 significant bits), and
// conversions between float64, float32 and such pairs on the integer units.
//
// GB300 executes a warp-wide float64 instruction in 64 cycles of a scheduler's
// FP64 unit, whatever it is: a fused multiply-add, a compare, a floor or a
// conversion to or from float32 (measured; 0.5 lanes a clock).  A pair
// addition is 11 float32 instructions, a product 6, a conversion 7 to 15
// integer ones, each a cycle: the refined form uses them where it needs more
// than float32 but where the last bits of a float64 do not show (its momenta,
// weights and moments are float32).
//
// Additions and products: Dekker, Numer. Math. 18 (1971) 224; the exact sum of
// two floats: Knuth, TAOCP vol. 2, 4.2.2.
#pragma once

#include <cuda_runtime.h>

namespace qsff {

struct Ff {
    float h, l;
    __host__ __device__ Ff() {}
    __host__ __device__ constexpr Ff(float h_, float l_) : h(h_), l(l_) {}
    // compile-time constants and host tables
    __host__ __device__ explicit constexpr Ff(double v) : h((float)v), l((float)(v - (double)(float)v)) {}
    __host__ __device__ explicit constexpr Ff(float v) : h(v), l(0.f) {}
    __host__ __device__ explicit constexpr Ff(int v) : h((float)v), l(0.f) {}
};

// the intrinsics keep the compiler from fusing a product into a sum that is
// meant to be of its rounded value
__device__ __forceinline__ Ff quick(float a, float b) {  // |a| >= |b| or a == 0
    const float s = __fadd_rn(a, b);
    return Ff(s, __fsub_rn(b, __fsub_rn(s, a)));
}
__device__ __forceinline__ Ff two_sum(float a, float b) {
    const float s = __fadd_rn(a, b), v = __fsub_rn(s, a);
    return Ff(s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, v)), __fsub_rn(b, v)));
}
__device__ __forceinline__ Ff two_prod(float a, float b) {
    const float p = __fmul_rn(a, b);
    return Ff(p, __fmaf_rn(a, b, -p));
}
__device__ __forceinline__ Ff operator+(Ff a, Ff b) {
    const Ff s = two_sum(a.h, b.h);
    return quick(s.h, __fadd_rn(s.l, __fadd_rn(a.l, b.l)));
}
__device__ __forceinline__ Ff operator-(Ff a) { return Ff(-a.h, -a.l); }
__device__ __forceinline__ Ff operator-(Ff a, Ff b) { return a + (-b); }
__device__ __forceinline__ Ff operator*(Ff a, Ff b) {
    const Ff p = two_prod(a.h, b.h);
    return quick(p.h, __fmaf_rn(a.h, b.l, __fmaf_rn(a.l, b.h, p.l)));
}
__device__ __forceinline__ Ff operator*(Ff a, float b) {
    const Ff p = two_prod(a.h, b);
    return quick(p.h, __fmaf_rn(a.l, b, p.l));
}
__device__ __forceinline__ Ff &operator+=(Ff &a, Ff b) { return a = a + b; }
__device__ __forceinline__ Ff &operator-=(Ff &a, Ff b) { return a = a - b; }

// 1 / d: one Newton step from the float32 reciprocal, the residual in pairs
__device__ __forceinline__ Ff recip(Ff d) {
    const float r = __frcp_rn(d.h);
    const Ff p = two_prod(d.h, r);
    // 1 - d r, small: its float32 value is enough
    const float e = __fsub_rn(__fsub_rn(__fsub_rn(1.f, p.h), p.l), __fmul_rn(d.l, r));
    return quick(r, __fmul_rn(r, __fmaf_rn(e, e, e)));
}

// (double)f, exact
__device__ __forceinline__ double widen(float f) {
    const unsigned u = __float_as_uint(f), m = u & 0x7fffffffu;
    if (m - 0x00800000u >= 0x7f000000u && m != 0u) return (double)f;  // denormal, inf, NaN
    const unsigned hi = m ? (m >> 3) + 0x38000000u : 0u;
    return __hiloint2double((int)(hi | (u & 0x80000000u)), (int)(u << 29));
}

// v as a pair: h is (float)v, h + l agrees with v to 2^-48
__device__ __forceinline__ Ff split(double v) {
    const unsigned hi = (unsigned)__double2hiint(v), lo = (unsigned)__double2loint(v);
    const int e = (int)((hi >> 20) & 0x7ffu) - 1023;
    if ((unsigned)(e + 70) >= 190u) {  // zero, or beyond what the pair's parts cover
        const float h = (float)v;
        return Ff(h, isfinite(h) ? (float)(v - (double)h) : 0.f);
    }
    const unsigned s = hi & 0x80000000u;
    const float t = __uint_as_float(s | ((unsigned)(e + 127) << 23) | ((hi & 0xfffffu) << 3) | (lo >> 29));
    const float r = (float)(lo & 0x1fffffffu);
    const float w = __uint_as_float(s | ((unsigned)(e + 75) << 23));  // 2^(e - 52), signed
    return quick(t, __fmul_rn(r, w));
}

// the pair as a float64: one FP64 addition
__device__ __forceinline__ double join(Ff a) { return widen(a.h) + widen(a.l); }

}  // namespace qsff
