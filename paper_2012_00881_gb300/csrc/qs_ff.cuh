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
    if ((unsigned)(e + 70) >= 190u) {
        if (((hi << 1) | lo) == 0u) return Ff(0.f, 0.f);
        // beyond what the pair's parts cover
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

// Integer part and fraction (as a pair) of 1/2 <= t < 4096 from its bits: a floor,
// a conversion and a difference would be three FP64-pipe instructions.  With
// t = s + 1/2 for a position s in cells, `cell` is the right one of the two
// cell centres around it and f its linear weight.
struct AxisBits {
    int cell;
    Ff f;
};
__device__ __forceinline__ AxisBits axis_bits(double t) {
    const unsigned hi = (unsigned)__double2hiint(t), lo = (unsigned)__double2loint(t);
    const int e = (int)(hi >> 20) - 1023;
    AxisBits b;
    if ((unsigned)(e + 1) > 12u) {  // outside the box (negative, or far beyond it)
        const double fl = floor(t);
        b.cell = (int)fl;
        b.f = split(t - fl);
        return b;
    }
    const unsigned mh = (hi & 0xfffffu) | 0x100000u;
    b.cell = (int)(mh >> (20 - e));
    // the fraction as 64 bits: shift the integer part out at the top
    const int sh = 12 + e;
    const unsigned fh = __funnelshift_l(lo, mh, sh), fl = lo << sh;
    const float h = (float)(fh & 0xffffff00u);
    const float l = (float)((fh << 24) | (fl >> 8));
    b.f = quick(h * 0x1p-32f, l * 0x1p-56f);
    return b;
}

// square root of a > 0: one Newton step from float32
__device__ __forceinline__ Ff sqrt_pair(Ff a) {
    const float r = rsqrtf(a.h), y = __fmul_rn(a.h, r);
    const Ff y2 = two_prod(y, y);
    const float e = __fadd_rn(__fsub_rn(__fsub_rn(a.h, y2.h), y2.l), a.l);  // a - y^2
    return quick(y, __fmul_rn(__fmul_rn(e, 0.5f), r));
}

// sine and cosine of |r| <= pi / 4 by their Taylor series: pairs for the terms
// above 2^-24 of the sum, float32 for the rest (truncated below 2^-52)
__device__ __forceinline__ void sincos_pair(Ff r, Ff &s, Ff &c) {
    constexpr double f3 = 6, f4 = 24, f5 = 120, f6 = 720, f7 = 5040, f8 = 40320, f9 = 362880,
                     f10 = 3628800, f11 = 39916800, f12 = 479001600, f13 = 6227020800,
                     f14 = 87178291200, f15 = 1307674368000, f16 = 20922789888000;
    const Ff z = r * r;
    const float zf = z.h;
    const float st = fmaf(zf, fmaf(zf, (float)(-1 / f15), (float)(1 / f13)), (float)(-1 / f11));
    const float ct = fmaf(zf, fmaf(zf, (float)(1 / f16), (float)(-1 / f14)), (float)(1 / f12));
    Ff p = Ff(1 / f9) + Ff(zf * st, 0.f);
    p = Ff(-1 / f7) + z * p;
    p = Ff(1 / f5) + z * p;
    p = Ff(-1 / f3) + z * p;
    s = r + (r * z) * p;
    Ff q = Ff(-1 / f10) + Ff(zf * ct, 0.f);
    q = Ff(1 / f8) + z * q;
    q = Ff(-1 / f6) + z * q;
    q = Ff(1 / f4) + z * q;
    q = Ff(-0.5) + z * q;
    c = Ff(1.f, 0.f) + z * q;
}

}  // namespace qsff
