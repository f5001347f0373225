// Complex double-float arithmetic on packed float pairs (the FP64 grids' three-pass FFT).
//
// A complex value is {hi, lo}, each a pair of floats (real, imaginary) in one 64-bit register
// pair: value = hi + lo per component, about 48 significant bits (dfloat.cuh).  Every operation
// below acts on both components with one f32x2 instruction.  On GB300 these do no more
// additions a cycle than scalar ones (measured: 124.8 against 120.8 lanes a cycle and SM), but
// they take half the instructions: the transforms were bound by instruction fetch (see
// kernels_fft64.cu), and half the issue slots are left for loads and integers.
#pragma once

#include "dfloat.cuh"

namespace mbk {
namespace {

using f2 = unsigned long long;          // two floats: x in the low word, y in the high word

__device__ __forceinline__ f2 pk(float x, float y)
{
    f2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
    return r;
}
__device__ __forceinline__ void unpk(f2 a, float& x, float& y)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(a));
}
__device__ __forceinline__ f2 add2(f2 a, f2 b)
{
    f2 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f2 mul2(f2 a, f2 b)
{
    f2 d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c)
{
    f2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
constexpr f2 NEG1 = 0xBF800000BF800000ull, HALF2 = 0x3F0000003F000000ull;
__device__ __forceinline__ f2 sub2(f2 a, f2 b) { return fma2(b, NEG1, a); }     // exact product
// (x, y) -> (-y, x)
__device__ __forceinline__ f2 rot2(f2 a)
{
    float x, y;
    unpk(a, x, y);
    return pk(-y, x);
}
// (x, y) -> (x, -y)
__device__ __forceinline__ f2 conj2(f2 a)
{
    float x, y;
    unpk(a, x, y);
    return pk(x, -y);
}

struct __align__(16) dc {               // a complex double-float
    f2 hi, lo;
};

__device__ __forceinline__ dc dc_make(dfloat x, dfloat y) { return dc{pk(x.hi, y.hi), pk(x.lo, y.lo)}; }
__device__ __forceinline__ dfloat dc_x(dc a)
{
    float h, l, t;
    unpk(a.hi, h, t);
    unpk(a.lo, l, t);
    return dfloat(h, l);
}
__device__ __forceinline__ dfloat dc_y(dc a)
{
    float h, l, t;
    unpk(a.hi, t, h);
    unpk(a.lo, t, l);
    return dfloat(h, l);
}

// s + e = a + b with |a| >= |b| or nearly so
__device__ __forceinline__ dc renorm(f2 s, f2 e)
{
    const f2 h = add2(s, e);
    return dc{h, sub2(e, sub2(h, s))};
}
__device__ __forceinline__ dc cadd(dc a, dc b)
{
    const f2 s = add2(a.hi, b.hi), bb = sub2(s, a.hi);
    const f2 e = add2(sub2(a.hi, sub2(s, bb)), sub2(b.hi, bb));
    return renorm(s, add2(e, add2(a.lo, b.lo)));
}
__device__ __forceinline__ dc csub(dc a, dc b)
{
    const f2 s = sub2(a.hi, b.hi), bb = sub2(s, a.hi);
    const f2 e = sub2(sub2(a.hi, sub2(s, bb)), add2(b.hi, bb));
    return renorm(s, add2(e, sub2(a.lo, b.lo)));
}
__device__ __forceinline__ dc crot(dc a) { return dc{rot2(a.hi), rot2(a.lo)}; }      // i a
__device__ __forceinline__ dc cswap(dc a)                  // (x, y) -> (y, x)
{
    float x, y, u, v;
    unpk(a.hi, x, y);
    unpk(a.lo, u, v);
    return dc{pk(y, x), pk(v, u)};
}
__device__ __forceinline__ dc cconj(dc a) { return dc{conj2(a.hi), conj2(a.lo)}; }
__device__ __forceinline__ dc chalf(dc a) { return dc{mul2(a.hi, HALF2), mul2(a.lo, HALF2)}; }

// A double-float real in both components.
struct __align__(16) dr {
    f2 hi, lo;
};
__device__ __forceinline__ dr dr_make(dfloat a) { return dr{pk(a.hi, a.hi), pk(a.lo, a.lo)}; }

// a r: Dekker's product with the FMA residual
__device__ __forceinline__ dc cscale(dc a, dr r)
{
    const f2 p = mul2(a.hi, r.hi);
    f2 e = fma2(a.hi, r.hi, mul2(p, NEG1));
    e = fma2(a.hi, r.lo, e);
    e = fma2(a.lo, r.hi, e);
    return renorm(p, e);
}
// a (wr + i wi): two renormalised products and their sum (one TwoSum over the unnormalised
// products takes four instructions less, but loses 40% more: 0.70 against 0.51 x 2^-48 rms)
__device__ __forceinline__ dc cmul(dc a, dr wr, dr wi) { return cadd(cscale(a, wr), cscale(crot(a), wi)); }
// a conj(wr + i wi)
__device__ __forceinline__ dc cmulc(dc a, dr wr, dr wi)
{
    return cmul(a, wr, dr{mul2(wi.hi, NEG1), mul2(wi.lo, NEG1)});
}

}  // namespace
}  // namespace mbk
