// Three-point Peskin kernel weights for the blob-grid coupling (Eq. delta).
#pragma once

#include <cuda_runtime.h>

namespace mbk {

// 1/sqrt(a) to about 2^-22, for 2^-126 <= a < 2^127: the hardware's float reciprocal square
// root between two moves of the exponent field (integer instructions, no FP64 conversion).
__device__ __forceinline__ double rsqrt_seed(double a)
{
    const unsigned hi = (unsigned)__double2hiint(a), lo = (unsigned)__double2loint(a);
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;"
        : "=f"(y) : "f"(__uint_as_float(((hi - (896u << 20)) << 3) | (lo >> 29))));
    const unsigned yb = __float_as_uint(y);
    return __hiloint2double((int)((yb >> 3) + (896u << 20)), (int)(yb << 29));
}

// s = sqrt(a) and h = 1/(2 sqrt(a)) by Goldschmidt's iteration (one step from the 22-bit seed,
// then s corrected by its residual a - s^2, exact in an FMA).  h is good to 2^-43 and s before
// its rounding to 2^-86: s is the correctly rounded root but for one argument in about 2^33.
__device__ __forceinline__ void sqrt_half_inverse(double a, double& s, double& h)
{
    const double y = rsqrt_seed(a);
    const double h0 = __hiloint2double(__double2hiint(y) - (1 << 20), __double2loint(y));  // y/2
    const double g = a * y;
    const double r = fma(-g, h0, 0.5);
    const double g1 = fma(g, r, g);
    h = fma(h0, r, h0);
    s = fma(fma(-g1, g1, a), h, g1);
}
// x / d from an approximate reciprocal of d (2^-43): rounded like sqrt_half_inverse's root.
__device__ __forceinline__ double quotient(double x, double d, double inv_d)
{
    const double q = x * inv_d;
    return fma(fma(-q, d, x), inv_d, q);
}
// sqrt_half_inverse and quotient need 2^-126 <= a < 2^127 (a squared distance, say)
__device__ __forceinline__ bool in_seed_range(double a)
{
    return (unsigned)__double2hiint(a) - (897u << 20) < (253u << 20);
}

__device__ __forceinline__ float peskin_sqrt(float a) { return sqrtf(a); }
__device__ __forceinline__ double peskin_sqrt(double a)      // 1/4 <= a <= 1
{
    double s, h;
    sqrt_half_inverse(a, s, h);
    return s;
}

// For a blob at fractional node coordinate x (x = q/h - shift, shift = 0 along the component's
// own axis and 1/2 across it on the MAC grid), the only nodes with non-zero weight are the
// nearest node i0 = floor(x + 1/2) and its two neighbours.  With t = x - i0 in [-1/2, 1/2) and
// s = sqrt(1 - 3 t^2), the Roma-Peskin-Berger function gives
//   Phi at i0 - 1 = (2 - 3t - s)/6,  Phi at i0 = (1 + s)/3,  Phi at i0 + 1 = (2 + 3t - s)/6,
// which sum to 1, have zero first moment and squares summing to 1/2 for every t.
// The offset is taken in FP64 (positions are FP64); the weights in R.
// Returns i0 - 1, the index of the first node of the window.
//
// GB300 issues two FP64 lanes a cycle and SM, so the windows are written for few FP64
// instructions (about 24 with floor, conversion and the library's root): the nearest node by adding and removing 1.5 * 2^52
// (its index is then the low word of the sum: no conversion; an exact tie may take either
// node, which gives the same three weights), and the square root by Goldschmidt's iteration.
template <typename R>
__device__ __forceinline__ int peskin_window(double x, R w[3])
{
    const double big = x + 6755399441055744.0;
    const R t = static_cast<R>(x - (big - 6755399441055744.0));
    const R s = peskin_sqrt(R(1) - R(3) * t * t);
    w[0] = (R(2) - R(3) * t - s) * R(1.0 / 6.0);
    w[1] = (R(1) + s) * R(1.0 / 3.0);
    w[2] = (R(2) + R(3) * t - s) * R(1.0 / 6.0);
    return __double2loint(big) - 1;
}

// The same weights and their derivatives with respect to x: with t = x - i0 and
// s = sqrt(1 - 3t^2), dPhi/dt at i0-1, i0, i0+1 = (t/s - 1)/2, -t/s, (1 + t/s)/2.
__device__ __forceinline__ int peskin_window_d(double x, double w[3], double dw[3])
{
    const double big = x + 6755399441055744.0;
    const double t = x - (big - 6755399441055744.0);
    double s, h;                               // s >= 1/2, h = 1/(2 s)
    sqrt_half_inverse(1.0 - 3.0 * t * t, s, h);
    w[0] = (2.0 - 3.0 * t - s) * (1.0 / 6.0);
    w[1] = (1.0 + s) * (1.0 / 3.0);
    w[2] = (2.0 + 3.0 * t - s) * (1.0 / 6.0);
    const double ts = quotient(t, s, 2.0 * h);
    dw[0] = 0.5 * (ts - 1.0);
    dw[1] = -ts;
    dw[2] = 0.5 * (1.0 + ts);
    return __double2loint(big) - 1;
}

// Six times the FP64 weights (2 - s - 3t, 2 + 2s, 2 - s + 3t): the factor 1/216 of three
// dimensions goes into the sum once instead of nine products a window set, and the root needs
// no refined reciprocal: 15 FP64 instructions a window.  An interpolated value is then closer to
// the truth, too (against 113-bit arithmetic 1.6e-16 instead of 2.5e-16: one rounded constant
// instead of three).
__device__ __forceinline__ int peskin_window6(double x, double w[3])
{
    const double big = x + 6755399441055744.0;
    const double t = x - (big - 6755399441055744.0);
    const double t3 = 3.0 * t, a = 1.0 - t3 * t;
    const double y = rsqrt_seed(a);
    const double h = __hiloint2double(__double2hiint(y) - (1 << 20), __double2loint(y));   // y / 2
    const double g = a * y, g1 = fma(g, fma(-g, h, 0.5), g);       // sqrt(a) to 2^-43
    const double s = fma(fma(-g1, g1, a), h, g1);                  // to 2^-65 before its rounding
    const double c = 2.0 - s;
    w[0] = c - t3;
    w[1] = fma(2.0, s, 2.0);
    w[2] = c + t3;
    return __double2loint(big) - 1;
}

// A blob's window along one dimension: three weights (FP64: times six) and the wrapped offsets
// (node index times stride) of their nodes; mask = nodes - 1.  A sum over a 3x3x3 window is to
// be multiplied by UNIT.
template <typename R> struct Win {
    static constexpr double UNIT = sizeof(R) == 8 ? 1.0 / 216.0 : 1.0;
    R w[3];
    int o[3];
    __device__ __forceinline__ void set(double x, int mask, int stride)
    {
        int i;
        if constexpr (sizeof(R) == 8) i = peskin_window6(x, w);
        else i = peskin_window<R>(x, w);
#pragma unroll
        for (int d = 0; d < 3; ++d) o[d] = ((i + d) & mask) * stride;
    }
};

// MAC node offset of component `comp` along dimension `dim`, in mesh units.
__device__ __forceinline__ double mac_shift(int comp, int dim) { return comp == dim ? 0.0 : 0.5; }

// Periodic wrap of a position after a displacement smaller than the box.
__device__ __forceinline__ double wrap_position(double x, double L)
{
    if (x < 0.0) {
        x += L;
        if (x >= L) x -= L;
    } else if (x >= L) {
        x -= L;
    }
    return x;
}

// Periodic image of any position in [0, L).
__device__ __forceinline__ double wrap_any(double x, double L)
{
    if (x >= 0.0 && x < L) return x;
    double y = fmod(x, L);
    if (y < 0.0) y += L;
    if (y >= L) y -= L;
    return y;
}

// |r| and a quotient by it from |r|^2, rounded like the correctly rounded operations (see
// sqrt_half_inverse): nine FP64 instructions for the two, where the library's root and division
// take over twenty.  Squares outside the float range take those.
struct Length {
    double len, inv;          // inv: 1 / len to 2^-43 (fast)
    bool fast;
    __device__ __forceinline__ explicit Length(double r2) : fast(in_seed_range(r2))
    {
        if (fast) {
            double h;
            sqrt_half_inverse(r2, len, h);
            inv = h + h;
        } else {
            len = __dsqrt_rn(r2);
            inv = 0.0;
        }
    }
    __device__ __forceinline__ double divide(double x) const
    {
        return fast ? quotient(x, len, inv) : __ddiv_rn(x, len);
    }
};

// d - L rint(d / L).  Below half the box (decided on the high words, so that the usual case
// takes no FP64 instruction) that is d itself, to the bit.
__device__ __forceinline__ double min_image(double d, double L)
{
    const int half = __double2hiint(L) - (1 << 20);           // high word of L / 2
    if ((__double2hiint(d) & 0x7fffffff) < half) return d;
    return d - L * rint(d / L);
}

}  // namespace mbk
