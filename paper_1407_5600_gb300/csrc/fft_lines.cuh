// Line FFTs held in registers, shared by the three-pass and five-pass fluid solvers.
//
// A line of N = N1 N2 points is done by N2 threads of one warp.  Thread t holds the N1 points
// x[N2 n1 + t] in registers, does an N1-point DFT, multiplies by W_N^{t k1}, and the line is
// exchanged once through shared memory; then each thread does N1/N2 DFTs of N2 points
// (X[k1 + N1 k2] = sum_n2 W_N2^{n2 k2} W_N^{n2 k1} sum_n1 x[N2 n1 + n2] W_N1^{n1 k1}).
#pragma once
#include "mb_internal.cuh"

namespace mbk {
namespace {

template <typename T> __device__ __forceinline__ T cm(T a, T b)
{
    return T{a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x};
}
template <typename T> __device__ __forceinline__ T cadd(T a, T b) { return T{a.x + b.x, a.y + b.y}; }
// The correctly rounded float reciprocal (a single intrinsic instead of a division).
__device__ __forceinline__ float recip(float x) { return __frcp_rn(x); }
// FP64: Newton's iteration from the hardware's float reciprocal (four FP64 instructions instead
// of the division's twenty or so) where argument and reciprocal are normal floats: 2^-126 <= x < 2^126.
// Good to 2^-85 before its rounding, so one in 2^32 may round to the other neighbour.
__device__ __forceinline__ double recip(double x)
{
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
    if (hi - (897u << 20) >= (252u << 20)) return 1.0 / x;
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;"
        : "=f"(y) : "f"(__uint_as_float(((hi - (896u << 20)) << 3) | (lo >> 29))));
    const unsigned yb = __float_as_uint(y);
    double r = __hiloint2double((int)((yb >> 3) + (896u << 20)), (int)(yb << 29));
    r = fma(r, fma(-x, r, 1.0), r);
    return fma(r, fma(-x, r, 1.0), r);
}
template <typename T> __device__ __forceinline__ T csub(T a, T b) { return T{a.x - b.x, a.y - b.y}; }

__host__ __device__ constexpr int bitrev(int i, int bits)
{
    int r = 0;
    for (int b = 0; b < bits; ++b) r |= ((i >> b) & 1) << (bits - 1 - b);
    return r;
}
__host__ __device__ constexpr int ilog2c(int n) { return n <= 1 ? 0 : 1 + ilog2c(n / 2); }

// cos and sin of 2 pi j / 16, j < 8 (the twiddles of the in-register DFTs of up to 16 points;
// after unrolling every index is a constant and the values fold into the arithmetic).
template <typename R> __device__ __forceinline__ R cos16(int j)
{
    switch (j) {
    case 0: return R(1.0);
    case 1: return R(0.92387953251128675613);
    case 2: return R(0.70710678118654752440);
    case 3: return R(0.38268343236508977173);
    case 4: return R(0.0);
    case 5: return R(-0.38268343236508977173);
    case 6: return R(-0.70710678118654752440);
    default: return R(-0.92387953251128675613);
    }
}
constexpr double TAN8 = 0.41421356237309504880;      // tan(pi / 8) = sqrt(2) - 1
// sin(2 pi j / 16) = cos(2 pi (j - 4) / 16), j < 8
template <typename R> __device__ __forceinline__ R sin16(int j) { return cos16<R>(j < 4 ? 4 - j : j - 4); }

// Butterfly (a, b) -> (a + w b, a - w b), w = W_16^j (forward) or W_16^-j (inverse), with
// W_16 = exp(-2 pi i / 16); j < 8.  The larger of w's cosine and sine is taken out (Linzer and
// Feig): w b = c (b.x -+ r b.y, b.y +- r b.x), |r| <= 1, so that a general one takes six fused
// operations instead of two products, two fused ones and four additions.
template <bool INV, typename T> __device__ __forceinline__ void butterfly(T& a, T& b, int j)
{
    using R = decltype(b.x);
    T u;
    if (j == 0) u = b;
    else if (j == 4) u = INV ? T{-b.y, b.x} : T{b.y, -b.x};
    if (j == 0 || j == 4) {
        b = csub(a, u);
        a = cadd(a, u);
        return;
    }
    const R c = cos16<R>(j), s = INV ? sin16<R>(j) : -sin16<R>(j);
    R f;                                     // the factor taken out
    if (j < 3 || j > 5) {                    // |cos| >= |sin|
        const R r = R((INV ? 1.0 : -1.0) * (j == 1 ? TAN8 : j == 2 ? 1.0 : j == 6 ? -1.0 : -TAN8));
        u = T{b.x - r * b.y, b.y + r * b.x};
        f = c;
    } else {                                 // j = 3, 5: w b = s (r b.x - b.y, r b.y + b.x)
        const R r = R((INV ? 1.0 : -1.0) * (j == 3 ? TAN8 : -TAN8));
        u = T{r * b.x - b.y, r * b.y + b.x};
        f = s;
    }
    b = T{a.x - f * u.x, a.y - f * u.y};
    a = T{a.x + f * u.x, a.y + f * u.y};
}

// One radix-2 stage (butterfly span LEN) of an in-register DIT DFT, then the next stage.  The
// span is a template argument so that every loop has a constant trip count and unrolls fully,
// which turns each twiddle index into a constant.
template <int P, int LEN, bool INV, typename T>
__device__ __forceinline__ void dft_stage(T (&x)[P])
{
    constexpr int HALF = LEN / 2;
#pragma unroll
    for (int s0 = 0; s0 < P; s0 += LEN) {
#pragma unroll
        for (int m = 0; m < HALF; ++m) {
            butterfly<INV>(x[s0 + m], x[s0 + m + HALF], m * (16 / LEN));
        }
    }
    if constexpr (LEN < P) dft_stage<P, 2 * LEN, INV>(x);
}

// In-register radix-2 DIT DFT of P <= 16 points with constant twiddles W_P^m = W_16^(16 m / P).
template <int P, bool INV, typename T>
__device__ __forceinline__ void reg_dft(T (&x)[P])
{
    static_assert(P <= 16, "in-register DFTs of at most 16 points");
    constexpr int bits = ilog2c(P);
#pragma unroll
    for (int i = 0; i < P; ++i) {
        const int r = bitrev(i, bits);
        if (r > i) {
            const T tmp = x[i];
            x[i] = x[r];
            x[r] = tmp;
        }
    }
    if constexpr (P > 1) dft_stage<P, 2, INV>(x);
}

template <int N> struct Split;                  // N = N1 * N2 with N1 >= N2, N1 % N2 == 0
template <> struct Split<4> { static constexpr int N1 = 2, N2 = 2; };
template <> struct Split<8> { static constexpr int N1 = 4, N2 = 2; };
template <> struct Split<16> { static constexpr int N1 = 4, N2 = 4; };
template <> struct Split<32> { static constexpr int N1 = 8, N2 = 4; };
template <> struct Split<64> { static constexpr int N1 = 8, N2 = 8; };
template <> struct Split<128> { static constexpr int N1 = 16, N2 = 8; };
template <> struct Split<256> { static constexpr int N1 = 16, N2 = 16; };

// FFTs of `lines` lines of N points held in shared memory; element j of line l is at
// buf[idx(l, j)].  All threads of the block call this; lines are spread over warps with the
// N2 threads of a line inside one warp, so only warp-level synchronisation is needed.
template <int N, bool INV, typename T, typename Idx>
__device__ __forceinline__ void lines_fft(T* buf, int lines, Idx idx, const T* __restrict__ tw)
{
    constexpr int N1 = Split<N>::N1, N2 = Split<N>::N2, M = N1 / N2;
    constexpr int LPW = 32 / N2;                 // lines per warp per round
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    // consecutive lanes take consecutive lines: with the callers' padded layouts the lanes of
    // a half-warp then fall on distinct shared-memory banks
    const int sub = lane % LPW, t = lane / LPW;
    for (int l0 = warp * LPW; l0 < lines; l0 += nw * LPW) {
        const int l = l0 + sub;
        const bool on = l < lines;
        T a[N1];
#pragma unroll
        for (int n1 = 0; n1 < N1; ++n1) a[n1] = on ? buf[idx(l, N2 * n1 + t)] : T{};
        reg_dft<N1, INV>(a);
#pragma unroll
        for (int k1 = 1; k1 < N1; ++k1) {
            T w = tw[(t * k1) & (N - 1)];
            if (INV) w.y = -w.y;
            a[k1] = cm(a[k1], w);
        }
        __syncwarp();
        if (on) {
#pragma unroll
            for (int k1 = 0; k1 < N1; ++k1) buf[idx(l, k1 * N2 + t)] = a[k1];
        }
        __syncwarp();
        T b[M][N2];
#pragma unroll
        for (int m = 0; m < M; ++m)
#pragma unroll
            for (int n2 = 0; n2 < N2; ++n2)
                b[m][n2] = on ? buf[idx(l, (t + N2 * m) * N2 + n2)] : T{};
#pragma unroll
        for (int m = 0; m < M; ++m) reg_dft<N2, INV>(b[m]);
        __syncwarp();
        if (on) {
#pragma unroll
            for (int m = 0; m < M; ++m)
#pragma unroll
                for (int k2 = 0; k2 < N2; ++k2) buf[idx(l, (t + N2 * m) + N1 * k2)] = b[m][k2];
        }
        __syncwarp();
    }
}

// One line of N = N1 N2 points at compile-time offsets: thread t (of N2) finds element N2 n1 + t
// at b1[c1(n1)], element (t + N2 m) N2 + n2 at b2[c2(m, n2)] and element t + N2 m + N1 k2 at
// b1[c3(m, k2)], so the transform spends no instructions on indexing.  (With run-time layouts the
// 256^3 passes issued 145 instructions a point, 43% of them integer.)
template <int N, bool INV, typename T, typename F1, typename F2, typename F3>
__device__ __forceinline__ void line_core(T* b1, const T* b2, int t, const T* __restrict__ tw, F1 c1,
                                          F2 c2, F3 c3)
{
    constexpr int N1 = Split<N>::N1, N2 = Split<N>::N2, M = N1 / N2;
    T a[N1];
#pragma unroll
    for (int n = 0; n < N1; ++n) a[n] = b1[c1(n)];
    reg_dft<N1, INV>(a);
#pragma unroll
    for (int k = 1; k < N1; ++k) {
        T w = tw[(t * k) & (N - 1)];
        if (INV) w.y = -w.y;
        a[k] = cm(a[k], w);
    }
    __syncwarp();
#pragma unroll
    for (int k = 0; k < N1; ++k) b1[c1(k)] = a[k];
    __syncwarp();
    T b[M][N2];
#pragma unroll
    for (int m = 0; m < M; ++m)
#pragma unroll
        for (int n = 0; n < N2; ++n) b[m][n] = b2[c2(m, n)];
#pragma unroll
    for (int m = 0; m < M; ++m) reg_dft<N2, INV>(b[m]);
    __syncwarp();
#pragma unroll
    for (int m = 0; m < M; ++m)
#pragma unroll
        for (int k = 0; k < N2; ++k) b1[c3(m, k)] = b[m][k];
    __syncwarp();
}

// Lines whose element j is at (j + j / N2) CL from the line's first, CL a compile-time stride:
// N2 n + t at (N2 + 1) n + t, and so on.
template <int N> __host__ __device__ constexpr int padded_line() { return N + N / Split<N>::N2; }
template <int N> __host__ __device__ __forceinline__ int pad_line(int j) { return j + j / Split<N>::N2; }
template <int N, bool INV, int CL, typename T>
__device__ __forceinline__ void line_fft(T* line, int t, const T* __restrict__ tw)
{
    constexpr int N1 = Split<N>::N1, N2 = Split<N>::N2;
    line_core<N, INV>(
        line + t * CL, line + (N2 + 1) * CL * t, t, tw, [](int n) { return (N2 + 1) * CL * n; },
        [](int m, int n) { return ((N2 + 1) * N2 * m + n) * CL; },
        [](int m, int k) { return (N2 + 1) * (m + N1 / N2 * k) * CL; });
}

template <bool INV, typename T, typename Idx>
__device__ __forceinline__ void lines_fft_n(int n, T* buf, int lines, Idx idx, const T* tw)
{
    switch (n) {
    case 4: lines_fft<4, INV>(buf, lines, idx, tw); break;
    case 8: lines_fft<8, INV>(buf, lines, idx, tw); break;
    case 16: lines_fft<16, INV>(buf, lines, idx, tw); break;
    case 32: lines_fft<32, INV>(buf, lines, idx, tw); break;
    case 64: lines_fft<64, INV>(buf, lines, idx, tw); break;
    default: lines_fft<128, INV>(buf, lines, idx, tw); break;
    }
}

// Padded position of element j of a line of n points: one spare slot every N2 elements (N2 of
// the line FFT), which spreads the strided accesses of the second stage over the banks.
__host__ __device__ __forceinline__ int pad_shift(int n)
{
    return n >= 64 ? 3 : (n >= 16 ? 2 : 1);
}
__host__ __device__ __forceinline__ int padded_len(int n) { return n + (n >> pad_shift(n)); }

// Asynchronous global-to-shared copy of one complex value (no register staging, so every copy
// of a thread is in flight at once), and the wait for all of a thread's copies.
template <typename T> __device__ __forceinline__ void async_copy(T* dst, const T* src)
{
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    if constexpr (sizeof(T) == 16)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(src) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void async_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

// Four consecutive grid values (x0 .. x0+3, x0 a multiple of 4) as one vector load.
__device__ __forceinline__ void load4(const float* p, float v[4])
{
    const float4 q = *reinterpret_cast<const float4*>(p);
    v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
}
__device__ __forceinline__ void load4(const double* p, double v[4])
{
    const double2 a = reinterpret_cast<const double2*>(p)[0];
    const double2 b = reinterpret_cast<const double2*>(p)[1];
    v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
}
__device__ __forceinline__ void store4(float* p, const float v[4])
{
    *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
}
__device__ __forceinline__ void store4(double* p, const double v[4])
{
    reinterpret_cast<double2*>(p)[0] = make_double2(v[0], v[1]);
    reinterpret_cast<double2*>(p)[1] = make_double2(v[2], v[3]);
}
// Adds mih D.T (mih = -1/h) on the faces of component `comp` at the cells x0 .. x0+3 of the rows
// (y0, z) and (y0 + 1, z) to r0 and r1: T is the staggered stress [9][N] of kernels_noise.cu,
// backward differences of T_aa, forward ones of T_ab.
template <typename R>
__device__ __forceinline__ void stress_rows(const R* __restrict__ T, int comp, const GridGeo& g,
                                            int x0, int y0, int z, R mih, R r0[4], R r1[4])
{
    const int nx = g.n[0], ny = g.n[1], nz = g.n[2];
    const int zr = z * ny, o0 = (zr + y0) * nx, o1 = o0 + nx;
    R c0[4], c1[4], e[4];
    {
        const R* t = T + (size_t)(3 * comp) * g.N;
        load4(t + o0 + x0, c0);
        load4(t + o1 + x0, c1);
        const bool back = comp == 0;
        const int xn = back ? (x0 - 1) & (nx - 1) : (x0 + 4) & (nx - 1);
        const R n0 = t[o0 + xn], n1 = t[o1 + xn];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const R d0 = back ? c0[i] - (i == 0 ? n0 : c0[i - 1]) : (i == 3 ? n0 : c0[i + 1]) - c0[i];
            const R d1 = back ? c1[i] - (i == 0 ? n1 : c1[i - 1]) : (i == 3 ? n1 : c1[i + 1]) - c1[i];
            r0[i] += mih * d0;
            r1[i] += mih * d1;
        }
    }
    {
        const R* t = T + (size_t)(3 * comp + 1) * g.N;
        const bool back = comp == 1;
        load4(t + o0 + x0, c0);
        load4(t + o1 + x0, c1);
        load4(t + (zr + ((back ? y0 - 1 : y0 + 2) & (ny - 1))) * nx + x0, e);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            r0[i] += mih * (back ? c0[i] - e[i] : c1[i] - c0[i]);
            r1[i] += mih * (back ? c1[i] - c0[i] : e[i] - c1[i]);
        }
    }
    {
        const R* t = T + (size_t)(3 * comp + 2) * g.N;
        const bool back = comp == 2;
        const int zn = (((back ? z - 1 : z + 1) & (nz - 1)) * ny + y0) * nx + x0;
        load4(t + o0 + x0, c0);
        load4(t + zn, e);
#pragma unroll
        for (int i = 0; i < 4; ++i) r0[i] += mih * (back ? c0[i] - e[i] : e[i] - c0[i]);
        load4(t + o1 + x0, c1);
        load4(t + zn + nx, e);
#pragma unroll
        for (int i = 0; i < 4; ++i) r1[i] += mih * (back ? c1[i] - e[i] : e[i] - c1[i]);
    }
}

}  // namespace
}  // namespace mbk
