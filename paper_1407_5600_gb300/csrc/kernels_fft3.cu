// Fluid update of FP32 grids in three passes over HBM (Eq. vf with the viscous stress,
// Crank-Nicolson in time, exact discrete projection), each component transformed on its own
// index grid (FP64 grids: kernels_fft64.cu):
//
//   pass A  per (box, component, z) plane: rhs = (rho/dt) v + (eta/2) L v + f + f_body, then
//           the 2-D real-to-complex FFT of the plane in shared memory     -> spec [z][kx][ky]
//   pass B  per (box, kx, block of ky): FFT along z of all three components, divide by
//           rho/dt + (eta/2) lambda(k), project with the MAC divergence and gradient symbols,
//           set the k = 0 mode, inverse FFT along z                      (in place)
//   pass C  per (box, component, z) plane: 2-D complex-to-real inverse FFT, scale 1/N -> v
//
// Line FFTs: the register-resident line transforms of fft_lines.cuh (lines of up to 128
// points here; the planes of longer sides do not fit in shared memory).
// Real rows are packed two per complex row and separated after the row transform.
#include <cstdlib>
#include <string>
#include <type_traits>

#include "mb_internal.cuh"
#include "fft_lines.cuh"

namespace mbk {

namespace {

__device__ __forceinline__ void load_table(float2* dst, const float2* src, int n)
{
    for (int i = threadIdx.x; i < n; i += blockDim.x) dst[i] = src[i];
}

}  // namespace

// Row stride (in complex) of the plane buffer: just room for the padded nx + 2 separated values
// (a 128 x 128 FP32 plane then takes 73 KiB, three blocks per SM).
__host__ __device__ inline int plane_ld(int nx)
{
    return nx + 2 + ((nx + 1) >> pad_shift(nx));
}

// Plane layouts.  Element (packed row p, slot j) of the plane buffer is P[L.at(p, j)]; rows()
// and cols() transform the ny/2 packed rows (slot j = x) and the nx/2 columns (element y of
// column k is slot 2k + (y & 1) of packed row y >> 1).
//
// PadPlane: any power-of-two plane; one pad slot every 2^pad_shift(nx) slots.
struct PadPlane {
    int nx, ny, S, sx;
    __device__ PadPlane(int nx_, int ny_) : nx(nx_), ny(ny_), S(plane_ld(nx_)), sx(pad_shift(nx_)) {}
    __device__ __forceinline__ int row(int p) const { return p * S; }
    __device__ __forceinline__ int off(int j) const { return j + (j >> sx); }
    __device__ __forceinline__ int at(int p, int j) const { return p * S + j + (j >> sx); }
    template <bool INV> __device__ __forceinline__ void rows(float2* P, const float2* tw) const
    {
        const int S_ = S, sx_ = sx;
        lines_fft_n<INV>(nx, P, ny / 2, [S_, sx_](int l, int j) { return l * S_ + j + (j >> sx_); }, tw);
    }
    template <bool INV> __device__ __forceinline__ void cols(float2* P, const float2* tw) const
    {
        const int S_ = S, sx_ = sx;
        lines_fft_n<INV>(ny, P, nx / 2, [S_, sx_](int k, int y) {
            const int j = 2 * k + (y & 1);
            return (y >> 1) * S_ + j + (j >> sx_);
        }, tw);
    }
};

// Skew128: 128 x 128 planes of float2.  Rows of 148 slots, one pad slot every 16 and a skew of
// SK[(p >> 2) & 7] slots per group of four packed rows, SK = {0, 6, 3, 9, 7, 5, 4, 0}; the row
// lines take lane = 4 t + (line - l0), the column lines lane = 8 (line - l0) + t.  A model of the
// shared-memory banks (8-byte accesses served per half-warp) over every access of the two plane
// passes (loads, both stages of the row and column line FFTs, the separation, the spectrum
// copies) gives this layout 0.63x the wavefronts of the padded one (1.2x the fewest possible);
// 64 rows x 148 slots x 8 B = 74 KiB keeps three planes per SM.  With 128-point lines split
// 16 x 8 (thread t of a line holds elements 8 n1 + t, then 8 (t + 8 m) + n2) every address is
// a per-thread base plus a compile-time offset, so the line FFTs spend no instructions on
// indexing.
struct Skew128 {
    static constexpr int S = 148;
    static constexpr unsigned SKW = 0x04579360u;              // SK[i] = (SKW >> 4 i) & 15
    __host__ __device__ static constexpr int sk(int i) { return (int)((SKW >> (4 * (i & 7))) & 15u); }
    __device__ Skew128(int, int) {}
    __device__ __forceinline__ int row(int p) const { return p * S + sk(p >> 2); }
    __device__ __forceinline__ int off(int j) const { return j + (j >> 4); }
    __device__ __forceinline__ int at(int p, int j) const { return p * S + sk(p >> 2) + j + (j >> 4); }
    // One round: 8 warps x 4 lines; lane = 4 t + (line - l0).  b1 addresses element 8 n1 + t
    // at offset c1(n1); b2 element 8 (t + 8 m) + n2 at c2(m, n2); b1 element (t + 8 m) + 16 k2
    // at c3(m, k2).
    template <bool INV, bool COL>
    __device__ __forceinline__ static void line_round(float2* P, int l, int t, const float2* tw)
    {
        int b1, b2;
        if (COL) {
            b1 = 148 * (t >> 1) + 2 * l + (t & 1) + (l >> 3);
            b2 = 592 * t + 2 * l + (l >> 3) + sk(t);
        } else {
            const int base = l * S + sk(l >> 2);
            b1 = base + t;
            b2 = base + 8 * t + (t >> 1);
        }
        auto c1 = [](int n1) { return COL ? 592 * n1 + sk(n1) : 8 * n1 + (n1 >> 1); };
        auto c2 = [](int m, int n2) { return COL ? 4736 * m + 148 * (n2 >> 1) + (n2 & 1) : 68 * m + n2; };
        auto c3 = [](int m, int k2) { return COL ? 1184 * k2 + 592 * m + sk(2 * k2 + m) : 8 * m + 17 * k2; };
        float2 a[16];
#pragma unroll
        for (int n1 = 0; n1 < 16; ++n1) a[n1] = P[b1 + c1(n1)];
        reg_dft<16, INV>(a);
#pragma unroll
        for (int k1 = 1; k1 < 16; ++k1) {
            float2 w = tw[(t * k1) & 127];
            if (INV) w.y = -w.y;
            a[k1] = cm(a[k1], w);
        }
        __syncwarp();
#pragma unroll
        for (int k1 = 0; k1 < 16; ++k1) P[b1 + c1(k1)] = a[k1];
        __syncwarp();
        float2 b[2][8];
#pragma unroll
        for (int m = 0; m < 2; ++m)
#pragma unroll
            for (int n2 = 0; n2 < 8; ++n2) b[m][n2] = P[b2 + c2(m, n2)];
#pragma unroll
        for (int m = 0; m < 2; ++m) reg_dft<8, INV>(b[m]);
        __syncwarp();
#pragma unroll
        for (int m = 0; m < 2; ++m)
#pragma unroll
            for (int k2 = 0; k2 < 8; ++k2) P[b1 + c3(m, k2)] = b[m][k2];
        __syncwarp();
    }
    template <bool INV, bool COL> __device__ __forceinline__ static void lines(float2* P, const float2* tw)
    {
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
        const int sub = COL ? lane >> 3 : lane & 3, t = COL ? lane & 7 : lane >> 2;
        for (int l0 = warp * 4; l0 < 64; l0 += nw * 4) line_round<INV, COL>(P, l0 + sub, t, tw);
    }
    template <bool INV> __device__ __forceinline__ void rows(float2* P, const float2* tw) const
    {
        lines<INV, false>(P, tw);
    }
    template <bool INV> __device__ __forceinline__ void cols(float2* P, const float2* tw) const
    {
        lines<INV, true>(P, tw);
    }
};

// PlaneT: the other planes with sides of 32, 64 and 128, at compile-time offsets.  One pad slot
// every N2 slots (of the row lines); rows differ by S = 4 (mod 16) slots, or 2 for 32-point rows,
// and by a skew per N2/2 packed rows, so that the lanes of a half-warp (4 rows x 4 threads, 2
// columns x 8) fall on different 8-byte banks in both stages of the line transforms.
template <int NX, int NY> struct PlaneT {
    static constexpr int X2 = Split<NX>::N2, Y2 = Split<NY>::N2, G = Y2 / 2;
    static constexpr int RAW = NX + 2 + (NX + 1) / X2 + 14;                  // pads and skew
    static constexpr int S = RAW + ((NX >= 64 ? 4 : 2) - RAW % 16 + 16) % 16;
    static constexpr unsigned SKW = Y2 == 8 ? (NX >= 64 ? 0xDC985410u : 0x55441100u)
                                            : (NX >= 64 ? 0x11001100u : 0u);
    __host__ __device__ static constexpr int sk(int i) { return (int)((SKW >> (4 * (i & 7))) & 15u); }
    __device__ PlaneT(int, int) {}
    __device__ __forceinline__ int row(int p) const { return p * S + sk(p / G); }
    __device__ __forceinline__ int off(int j) const { return j + j / X2; }
    __device__ __forceinline__ int at(int p, int j) const { return row(p) + off(j); }
    template <bool INV> __device__ __forceinline__ void rows(float2* P, const float2* tw) const
    {
        constexpr int LPW = 32 / X2;
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
        for (int l0 = warp * LPW; l0 < NY / 2; l0 += nw * LPW)
            line_fft<NX, INV, 1>(P + row(l0 + lane % LPW), lane / LPW, tw);
    }
    template <bool INV> __device__ __forceinline__ void cols(float2* P, const float2* tw) const
    {
        constexpr int LPW = 32 / Y2, N1 = Split<NY>::N1;
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
        const int t = lane % Y2;
        // element y of column k: slot 2k + (y & 1) of packed row y / 2
        for (int k0 = warp * LPW; k0 < NX / 2; k0 += nw * LPW) {
            const int c = off(2 * (k0 + lane / Y2));
            line_core<NY, INV>(
                P + (t >> 1) * S + (t & 1) + c, P + G * t * S + sk(t) + c, t, tw,
                [](int n) { return G * n * S + sk(n); },
                [](int m, int n) { return (G * Y2 * m + (n >> 1)) * S + (n & 1); },
                [](int m, int k) { return (G * m + N1 / 2 * k) * S + sk(m + N1 / Y2 * k); });
        }
    }
};

// Blocks an SM: four (64 registers a thread) where no line is longer than 64 points (32 boxes of
// 64^3: forward 100 -> 90 us); lines of 128 spill at that (64 x 128 x 32: 16.4 -> 18.4).
template <typename L> struct PlaneBlocks { static constexpr int N = 3; };
template <int NX, int NY> struct PlaneBlocks<PlaneT<NX, NY>> {
    static constexpr int N = NX > 64 || NY > 64 ? 3 : 4;
};

template <typename L> struct PlaneSlots;
template <> struct PlaneSlots<PadPlane> { static size_t count(int nx, int ny) { return (size_t)(ny / 2) * plane_ld(nx); } };
template <> struct PlaneSlots<Skew128> { static size_t count(int, int) { return 64 * (size_t)Skew128::S; } };
template <int NX, int NY> struct PlaneSlots<PlaneT<NX, NY>> {
    static size_t count(int, int) { return (size_t)(NY / 2) * PlaneT<NX, NY>::S; }
};

// ------------------------------------------------------------------------------------------
// Pass A.  Plane buffer P[p][pad(j)], p < ny/2: first rows 2p, 2p+1 packed as re + i im; after
// the row FFT and the in-place separation, logical slot 2k + e of row p holds X_{2p+e}[k],
// k <= nx/2.  pad(j) = j + (j >> pad_shift(nx)).
template <typename L, bool STRESS>
__global__ void __launch_bounds__(256, PlaneBlocks<L>::N)
k_plane_fwd(FluidArgs<float> a, GridGeo g)
{
    dep_wait();
    dep_release();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int nx = g.n[0], ny = g.n[1], nz = g.n[2], nxh = nx / 2 + 1;
    const L lay(nx, ny);
    float2* P = reinterpret_cast<float2*>(smem_raw);
    const float2* twx = reinterpret_cast<const float2*>(a.twk[0]);      // twiddles through L1
    const float2* twy = reinterpret_cast<const float2*>(a.twk[1]);
    const int z = blockIdx.x, bc = blockIdx.y, comp = bc % 3;
    const float* vc = a.v + (size_t)bc * g.N;
    const float* fc = a.f ? a.f + (size_t)bc * g.N : nullptr;
    const float ih2 = kparam<float>(a.inv_h2, a.inv_h2_32), rho_dt = kparam<float>(a.rho_dt, a.rho_dt32),
            half_eta = kparam<float>(a.half_eta, a.half_eta32);
    const bool body = a.body_prof && comp == a.body_axis;
    const float* pz = vc + (size_t)z * ny * nx;
    const float* pzp = vc + (size_t)((z + 1) & (nz - 1)) * ny * nx;
    const float* pzm = vc + (size_t)((z - 1) & (nz - 1)) * ny * nx;
    // planes that nothing was spread into are zero: neither read nor cleared
    const bool spread = fc && !(a.f_dirty && a.f_dirty[(bc / 3) * nz + z] == 0);
    const float* pf = spread ? fc + (size_t)z * ny * nx : nullptr;
    float* pclr = a.f_clear && spread ? a.f_clear + (size_t)bc * g.N + (size_t)z * ny * nx : nullptr;
    // each work unit: 4 consecutive x of the two rows 2p, 2p+1
    const int qx = nx / 4, lq = 31 - __clz(qx);   // nx is a power of two
    for (int u = threadIdx.x; u < qx * (ny / 2) && a.no_v; u += blockDim.x) {
        // Stokes limit: the right-hand side is the force density (and body force) alone
        const int x0 = 4 * (u & (qx - 1)), p = u >> lq;
        const int y0 = 2 * p, y1 = y0 + 1;
        const float z0 = 0.0f;
        float r0[4] = {z0, z0, z0, z0}, r1[4] = {z0, z0, z0, z0};
        if (pf) {
            load4(pf + (size_t)y0 * nx + x0, r0);
            load4(pf + (size_t)y1 * nx + x0, r1);
        }
        if (body) {
            for (int i = 0; i < 4; ++i) {
                const int x = x0 + i;
                r0[i] += (a.body_prof[a.body_dir == 0 ? x : (a.body_dir == 1 ? y0 : z)]);
                r1[i] += (a.body_prof[a.body_dir == 0 ? x : (a.body_dir == 1 ? y1 : z)]);
            }
        }
        float2* rowp = P + lay.row(p);
        for (int i = 0; i < 4; ++i) rowp[lay.off(x0 + i)] = float2{r0[i], r1[i]};
    }
    for (int u = threadIdx.x; u < qx * (ny / 2) && !a.no_v; u += blockDim.x) {
        const int x0 = 4 * (u & (qx - 1)), p = u >> lq;
        const int y0 = 2 * p, y1 = y0 + 1;
        const int ym = (y0 - 1) & (ny - 1), yp = (y1 + 1) & (ny - 1);
        float c0[4], c1[4], am[4], ap[4], t[4];
        load4(pz + (size_t)y0 * nx + x0, c0);
        load4(pz + (size_t)y1 * nx + x0, c1);
        load4(pz + (size_t)ym * nx + x0, am);
        load4(pz + (size_t)yp * nx + x0, ap);
        float l0[4], l1[4];
        for (int i = 0; i < 4; ++i) {
            l0[i] = am[i] + c1[i] - 6.0f * c0[i];
            l1[i] = c0[i] + ap[i] - 6.0f * c1[i];
        }
        load4(pzp + (size_t)y0 * nx + x0, t);
        for (int i = 0; i < 4; ++i) l0[i] += t[i];
        load4(pzm + (size_t)y0 * nx + x0, t);
        for (int i = 0; i < 4; ++i) l0[i] += t[i];
        load4(pzp + (size_t)y1 * nx + x0, t);
        for (int i = 0; i < 4; ++i) l1[i] += t[i];
        load4(pzm + (size_t)y1 * nx + x0, t);
        for (int i = 0; i < 4; ++i) l1[i] += t[i];
        const int xm = (x0 - 1) & (nx - 1), xp = (x0 + 4) & (nx - 1);
        const float e0m = (pz[(size_t)y0 * nx + xm]), e0p = (pz[(size_t)y0 * nx + xp]);
        const float e1m = (pz[(size_t)y1 * nx + xm]), e1p = (pz[(size_t)y1 * nx + xp]);
        for (int i = 0; i < 4; ++i) {
            l0[i] += (i == 0 ? e0m : c0[i - 1]) + (i == 3 ? e0p : c0[i + 1]);
            l1[i] += (i == 0 ? e1m : c1[i - 1]) + (i == 3 ? e1p : c1[i + 1]);
        }
        float r0[4], r1[4];
        for (int i = 0; i < 4; ++i) {
            r0[i] = rho_dt * c0[i] + half_eta * (l0[i] * ih2);
            r1[i] = rho_dt * c1[i] + half_eta * (l1[i] * ih2);
        }
        if (pf) {
            load4(pf + (size_t)y0 * nx + x0, t);
            for (int i = 0; i < 4; ++i) r0[i] += t[i];
            load4(pf + (size_t)y1 * nx + x0, t);
            for (int i = 0; i < 4; ++i) r1[i] += t[i];
        }
        if (STRESS)
            stress_rows(a.W + (size_t)(bc / 3) * 9 * g.N, comp, g, x0, y0, z, -a.inv_h32, r0, r1);
        if (body) {
            for (int i = 0; i < 4; ++i) {
                const int x = x0 + i;
                r0[i] += (a.body_prof[a.body_dir == 0 ? x : (a.body_dir == 1 ? y0 : z)]);
                r1[i] += (a.body_prof[a.body_dir == 0 ? x : (a.body_dir == 1 ? y1 : z)]);
            }
        }
        float2* rowp = P + lay.row(p);
        for (int i = 0; i < 4; ++i) rowp[lay.off(x0 + i)] = float2{r0[i], r1[i]};
    }
    __syncthreads();
    // leave f zeroed for the next accumulation: behind the barrier, since a store between the loads
    // keeps the next ones back (128^3 Stokes 47 -> 25 us, 64 x 128 x 32 with stress 16.4 -> 12.7)
    if (pclr)
        for (int i = threadIdx.x; i < nx * ny / 4; i += blockDim.x)
            reinterpret_cast<float4*>(pclr)[i] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    if (STRESS && a.step_index && (blockIdx.x | blockIdx.y | threadIdx.x) == 0)
        *a.step_index += 1;                // the stress of this step has been drawn
    lay.template rows<false>(P, twx);
    __syncthreads();
    // separate the two real rows of each packed row (one warp per packed row, in place)
    {
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
        for (int p = warp; p < ny / 2; p += nw) {
            float2* rowp = P + lay.row(p);
            float2 ev[3], od[3];        // nx/2 + 1 <= 65 values: at most 3 per lane
#pragma unroll
            for (int r = 0; r < 3; ++r) {
                const int k = lane + 32 * r;
                if (k < nxh) {
                    const int kr = (nx - k) & (nx - 1);
                    const float2 Z = rowp[lay.off(k)], Zr = rowp[lay.off(kr)];
                    ev[r] = float2{(Z.x + Zr.x) * 0.5f, (Z.y - Zr.y) * 0.5f};
                    od[r] = float2{(Z.y + Zr.y) * 0.5f, (Zr.x - Z.x) * 0.5f};
                }
            }
            __syncwarp();
#pragma unroll
            for (int r = 0; r < 3; ++r) {
                const int k = lane + 32 * r;
                if (k < nxh) {
                    rowp[lay.off(2 * k)] = ev[r];
                    rowp[lay.off(2 * k + 1)] = od[r];
                }
            }
            __syncwarp();
        }
    }
    __syncthreads();
    auto col = [lay](int k, int y) { return lay.at(y >> 1, 2 * k + (y & 1)); };
    // columns k = 0 and k = nx/2 are real: transform them as one complex column
    // Z_y = X_y[0] + i X_y[nx/2], so that nx/2 column lines remain
    for (int y = threadIdx.x; y < ny; y += blockDim.x)
        P[col(0, y)] = float2{P[col(0, y)].x, P[col(nx / 2, y)].x};
    __syncthreads();
    lay.template cols<false>(P, twy);
    __syncthreads();
    // A = FFT X[0] = (Z_k + conj Z_-k) / 2,  B = FFT X[nx/2] = (Z_k - conj Z_-k) / (2i)
    if (threadIdx.x < 32) {
        float2 av[4], bv[4];            // ny <= 128: at most 4 per lane
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const int k = threadIdx.x + 32 * r;
            if (k < ny) {
                const float2 Zk = P[col(0, k)], Zr = P[col(0, (ny - k) & (ny - 1))];
                av[r] = float2{(Zk.x + Zr.x) * 0.5f, (Zk.y - Zr.y) * 0.5f};
                bv[r] = float2{(Zk.y + Zr.y) * 0.5f, (Zr.x - Zk.x) * 0.5f};
            }
        }
        __syncwarp();
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const int k = threadIdx.x + 32 * r;
            if (k < ny) {
                P[col(0, k)] = av[r];
                P[col(nx / 2, k)] = bv[r];
            }
        }
    }
    __syncthreads();
    float2* out = reinterpret_cast<float2*>(a.spec) + ((size_t)bc * nz + z) * (size_t)nxh * ny;
    const int ly = 31 - __clz(ny);
    if (blockDim.x % ny == 0) {
        // a thread keeps its y (so its packed row and parity) and steps through k
        const int y = threadIdx.x & (ny - 1), e = y & 1, dk = blockDim.x >> ly;
        const float2* rowp = P + lay.row(y >> 1);
        for (int k = threadIdx.x >> ly; k < nxh; k += dk) out[k * ny + y] = rowp[lay.off(2 * k + e)];
    } else {
        for (int i = threadIdx.x; i < nxh * ny; i += blockDim.x) out[i] = P[col(i >> ly, i & (ny - 1))];
    }
}

// ------------------------------------------------------------------------------------------
// Pass B.  CTA = (ky block of width C, kx, box).  NZ: the line length where the kernel has it at
// compile time (NZ / N1 threads a line, 3 C of them one round; element z of component c, column k
// at ((c * padded_line + z + z / N2) * CL + k), or 0 for any length, buffer [3][pad(nz)][C + 4].
template <int C, int NZ>
__global__ void __launch_bounds__(3 * C * 8, 768 / (3 * C * 8))
k_zsolve(FluidArgs<float> a, GridGeo g)
{
    constexpr bool FIX = NZ != 0;
    constexpr int NL = FIX ? NZ : 4, Z2 = Split<NL>::N2, ZP = padded_line<NL>();
    // half-warps of 4 lines x 4 threads (strides of 12 slots) or 8 x 2 (8 slots) on different banks
    constexpr int CL = FIX && Z2 == 4 ? 8 : C + 4, LPW = 32 / Z2;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int nx = g.n[0], ny = g.n[1], nz = FIX ? NZ : g.n[2], nxh = nx / 2 + 1;
    const int lz = 31 - __clz(nz);
    const int sz = pad_shift(nz), nzp = FIX ? ZP : padded_len(nz);
    float2* Bf = reinterpret_cast<float2*>(smem_raw);
    float2* twz = Bf + 3 * nzp * CL;
    load_table(twz, reinterpret_cast<const float2*>(a.twk[2]), nz);   // set up once: no wait
    dep_wait();
    dep_release();
    const int ky0 = blockIdx.x * C, kx = blockIdx.y, box = blockIdx.z;
    if (a.f_dirty && blockIdx.x == 0 && kx == 0)          // pass A has read them
        for (int i = threadIdx.x; i < nz; i += blockDim.x) a.f_dirty[box * nz + i] = 0;
    const size_t zstride = (size_t)nxh * ny;
    const size_t cstride = (size_t)nz * zstride;
    float2* base = reinterpret_cast<float2*>(a.spec) + (size_t)(box * 3) * cstride + (size_t)kx * ny + ky0;
    auto at = [=](int c, int z, int k) {
        return (c * nzp + (FIX ? pad_line<NL>(z) : z + (z >> sz))) * CL + k;
    };
    const int total = 3 * nz * C;
    // compile-time lines: thread (row r = 2 tid / C, columns k, k + 1) moves 16 bytes of the elements
    // z = z0 + 2 N2 j of component r / (2 N2), at fixed strides on both sides; z0 = r % (2 N2) with
    // its low bits swapped, so that the two rows of a quarter-warp (CL = 12: 96 bytes apart for
    // neighbours, 64 mod 128 for every other) fall on different banks.  8 -> 16 bytes: 32 boxes of
    // 64^3 68.2 -> 64.0 us, 128^3 20.4 -> 19.2
    const int fk = 2 * (threadIdx.x % (C / 2)), fr = threadIdx.x / (C / 2), f0 = fr % (2 * Z2);
    const int fz = Z2 == 4 ? f0 : (f0 & ~3) | (f0 & 1) << 1 | (f0 >> 1 & 1);
    float2* fs = Bf + (fr / (2 * Z2) * ZP + pad_line<NL>(fz)) * CL + fk;
    float2* fg = base + fr / (2 * Z2) * cstride + (size_t)fz * zstride + fk;
    if constexpr (FIX) {
#pragma unroll
        for (int j = 0; j < NL / (2 * Z2); ++j)
            async_copy(reinterpret_cast<float4*>(fs + 2 * (Z2 + 1) * CL * j),
                       reinterpret_cast<const float4*>(fg + (size_t)(2 * Z2 * j) * zstride));
    } else {
        for (int i = threadIdx.x; i < total; i += blockDim.x) {
            const int k = i % C, zc = i / C, z = zc & (nz - 1), c = zc >> lz;
            async_copy(&Bf[at(c, z, k)], &base[c * cstride + (size_t)z * zstride + k]);
        }
    }
    async_wait_all();
    __syncthreads();
    auto idx = [=](int l, int z) { return at(l / C, z, l % C); };
    const int lane = threadIdx.x & 31, l = (threadIdx.x >> 5) * LPW + lane % LPW;
    float2* mine = Bf + l / C * (ZP * CL) + l % C;
    if constexpr (FIX) line_fft<NL, false, CL>(mine, lane / LPW, twz);
    else lines_fft_n<false>(nz, Bf, 3 * C, idx, twz);
    __syncthreads();
    const float* sym = reinterpret_cast<const float*>(a.symk);     // [9][256] cos, sin, lambda
    const float ih = kparam<float>(a.inv_h, a.inv_h32);
    const float csx = sym[0 * 256 + kx], snx = sym[1 * 256 + kx], lx = sym[2 * 256 + kx];
    const float rho_dt = kparam<float>(a.rho_dt, a.rho_dt32);
    const float half_eta = kparam<float>(a.half_eta, a.half_eta32);
    // with blockDim a multiple of C a thread keeps its column k (and ky's symbols) throughout
    const int kfix = threadIdx.x % C;
    const float csy = sym[3 * 256 + ky0 + kfix], sny = sym[4 * 256 + ky0 + kfix];
    const float lxy = lx + sym[5 * 256 + ky0 + kfix];
    const bool colfix = blockDim.x % C == 0;
    for (int i = threadIdx.x; i < nz * C; i += blockDim.x) {
        const int k = colfix ? kfix : i % C, kz = i / C, ky = ky0 + k;
        const float cs[3] = {csx, colfix ? csy : sym[3 * 256 + ky], sym[6 * 256 + kz]};
        const float sn[3] = {snx, colfix ? sny : sym[4 * 256 + ky], sym[7 * 256 + kz]};
        const float lam = (colfix ? lxy : lx + sym[5 * 256 + ky]) + sym[8 * 256 + kz];
        const float cinv = recip(rho_dt + half_eta * lam);
        float2 W[3];
        for (int c = 0; c < 3; ++c) {
            const float2 v = Bf[at(c, kz, k)];
            W[c] = float2{v.x * cinv, v.y * cinv};
        }
        if (kx == 0 && ky == 0 && kz == 0) {
            for (int c = 0; c < 3; ++c) {
                if (a.mean_state) {              // the only thread of this box at k = 0
                    double m = a.mean_state[3 * box + c];
                    if (a.mean_force) m += a.mean_scale * a.mean_force[3 * box + c];
                    a.mean_state[3 * box + c] = m;
                    W[c] = float2{(float)((double)g.N * m), 0.0f};
                } else if (a.mean_override) {
                    W[c] = float2{(float)((double)g.N * a.mean_override[3 * box + c]), 0.0f};
                } else if (a.mean_mode == 1) {
                    W[c] = float2{0.0f, 0.0f};
                }
            }
        } else {
            // D_a = (e^{i th} - 1)/h, G_a = (1 - e^{-i th})/h, D.G = -lambda:
            // P W = W + G (D.W) / lambda
            float dr = 0.0f, di = 0.0f;
            for (int c = 0; c < 3; ++c) {
                const float Dr = (cs[c] - 1.0f) * ih, Di = sn[c] * ih;
                dr += Dr * W[c].x - Di * W[c].y;
                di += Dr * W[c].y + Di * W[c].x;
            }
            const float il = recip(lam);
            dr *= il;
            di *= il;
            for (int c = 0; c < 3; ++c) {
                const float Gr = (1.0f - cs[c]) * ih, Gi = sn[c] * ih;
                W[c].x += Gr * dr - Gi * di;
                W[c].y += Gr * di + Gi * dr;
            }
        }
        for (int c = 0; c < 3; ++c) Bf[at(c, kz, k)] = W[c];
    }
    __syncthreads();
    if constexpr (FIX) line_fft<NL, true, CL>(mine, lane / LPW, twz);
    else lines_fft_n<true>(nz, Bf, 3 * C, idx, twz);
    __syncthreads();
    if constexpr (FIX) {
#pragma unroll
        for (int j = 0; j < NL / (2 * Z2); ++j)
            *reinterpret_cast<float4*>(fg + (size_t)(2 * Z2 * j) * zstride) =
                *reinterpret_cast<const float4*>(fs + 2 * (Z2 + 1) * CL * j);
    } else {
        for (int i = threadIdx.x; i < total; i += blockDim.x) {
            const int k = i % C, zc = i / C, z = zc & (nz - 1), c = zc >> lz;
            base[c * cstride + (size_t)z * zstride + k] = Bf[at(c, z, k)];
        }
    }
}

// ------------------------------------------------------------------------------------------
// Pass C.  Inverse of pass A: columns, then the packed rows Z = X_{2p} + i X_{2p+1} (with the
// Hermitian extension X[nx - k] = conj X[k]), then the real rows, scaled by 1/N.
template <typename L>
__global__ void __launch_bounds__(256, 3)
k_plane_inv(FluidArgs<float> a, GridGeo g)
{
    // no early release: the next kernel (the interpolation's persistent grid, which splits the
    // blobs evenly over its warps) then starts all its blocks together, not first on the SMs
    // this pass leaves early
    dep_wait();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int nx = g.n[0], ny = g.n[1], nz = g.n[2], nxh = nx / 2 + 1;
    const L lay(nx, ny);
    float2* P = reinterpret_cast<float2*>(smem_raw);
    const float2* twx = reinterpret_cast<const float2*>(a.twk[0]);      // twiddles through L1
    const float2* twy = reinterpret_cast<const float2*>(a.twk[1]);
    const int z = blockIdx.x, bc = blockIdx.y;
    const float2* in = reinterpret_cast<const float2*>(a.spec) + ((size_t)bc * nz + z) * (size_t)nxh * ny;
    auto col = [lay](int k, int y) { return lay.at(y >> 1, 2 * k + (y & 1)); };
    const int ly = 31 - __clz(ny);
    if (blockDim.x % ny == 0) {
        const int y = threadIdx.x & (ny - 1), e = y & 1, dk = blockDim.x >> ly;
        float2* rowp = P + lay.row(y >> 1);
        for (int k = threadIdx.x >> ly; k < nxh; k += dk) async_copy(&rowp[lay.off(2 * k + e)], &in[k * ny + y]);
    } else {
        for (int i = threadIdx.x; i < nxh * ny; i += blockDim.x) async_copy(&P[col(i >> ly, i & (ny - 1))], &in[i]);
    }
    async_wait_all();
    __syncthreads();
    // columns k = 0 and k = nx/2 invert to real sequences: transform their Hermitian parts as
    // one complex column Z = herm(A) + i herm(B), whose inverse is Re(IFFT A) + i Re(IFFT B)
    if (threadIdx.x < 32) {
        float2 zv[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const int k = threadIdx.x + 32 * r;
            if (k < ny) {
                const int kr = (ny - k) & (ny - 1);
                const float2 A = P[col(0, k)], Ar = P[col(0, kr)];
                const float2 Bv = P[col(nx / 2, k)], Br = P[col(nx / 2, kr)];
                // herm(A) = (A_k + conj A_-k) / 2, herm(B) likewise; Z = herm(A) + i herm(B)
                const float2 ha = float2{(A.x + Ar.x) * 0.5f, (A.y - Ar.y) * 0.5f};
                const float2 hb = float2{(Bv.x + Br.x) * 0.5f, (Bv.y - Br.y) * 0.5f};
                zv[r] = float2{ha.x - hb.y, ha.y + hb.x};
            }
        }
        __syncwarp();
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const int k = threadIdx.x + 32 * r;
            if (k < ny) P[col(0, k)] = zv[r];
        }
    }
    __syncthreads();
    lay.template cols<true>(P, twy);
    __syncthreads();
    for (int y = threadIdx.x; y < ny; y += blockDim.x) {
        const float2 zc = P[col(0, y)];
        P[col(0, y)] = float2{zc.x, 0.0f};
        P[col(nx / 2, y)] = float2{zc.y, 0.0f};
    }
    __syncthreads();
    {
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
        for (int p = warp; p < ny / 2; p += nw) {
            float2* rowp = P + lay.row(p);
            float2 zv[4];              // nx <= 128 values: at most 4 per lane
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const int k = lane + 32 * r;
                if (k < nx) {
                    const int kk = k <= nx / 2 ? k : nx - k;
                    float2 e = rowp[lay.off(2 * kk)], o = rowp[lay.off(2 * kk + 1)];
                    if (k == 0 || k == nx / 2) { e.y = 0.0f; o.y = 0.0f; }
                    if (k > nx / 2) { e.y = -e.y; o.y = -o.y; }
                    zv[r] = float2{e.x - o.y, e.y + o.x};
                }
            }
            __syncwarp();
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const int k = lane + 32 * r;
                if (k < nx) rowp[lay.off(k)] = zv[r];
            }
            __syncwarp();
        }
    }
    __syncthreads();
    lay.template rows<true>(P, twx);
    __syncthreads();
    const float scale = kparam<float>(a.inv_n, a.inv_n32);
    float* out = a.v_out + (size_t)bc * g.N + (size_t)z * ny * nx;
    const int qx = nx / 4, lq = 31 - __clz(qx);   // nx is a power of two
    for (int u = threadIdx.x; u < qx * (ny / 2); u += blockDim.x) {
        const int x0 = 4 * (u & (qx - 1)), p = u >> lq;
        float r0[4], r1[4];
        const float2* rowp = P + lay.row(p);
        for (int i = 0; i < 4; ++i) {
            const float2 zv = rowp[lay.off(x0 + i)];
            r0[i] = zv.x * scale;
            r1[i] = zv.y * scale;
        }
        store4(out + (size_t)(2 * p) * nx + x0, r0);
        store4(out + (size_t)(2 * p + 1) * nx + x0, r1);
        if (a.v_sum_out) {               // v^n + v^{n+1} for the corrector's single gather
            const size_t o0 = (size_t)bc * g.N + (size_t)z * ny * nx + (size_t)(2 * p) * nx + x0;
            float b0[4], b1[4];
            load4(a.v_sum_base + o0, b0);
            load4(a.v_sum_base + o0 + nx, b1);
            for (int i = 0; i < 4; ++i) {
                b0[i] += r0[i];
                b1[i] += r1[i];
            }
            store4(a.v_sum_out + o0, b0);
            store4(a.v_sum_out + o0 + nx, b1);
        }
    }
}

using PlaneKernel = void (*)(FluidArgs<float>, GridGeo);
struct PlanePass {
    PlaneKernel fwd[2], inv;               // fwd[1]: with the fluid stress
    size_t slots;
    int threads, resident;                 // resident: blocks of fwd an SM holds
};
template <typename L> PlanePass plane_pass(int nx, int ny, int threads)
{
    PlanePass p{{k_plane_fwd<L, false>, k_plane_fwd<L, true>}, k_plane_inv<L>,
                PlaneSlots<L>::count(nx, ny), threads, 1};
    static std::atomic<unsigned> attr{0};     // per layout
    static std::atomic<int> resident{0};
    if (first_on_device(attr))
        for (PlaneKernel k : {p.fwd[0], p.fwd[1], p.inv})
            cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
    p.resident = resident_blocks(resident, p.fwd[0], threads, p.slots * sizeof(float2));
    return p;
}
// as many threads as one round of lines takes, at most 256
template <int NX, int NY> PlanePass plane_fixed()
{
    constexpr int r = NY / 2 * Split<NX>::N2, c = NX / 2 * Split<NY>::N2, m = r > c ? r : c;
    using L = std::conditional_t<NX == 128 && NY == 128, Skew128, PlaneT<NX, NY>>;
    return plane_pass<L>(NX, NY, m < 256 ? m : 256);
}
template <int NX> PlanePass plane_of(int ny)
{
    return ny == 32 ? plane_fixed<NX, 32>() : (ny == 64 ? plane_fixed<NX, 64>() : plane_fixed<NX, 128>());
}

template <>
cudaError_t launch_fluid3<float>(Chain chain, int B, const GridGeo& g, const FluidArgs<float>& a_in,
                          cudaEvent_t* marks)
{
    cudaStream_t st = chain.st;                      // always a chain of programmatic dependents
    const FluidArgs<float> a = with_derived(a_in, g);
    const int nx = g.n[0], ny = g.n[1], nz = g.n[2], nxh = nx / 2 + 1;
    // planes of sides from 32 to 128 have layouts at compile-time offsets; MB_PLANE_LAYOUT=pad
    // keeps the padded run-time one, for comparison.  32 boxes of 64^3, run-time / compile-time:
    // forward 128 / 90 us (with the untouched planes of f left out), inverse 114 / 75 (without
    // the sum v^n + v^{n+1}), z 77 / 64; the L1 is then 83 to 88% busy
    static const bool pad = [] {
        const char* e = std::getenv("MB_PLANE_LAYOUT");
        return e && std::string(e) == "pad";
    }();
    const bool fixed = !pad && nx >= 32 && ny >= 32;
    const PlanePass pp = !fixed ? plane_pass<PadPlane>(nx, ny, 256)
                         : nx == 128 ? plane_of<128>(ny)
                         : nx == 64 ? plane_of<64>(ny) : plane_of<32>(ny);
    const size_t smem_plane = pp.slots * sizeof(float2);
    // z lines of 32 to 128 points at compile-time offsets, 8 columns a block
    const int C = ny >= 8 ? 8 : 4, zfix = C == 8 && nz >= 32 ? nz : 0;
    PlaneKernel zs = zfix == 128 ? k_zsolve<8, 128> : zfix == 64 ? k_zsolve<8, 64>
                     : zfix == 32 ? k_zsolve<8, 32> : C == 8 ? k_zsolve<8, 0> : k_zsolve<4, 0>;
    const int Z2 = zfix == 32 ? 4 : 8, CL = zfix == 32 ? 8 : C + 4;
    const unsigned tz = zfix ? 3 * C * Z2 : 3 * C * 8;
    const size_t smem_z = ((size_t)3 * (zfix ? nz + nz / Z2 : padded_len(nz)) * CL + nz) * sizeof(float2);
    static std::atomic<unsigned> attr{0};
    if (first_on_device(attr))
        for (PlaneKernel k : {k_zsolve<8, 128>, k_zsolve<8, 64>, k_zsolve<8, 32>, k_zsolve<8, 0>, k_zsolve<4, 0>})
            cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
    auto mark = [&](int i) { if (marks) cudaEventRecord(marks[i], st); };
    mark(0);
    const dim3 gp(nz, 3 * B), gz(ny / C, nxh, B);
    // Steps with this pass always a dependent / as the rule says, 4,160 blobs: 128 x 128 x 32
    // 79.5 / 54.9 us, 128 x 128 x 64 82.9 / 70.1, 64^3 46.6 / 41.4.  Planes of less than 64 x 64 gain by
    // lying evenly only behind the nine-lane spreading, which ends at once (64 x 32 x 32 38.7 / 35.4; behind
    // the tiles, which hold all SMs, the early start hides the launch: two boxes of 32^3, 20,000 blobs
    // 48.0 / 52.3), those of 16 x 16 not even there (four boxes, 4,160 blobs 32.8 / 34.2).
    const int cells = nx * ny;
    const bool even = cells >= 64 * 64 || (a.after_short && cells >= 32 * 32);
    cudaError_t e = launch_on(Chain(st, !even || start_early((int64_t)nz * 3 * B, pp.resident)),
                              pp.fwd[a.W ? 1 : 0], gp, dim3(pp.threads), smem_plane, a, g);
    if (e != cudaSuccess) return e;
    mark(1);
    mark(2);
    e = launch_dep(zs, gz, dim3(tz), smem_z, st, a, g);
    if (e != cudaSuccess) return e;
    mark(3);
    mark(4);
    e = launch_dep(pp.inv, gp, dim3(pp.threads), smem_plane, st, a, g);
    if (e != cudaSuccess) return e;
    mark(5);
    return cudaGetLastError();
}

}  // namespace mbk
