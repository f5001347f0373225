// Fluid update on the periodic MAC grid: Crank-Nicolson viscous step and exact discrete
// projection (Eq. vf with the viscous stress), solved in Fourier space.
//
// Pipeline per box and component (each component transformed on its own index grid):
//   pass 1  rhs = (rho/dt) v + (eta/2) L v + f + f_body, then real-to-complex FFT along x
//           (two real rows packed into one complex row)           -> spec [z][y][kx]
//   pass 2  complex FFT along y                                     (in place)
//   pass 3  complex FFT along z, divide by rho/dt + (eta/2) lambda(k), project with the MAC
//           divergence/gradient symbols, set the k = 0 mode, inverse FFT along z
//   pass 4  inverse FFT along y
//   pass 5  complex-to-real inverse FFT along x, scale 1/N         -> v_out
// Every pass stages its lines in shared memory (padded against bank conflicts) and transforms
// them with the register line FFTs of fft_lines.cuh; global traffic is one coalesced read and
// one write of the half spectrum per pass.  This pipeline takes sides of up to 256 points.
//
// Spectrum rows are padded to whole 64-byte runs (spec_row), so that a chunk of columns starts
// on a sector: at nx/2 + 1 values a row a chunk of 8 touched three sectors instead of two.  A
// block has as many threads as its lines need (n / N1 each, lines_threads): with 256 threads
// whatever the sides, the 64-point passes left six of eight warps without a line.  256-point
// lines have layouts of their own with compile-time offsets (line_fft).  Times before and after:
// FP32 256^3 rhs (with the stress divergence, a pass of its own before) 165 + 180 -> 258 us,
// y 134 -> 78, z and solve 275 -> 167, c2r 196 -> 110; FP64 256 x 64 x 64 800 -> 590 us in all.
#include "mb_internal.cuh"
#include "fft_lines.cuh"

namespace mbk {

// Padded position of element j of a line of n points (one spare slot every 2^pad_shift).
__device__ __forceinline__ int pj(int j, int sh) { return j + (j >> sh); }

// Layouts of 256-point lines in the passes: columns of the y and z passes at these strides, rows
// of the x passes at ROW256, chosen so that the lanes of a half-warp (a quarter-warp of 16-byte
// values: eight threads of two lines, four of two) fall on different banks in every access.
template <typename R> struct Lay256 {
    static constexpr int YL = 3, CY = 1 << YL;       // columns of a y block
    static constexpr int ZL = 3, CZ = 1 << ZL;       // columns of a z block
    static constexpr int YS = CY + 2, ZS = CZ + 2;
    static constexpr int ROW = sizeof(R) == 4 ? 280 : 276;
};

// Threads that share a line of n points in lines_fft (N2 of its split).
inline int line_threads(int n) { return n == 256 ? 16 : (n >= 64 ? 8 : (n >= 16 ? 4 : 2)); }
// Lines a block of about `threads` threads transforms at once, a power of two, at most `most`
// rounded up to one.
inline int lines_per_block(int n, int threads, int most)
{
    int l = threads / line_threads(n);
    while (l > 1 && l / 2 >= most) l /= 2;
    return l;
}
inline unsigned block_threads(int lines, int n)
{
    return (unsigned)((lines * line_threads(n) + 31) & ~31);            // whole warps
}

// ------------------------------------------------------------------------------------------
// Pass 1: rhs stencil + R2C along x.  CTA = RP row pairs of one (box, component, z) plane.
template <typename R, bool STRESS, bool L256>
__global__ void __launch_bounds__(sizeof(R) == 4 ? 256 : 128, sizeof(R) == 4 ? 3 : 2)
k_rhs_fft_x(FluidArgs<R> a, GridGeo g, int RP)
{
    using T = typename C2<R>::T;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T* sb = reinterpret_cast<T*>(smem_raw);
    const int nx = g.n[0], ny = g.n[1], nz = g.n[2], ld_s = spec_row(nx);
    const int sx = pad_shift(nx), ld = L256 ? Lay256<R>::ROW : padded_len(nx) + 1;
    auto px = [sx](int j) { return L256 ? pad_line<256>(j) : pj(j, sx); };
    const int yp0 = blockIdx.x * RP;
    const int z = blockIdx.y;
    const int bc = blockIdx.z;
    const int comp = bc % 3;
    const R* vc = a.v + (size_t)bc * g.N;
    const R* fc = a.f ? a.f + (size_t)bc * g.N : nullptr;
    // rhs = (rho/dt) v + beta L v + f, L v = sum of the six neighbours - 6 v formed first: a rounding
    // of rho/dt - 6 beta would not cancel on smooth fields and scale every low mode, the same way
    // each step (at eta dt / (rho h^2) = 10, FP32: 5.3e-7 a step; 0.8e-7 this way, the transforms')
    const R beta = kparam<R>(a.half_eta * a.inv_h2, a.half_eta32 * a.inv_h2_32);
    const R rho_dt = kparam<R>(a.rho_dt, a.rho_dt32);
    const bool body = a.body_prof && comp == a.body_axis;
    const size_t zp = (size_t)((z + 1) & (nz - 1)) * ny, zm = (size_t)((z - 1) & (nz - 1)) * ny;
    const size_t z0 = (size_t)z * ny;
    // each work unit: 4 consecutive x (one vector load) of the row pair 2p, 2p+1
    const int qx = nx / 4, lq = 31 - __clz(qx);
    const R* pz = vc + z0 * nx;
    const R* pzp = vc + zp * nx;
    const R* pzm = vc + zm * nx;
    const R* pf = fc ? fc + z0 * nx : nullptr;
    for (int u = threadIdx.x; u < qx * RP; u += blockDim.x) {
        const int x0 = 4 * (u & (qx - 1)), p = u >> lq;
        const int y0 = 2 * (yp0 + p), y1 = y0 + 1;
        R r0[4] = {R(0), R(0), R(0), R(0)}, r1[4] = {R(0), R(0), R(0), R(0)}, t[4];
        if (!a.no_v) {              // Stokes limit (no_v): the right-hand side is f + f_body
            const int ym = (y0 - 1) & (ny - 1), yp = (y1 + 1) & (ny - 1);
            R c0[4], c1[4], am[4], ap[4], l0[4], l1[4];
            load4(pz + (size_t)y0 * nx + x0, c0);
            load4(pz + (size_t)y1 * nx + x0, c1);
            load4(pz + (size_t)ym * nx + x0, am);
            load4(pz + (size_t)yp * nx + x0, ap);
            for (int i = 0; i < 4; ++i) {
                l0[i] = am[i] + c1[i] - R(6) * c0[i];
                l1[i] = c0[i] + ap[i] - R(6) * c1[i];
            }
            load4(pzp + (size_t)y0 * nx + x0, t);
            for (int i = 0; i < 4; ++i) l0[i] += t[i];
            load4(pzm + (size_t)y0 * nx + x0, t);
            for (int i = 0; i < 4; ++i) l0[i] += t[i];
            load4(pzp + (size_t)y1 * nx + x0, t);
            for (int i = 0; i < 4; ++i) l1[i] += t[i];
            load4(pzm + (size_t)y1 * nx + x0, t);
            for (int i = 0; i < 4; ++i) l1[i] += t[i];
            const int xm = (x0 - 1) & (nx - 1), xq = (x0 + 4) & (nx - 1);
            const R e0m = pz[(size_t)y0 * nx + xm], e0p = pz[(size_t)y0 * nx + xq];
            const R e1m = pz[(size_t)y1 * nx + xm], e1p = pz[(size_t)y1 * nx + xq];
            for (int i = 0; i < 4; ++i) {
                l0[i] += (i == 0 ? e0m : c0[i - 1]) + (i == 3 ? e0p : c0[i + 1]);
                l1[i] += (i == 0 ? e1m : c1[i - 1]) + (i == 3 ? e1p : c1[i + 1]);
                r0[i] = rho_dt * c0[i] + beta * l0[i];
                r1[i] = rho_dt * c1[i] + beta * l1[i];
            }
        }
        if (pf) {
            load4(pf + (size_t)y0 * nx + x0, t);
            for (int i = 0; i < 4; ++i) r0[i] += t[i];
            load4(pf + (size_t)y1 * nx + x0, t);
            for (int i = 0; i < 4; ++i) r1[i] += t[i];
        }
        if (STRESS) stress_rows(a.W + (size_t)(bc / 3) * 9 * g.N, comp, g, x0, y0, z, R(-a.inv_h), r0, r1);
        if (body) {
            for (int i = 0; i < 4; ++i) {
                const int x = x0 + i;
                r0[i] += a.body_prof[a.body_dir == 0 ? x : (a.body_dir == 1 ? y0 : z)];
                r1[i] += a.body_prof[a.body_dir == 0 ? x : (a.body_dir == 1 ? y1 : z)];
            }
        }
        for (int i = 0; i < 4; ++i) sb[p * ld + px(x0 + i)] = T{r0[i], r1[i]};
    }
    __syncthreads();
    if constexpr (L256)
        line_fft<256, false, 1>(sb + (2 * (threadIdx.x >> 5) + (threadIdx.x & 1)) * ld, (threadIdx.x & 31) >> 1,
                       reinterpret_cast<const T*>(a.twf[0]));
    else
        lines_fft_n<false>(nx, sb, RP, [ld, sx](int l, int j) { return l * ld + pj(j, sx); },
                        reinterpret_cast<const T*>(a.twf[0]));
    __syncthreads();
    if (STRESS && a.step_index && (blockIdx.x | blockIdx.y | blockIdx.z | threadIdx.x) == 0)
        *a.step_index += 1;            // the stress of this step has been drawn
    T* out = a.spec + ((size_t)bc * nz + z) * (size_t)ny * ld_s;
    // row p, frequency k <= nx/2: even row (Z + conj Zr)/2, odd row -i (Z - conj Zr)/2
    auto emit = [&](int p, int k) {
        const T Z = sb[p * ld + px(k)];
        const T Zr = sb[p * ld + px((nx - k) & (nx - 1))];
        const T Xa{(Z.x + Zr.x) * R(0.5), (Z.y - Zr.y) * R(0.5)};
        const T Xb{(Z.y + Zr.y) * R(0.5), (Zr.x - Z.x) * R(0.5)};
        const int y = 2 * (yp0 + p);
        out[(size_t)y * ld_s + k] = Xa;
        out[(size_t)(y + 1) * ld_s + k] = Xb;
    };
    const int hx = nx / 2, lh = 31 - __clz(hx);
    for (int t = threadIdx.x; t < RP * hx; t += blockDim.x) emit(t >> lh, t & (hx - 1));
    for (int p = threadIdx.x; p < RP; p += blockDim.x) emit(p, hx);
}

// Pass 2 / 4: complex FFT along y.  CTA = C = 2^lc consecutive kx columns of one (box, comp, z).
template <typename R, bool INV, bool L256>
__global__ void __launch_bounds__(sizeof(R) == 4 ? 256 : 128, 3)
k_fft_y(typename C2<R>::T* spec, const R* twy, GridGeo g, int lc)
{
    using T = typename C2<R>::T;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T* sb = reinterpret_cast<T*>(smem_raw);
    const int nx = g.n[0], ny = g.n[1], nz = g.n[2], nxh = nx / 2 + 1, ld_s = spec_row(nx);
    if (L256) lc = Lay256<R>::YL;
    const int C = 1 << lc, kx0 = blockIdx.x * C;
    const int cw = min(C, nxh - kx0);
    const int sy = pad_shift(ny), CL = L256 ? Lay256<R>::YS : C + 1;
    auto at = [=](int y, int c) { return (L256 ? pad_line<256>(y) : pj(y, sy)) * CL + c; };
    T* plane = spec + ((size_t)blockIdx.z * nz + blockIdx.y) * (size_t)ny * ld_s + kx0;
    // every copy of a thread in flight at once (columns past the last kx are transformed as
    // garbage and not stored).  256 points, sixteen threads a column: a thread's elements y0 + 16 j
    // are at fixed strides on both sides
    const int fc = threadIdx.x & (C - 1), fy = threadIdx.x >> lc;
    if constexpr (L256) {
        if (fc < cw) {
#pragma unroll
            for (int j = 0; j < 16; ++j)
                async_copy(sb + fy * CL + fc + 17 * Lay256<R>::YS * j,
                           plane + (size_t)fy * ld_s + fc + (size_t)(16 * j) * ld_s);
        }
    } else {
        for (int t = threadIdx.x; t < ny * C; t += blockDim.x) {
            const int y = t >> lc, c = t & (C - 1);
            if (c < cw) async_copy(&sb[at(y, c)], &plane[(size_t)y * ld_s + c]);
        }
    }
    async_wait_all();
    __syncthreads();
    const T* tw = reinterpret_cast<const T*>(twy);
    if constexpr (L256)
        line_fft<256, INV, Lay256<R>::YS>(sb + 2 * (threadIdx.x >> 5) + (threadIdx.x & 1),
                                    (threadIdx.x & 31) >> 1, tw);
    else
        lines_fft_n<INV>(ny, sb, C, [CL, sy](int l, int j) { return pj(j, sy) * CL + l; }, tw);
    __syncthreads();
    if constexpr (L256) {
        if (fc < cw) {
#pragma unroll
            for (int j = 0; j < 16; ++j)
                plane[(size_t)fy * ld_s + fc + (size_t)(16 * j) * ld_s] =
                    sb[fy * CL + fc + 17 * Lay256<R>::YS * j];
        }
    } else {
        for (int t = threadIdx.x; t < ny * C; t += blockDim.x) {
            const int y = t >> lc, c = t & (C - 1);
            if (c < cw) plane[(size_t)y * ld_s + c] = sb[at(y, c)];
        }
    }
}

// Pass 3: FFT along z, Crank-Nicolson divide, projection, k = 0 mode, inverse FFT along z.
// CTA = C = 2^LC consecutive kx columns at one ky of one box, all three components.
template <typename R, bool L256>
__global__ void __launch_bounds__(384, sizeof(R) == 4 ? 2 : 1)
k_fft_z_solve(FluidArgs<R> a, GridGeo g, int LC)
{
    using T = typename C2<R>::T;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T* sb = reinterpret_cast<T*>(smem_raw);    // [3][nz][C]
    const int nx = g.n[0], ny = g.n[1], nz = g.n[2], nxh = nx / 2 + 1, ld_s = spec_row(nx);
    if (L256) LC = Lay256<R>::ZL;
    const int C = 1 << LC, kx0 = blockIdx.x * C;
    const int cw = min(C, nxh - kx0);
    const int ky = blockIdx.y;
    const int box = blockIdx.z;
    const size_t zstride = (size_t)ny * ld_s;
    T* col[3];
    for (int c = 0; c < 3; ++c)
        col[c] = a.spec + ((size_t)(box * 3 + c) * nz) * zstride + (size_t)ky * ld_s + kx0;
    const int sz = pad_shift(nz), PZ = L256 ? padded_line<256>() : padded_len(nz), CL = L256 ? Lay256<R>::ZS : C + 1;
    auto at = [=](int c, int z, int k) { return (c * PZ + (L256 ? pad_line<256>(z) : pj(z, sz))) * CL + k; };
    // z twiddles in shared memory, after the three component columns (ready at the barrier
    // that follows the column copies)
    T* twz = sb + 3 * PZ * CL;
    for (int i = threadIdx.x; i < nz; i += blockDim.x) twz[i] = reinterpret_cast<const T*>(a.twf[2])[i];
    const int lz = 31 - __clz(nz);
    // index arithmetic in shifts (C and nz are powers of two); columns past the last kx are
    // transformed as garbage and not stored
    // 256 points: thread (row r = tid / CZ, column k) moves the elements z = r % 16 + 16 j of
    // component r / 16, at fixed strides on both sides
    const int fk = threadIdx.x & (Lay256<R>::CZ - 1), fr = threadIdx.x >> Lay256<R>::ZL;
    T* fs = sb + ((fr >> 4) * padded_line<256>() + (fr & 15)) * Lay256<R>::ZS + fk;
    T* fg = a.spec + ((size_t)(box * 3 + (fr >> 4)) * nz + (fr & 15)) * zstride + (size_t)ky * ld_s + kx0 + fk;
    if constexpr (L256) {
        if (fk < cw) {
#pragma unroll
            for (int j = 0; j < 16; ++j)
                async_copy(fs + 17 * Lay256<R>::ZS * j, fg + (size_t)(16 * j) * zstride);
        }
    } else {
        for (int t = threadIdx.x; t < 3 * nz * C; t += blockDim.x) {
            const int k = t & (C - 1), z = (t >> LC) & (nz - 1), c = t >> (LC + lz);
            if (k < cw) async_copy(&sb[at(c, z, k)], &col[c][(size_t)z * zstride + k]);
        }
    }
    async_wait_all();
    __syncthreads();
    // 256 points: two lines a warp
    auto idx = [=](int l, int j) { return at(l >> LC, j, l & (C - 1)); };
    const int l2 = 2 * (threadIdx.x >> 5) + (threadIdx.x & 1);
    T* mine = sb + (l2 >> Lay256<R>::ZL) * (padded_line<256>() * Lay256<R>::ZS) + (l2 & (Lay256<R>::CZ - 1));
    if constexpr (L256) line_fft<256, false, Lay256<R>::ZS>(mine, (threadIdx.x & 31) >> 1, twz);
    else lines_fft_n<false>(nz, sb, 3 * C, idx, twz);
    __syncthreads();

    const R* sym = reinterpret_cast<const R*>(a.symr);      // [9][256] cos, sin, lambda
    const R* cosx = sym + 0 * 256;
    const R* sinx = sym + 1 * 256;
    const R* lamx = sym + 2 * 256;
    const R* cosy = sym + 3 * 256;
    const R* siny = sym + 4 * 256;
    const R* lamy = sym + 5 * 256;
    const R* cosz = sym + 6 * 256;
    const R* sinz = sym + 7 * 256;
    const R* lamz = sym + 8 * 256;
    const R h2 = kparam<R>(1.0 / a.inv_h2, 1.0f / a.inv_h2_32);
    const R rho_dt = kparam<R>(a.rho_dt, a.rho_dt32);
    const R half_eta = kparam<R>(a.half_eta, a.half_eta32);
    // the block has a multiple of C threads: a thread keeps its column
    const int k = threadIdx.x & (C - 1), kx = kx0 + k;
    const R cx = R(cosx[kx]) - R(1), sx = R(sinx[kx]), cy = R(cosy[ky]) - R(1), sy = R(siny[ky]);
    const R lxy = R(lamx[kx]) + R(lamy[ky]);
    for (int kz = threadIdx.x >> LC; kz < nz; kz += blockDim.x >> LC) {
        T W[3];
        const R lam = lxy + R(lamz[kz]);
        const R cinv = recip(rho_dt + half_eta * lam);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const T v = sb[at(c, kz, k)];
            W[c] = T{v.x * cinv, v.y * cinv};
        }
        if (kx == 0 && ky == 0 && kz == 0) {
            for (int c = 0; c < 3; ++c) {
                if (a.mean_override) W[c] = T{R((double)g.N * a.mean_override[3 * box + c]), R(0)};
                else if (a.mean_mode == 1) W[c] = T{R(0), R(0)};
            }
        } else {
            // D_a = (e^{i th} - 1)/h (faces -> centres), G_a = (1 - e^{-i th})/h = -conj D_a
            // (centres -> faces); D.G = -lambda, so P W = W + G (D.W) / lambda.  The symbols
            // are taken without 1/h, whose square goes into 1/lambda.
            const R cr[3] = {cx, cy, R(cosz[kz]) - R(1)}, sn[3] = {sx, sy, R(sinz[kz])};
            R dr = R(0), di = R(0);
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                dr += cr[c] * W[c].x - sn[c] * W[c].y;
                di += cr[c] * W[c].y + sn[c] * W[c].x;
            }
            const R il = recip(lam * h2);
            dr *= il;
            di *= il;
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                W[c].x -= cr[c] * dr + sn[c] * di;
                W[c].y -= cr[c] * di - sn[c] * dr;
            }
        }
#pragma unroll
        for (int c = 0; c < 3; ++c) sb[at(c, kz, k)] = W[c];
    }
    __syncthreads();
    if constexpr (L256) line_fft<256, true, Lay256<R>::ZS>(mine, (threadIdx.x & 31) >> 1, twz);
    else lines_fft_n<true>(nz, sb, 3 * C, idx, twz);
    __syncthreads();
    if constexpr (L256) {
        if (fk < cw) {
#pragma unroll
            for (int j = 0; j < 16; ++j) fg[(size_t)(16 * j) * zstride] = fs[17 * Lay256<R>::ZS * j];
        }
    } else {
        for (int t = threadIdx.x; t < 3 * nz * C; t += blockDim.x) {
            const int k = t & (C - 1), z = (t >> LC) & (nz - 1), c = t >> (LC + lz);
            if (k < cw) col[c][(size_t)z * zstride + k] = sb[at(c, z, k)];
        }
    }
}

// Pass 5: C2R along x.  Two half-spectrum rows form Z = Xa + i Xb (Hermitian extension),
// one inverse complex FFT gives both real rows.
template <typename R, bool L256>
__global__ void __launch_bounds__(sizeof(R) == 4 ? 256 : 128, sizeof(R) == 4 ? 3 : 2)
k_fft_x_c2r(FluidArgs<R> a, GridGeo g, int RP)
{
    using T = typename C2<R>::T;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T* sb = reinterpret_cast<T*>(smem_raw);
    const int nx = g.n[0], ny = g.n[1], nz = g.n[2], ld_s = spec_row(nx);
    const int sx = pad_shift(nx), ld = L256 ? Lay256<R>::ROW : padded_len(nx) + 1;
    auto px = [sx](int j) { return L256 ? pad_line<256>(j) : pj(j, sx); };
    const int yp0 = blockIdx.x * RP;
    const int z = blockIdx.y;
    const int bc = blockIdx.z;
    const T* in = a.spec + ((size_t)bc * nz + z) * (size_t)ny * ld_s;
    // each frequency read once, for its own place and its mirror's (k = 0 with nx/2, both real)
    const int hx = nx / 2, lh = 31 - __clz(hx);
#pragma unroll 4
    for (int t = threadIdx.x; t < RP * hx; t += blockDim.x) {
        const int k = t & (hx - 1), p = t >> lh;
        const T* row = in + (size_t)(2 * (yp0 + p)) * ld_s;
        const T Xa = __ldg(row + k), Xb = __ldg(row + ld_s + k);
        T* Z = sb + p * ld;
        if (k == 0) {
            Z[px(0)] = T{Xa.x, Xb.x};
            Z[px(hx)] = T{__ldg(row + hx).x, __ldg(row + ld_s + hx).x};
        } else {
            Z[px(k)] = T{Xa.x - Xb.y, Xa.y + Xb.x};
            Z[px(nx - k)] = T{Xa.x + Xb.y, Xb.x - Xa.y};
        }
    }
    __syncthreads();
    if constexpr (L256)
        line_fft<256, true, 1>(sb + (2 * (threadIdx.x >> 5) + (threadIdx.x & 1)) * ld, (threadIdx.x & 31) >> 1,
                       reinterpret_cast<const T*>(a.twf[0]));
    else
        lines_fft_n<true>(nx, sb, RP, [ld, sx](int l, int j) { return l * ld + pj(j, sx); },
                        reinterpret_cast<const T*>(a.twf[0]));
    __syncthreads();
    const R scale = kparam<R>(a.inv_n, a.inv_n32);
    R* out = a.v_out + (size_t)bc * g.N + (size_t)z * ny * nx;
    const int qx = nx / 4, lq = 31 - __clz(qx);
    for (int u = threadIdx.x; u < qx * RP; u += blockDim.x) {
        const int x0 = 4 * (u & (qx - 1)), p = u >> lq;
        R r0[4], r1[4];
        for (int i = 0; i < 4; ++i) {
            const T zv = sb[p * ld + px(x0 + i)];
            r0[i] = zv.x * scale;
            r1[i] = zv.y * scale;
        }
        store4(out + (size_t)(2 * (yp0 + p)) * nx + x0, r0);
        store4(out + (size_t)(2 * (yp0 + p) + 1) * nx + x0, r1);
    }
}

template <typename R>
cudaError_t launch_fluid(cudaStream_t st, int B, const GridGeo& g, const FluidArgs<R>& a_in,
                         cudaEvent_t* marks)
{
    const FluidArgs<R> a = with_derived(a_in, g);
    using T = typename C2<R>::T;
    const int nx = g.n[0], ny = g.n[1], nz = g.n[2], nxh = nx / 2 + 1;
    using L = Lay256<R>;
    const bool x256 = nx == 256, y256 = ny == 256, z256 = nz == 256;
    auto rhs = a.W ? (x256 ? k_rhs_fft_x<R, true, true> : k_rhs_fft_x<R, true, false>)
                   : (x256 ? k_rhs_fft_x<R, false, true> : k_rhs_fft_x<R, false, false>);
    auto yf = y256 ? k_fft_y<R, false, true> : k_fft_y<R, false, false>;
    auto yi = y256 ? k_fft_y<R, true, true> : k_fft_y<R, true, false>;
    auto zs = z256 ? k_fft_z_solve<R, true> : k_fft_z_solve<R, false>;
    auto c2r = x256 ? k_fft_x_c2r<R, true> : k_fft_x_c2r<R, false>;
    static std::atomic<unsigned> attr{0};     // per instantiation
    if (first_on_device(attr)) {
        const int lim = 200 * 1024;
        for (auto k : {k_rhs_fft_x<R, true, true>, k_rhs_fft_x<R, true, false>,
                       k_rhs_fft_x<R, false, true>, k_rhs_fft_x<R, false, false>,
                       k_fft_x_c2r<R, true>, k_fft_x_c2r<R, false>, k_fft_z_solve<R, true>,
                       k_fft_z_solve<R, false>})
            cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
        for (auto k : {k_fft_y<R, false, true>, k_fft_y<R, false, false>, k_fft_y<R, true, true>,
                       k_fft_y<R, true, false>})
            cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
    }
    // Block sizes (times at 256^3, FP32): x passes of one warp (two 256-point row pairs) keep
    // more blocks in different phases on an SM than wider ones: 276 / 126 us with 256 threads,
    // 258 / 112 with 64, 250 / 110 with 32 (before the centre's own instruction).  y blocks of 8 columns (64-byte runs) 78 us, of 16
    // 87 us; z blocks of 8 columns 167 us, of 4 (32-byte runs) 178 us.  FP64 blocks are bound by
    // the FP64 pipe (80-84% busy) at four warps.
    const int rp = lines_per_block(nx, sizeof(R) == 4 ? 32 : 128, ny / 2), RP = rp < ny / 2 ? rp : ny / 2;
    // the z pass holds three components of its columns: 64 threads' worth of them each
    const int Cy = y256 ? L::CY : lines_per_block(ny, sizeof(R) == 4 ? 256 : 128, nxh);
    const int Cz = z256 ? L::CZ : lines_per_block(nz, 64, nxh);
    auto log2i = [](int n) { int l = 0; while ((1 << l) < n) ++l; return l; };
    const size_t smem_x = (size_t)RP * (x256 ? L::ROW : padded_len(nx) + 1) * sizeof(T);
    const size_t smem_y = (y256 ? (size_t)padded_line<256>() * L::YS : (size_t)padded_len(ny) * (Cy + 1)) * sizeof(T);
    const size_t smem_z = ((z256 ? (size_t)3 * padded_line<256>() * L::ZS : (size_t)3 * padded_len(nz) * (Cz + 1)) + nz) *
                          sizeof(T);
    const dim3 gx(ny / 2 / RP, nz, 3 * B), gy((nxh + Cy - 1) / Cy, nz, 3 * B),
        gz((nxh + Cz - 1) / Cz, ny, B);
    const unsigned tx = block_threads(RP, nx), ty = block_threads(Cy, ny), tz = block_threads(3 * Cz, nz);
    auto mark = [&](int i) { if (marks) cudaEventRecord(marks[i], st); };
    mark(0);
    rhs<<<gx, tx, smem_x, st>>>(a, g, RP);
    mark(1);
    yf<<<gy, ty, smem_y, st>>>(a.spec, a.twf[1], g, log2i(Cy));
    mark(2);
    zs<<<gz, tz, smem_z, st>>>(a, g, log2i(Cz));
    mark(3);
    yi<<<gy, ty, smem_y, st>>>(a.spec, a.twf[1], g, log2i(Cy));
    mark(4);
    c2r<<<gx, tx, smem_x, st>>>(a, g, RP);
    mark(5);
    return cudaGetLastError();
}
template cudaError_t launch_fluid<float>(cudaStream_t, int, const GridGeo&,
                                         const FluidArgs<float>&, cudaEvent_t*);
template cudaError_t launch_fluid<double>(cudaStream_t, int, const GridGeo&,
                                          const FluidArgs<double>&, cudaEvent_t*);

}  // namespace mbk
