// Fluid update of FP64 grids in three passes over HBM (sides of up to 128 cells): the same
// plane / z / plane pipeline as kernels_fft3.cu, in complex double-float arithmetic on packed
// float pairs (dpack.cuh).
//
// The line transforms are radix-4 (one radix-2 stage when log2 n is odd), in place in shared
// memory, one loop over the stages: the forward ones by decimation in frequency leave the
// frequencies in digit-reversed positions, the inverse ones by decimation in time take them
// there, and everything between (separation of packed real rows, solve) works on positions, so
// nothing is reordered.  A thread holds four points, so a plane has as many threads at work as
// it has points / 4, and a kernel is a few KiB of code.  The unrolled register transforms that
// these passes used before (16 points a thread, every size in one kernel of 550-590 KiB) were
// bound by instruction fetch: ncu showed "no instruction" as the largest or second-largest
// stall at every size, a 32^3 plane pass took 37 us with a handful of warps at work.
// Now the FP32 pipes bound them (ncu at 128^3: math-pipe throttle, 48-56% issue of two-cycle
// instructions).  Launch times (ncu), plane forward / z / plane inverse: 32^3 37.3 / 35.4 / 34.1
// -> 11.8 / 9.5 / 8.5 us, 64^3 47.8 / 40.4 / 50.5 -> 21.2 / 18.7 / 24.3 us, 128^3 254 / 197 / 179
// -> 165 / 100 / 133 us (forward 8 us more with the centre in the sum, below).  The error against 64 bits stays what it was (1.04e-14 at 128^3).
//
// Shared layout of a plane: packed row p holds nx values, stride S = nx + 5; after the
// separation the even row's columns at k and the odd row's at nx/2 + 4 + k.  Consecutive lanes
// take consecutive lines: rows differ by S = 5 (mod 8) 16-byte slots, columns by one, so the
// eight lanes of a 128-byte access fall on different banks in every stage.
#include "mb_internal.cuh"
#include "fft_lines.cuh"
#include "dpack.cuh"

namespace mbk {

namespace {

// Frequency at position p of a digit-reversed line of 2^L points (base-4 digits, one last base-2
// digit when L is odd), and the position of a frequency.
__device__ __forceinline__ int swap_pairs(int r, int L)
{
    const int m = (1 << (L & ~1)) - 1, lo = r & m;
    return (r & ~m) | ((lo & 0x55) << 1) | ((lo >> 1) & 0x55);
}
__device__ __forceinline__ int freq_of(int p, int L) { return swap_pairs((int)(__brev((unsigned)p) >> (32 - L)), L); }
__device__ __forceinline__ int pos_of(int k, int L) { return (int)(__brev((unsigned)swap_pairs(k, L)) >> (32 - L)); }

// Twiddles W_n^j = exp(-2 pi i j / n), expanded for packed products.
struct __align__(16) Tw {
    dr re, im;
};
__device__ __forceinline__ void load_tw(Tw* dst, const void* table, int n)
{
    const float4* t = static_cast<const float4*>(table);     // {re.hi, re.lo, im.hi, im.lo}
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        const float4 w = t[i];
        dst[i] = Tw{dr{pk(w.x, w.x), pk(w.y, w.y)}, dr{pk(w.z, w.z), pk(w.w, w.w)}};
    }
}

// In-place transforms of LINES = 2^lines_log (or `lines`) lines of n = 2^L points; element j of
// line l at P[at(l, j)].  Ends with a block barrier.
template <bool INV, typename Line, typename At>
__device__ __forceinline__ void lines64(dc* P, int items, int L, const Tw* tw, Line line, At at)
{
    auto radix2 = [&]() {
        for (int i = threadIdx.x; i < 2 * items; i += blockDim.x) {
            int l, j;
            line(i, l, j);
            dc* a = P + at(l, 2 * j);
            dc* b = P + at(l, 2 * j + 1);
            const dc u = *a, v = *b;
            *a = cadd(u, v);
            *b = csub(u, v);
        }
        __syncthreads();
    };
    if (INV && (L & 1)) radix2();
    for (int s = 0; s < (L >> 1); ++s) {
        // log2 of the quarter of this stage's sub-lines
        const int lq = INV ? (L & 1) + 2 * s : L - 2 - 2 * s, q = 1 << lq;
#pragma unroll 1
        for (int i = threadIdx.x; i < items; i += blockDim.x) {
            int l, t;
            line(i, l, t);                       // t < n / 4
            const int j = t & (q - 1), b = ((t >> lq) << (lq + 2)) + j;
            // twiddle index of W_{4q}^j; j = 0 needs none (a warp's lanes are lines, so they share
            // j where there are 32 of them: 44% of the products of 64-point lines, 22% of 128)
            const int w = j << (L - 2 - lq);
            dc* p0 = P + at(l, b);
            dc* p1 = P + at(l, b + q);
            dc* p2 = P + at(l, b + 2 * q);
            dc* p3 = P + at(l, b + 3 * q);
            dc a0 = *p0, a1 = *p1, a2 = *p2, a3 = *p3;
            if (INV && j != 0) {
                const Tw w1 = tw[w], w2 = tw[2 * w], w3 = tw[3 * w];
                a1 = cmulc(a1, w1.re, w1.im);
                a2 = cmulc(a2, w2.re, w2.im);
                a3 = cmulc(a3, w3.re, w3.im);
            }
            const dc s0 = cadd(a0, a2), d0 = csub(a0, a2), s1 = cadd(a1, a3), d1 = crot(csub(a1, a3));
            *p0 = cadd(s0, s1);
            // forward: d0 - i d1 to position 1, d0 + i d1 to 3; inverse the other way round
            dc y1 = INV ? cadd(d0, d1) : csub(d0, d1), y3 = INV ? csub(d0, d1) : cadd(d0, d1);
            dc y2 = csub(s0, s1);
            if (!INV && j != 0) {
                const Tw w1 = tw[w], w2 = tw[2 * w], w3 = tw[3 * w];
                y1 = cmul(y1, w1.re, w1.im);
                y2 = cmul(y2, w2.re, w2.im);
                y3 = cmul(y3, w3.re, w3.im);
            }
            *p1 = y1;
            *p2 = y2;
            *p3 = y3;
        }
        __syncthreads();
    }
    if (!INV && (L & 1)) radix2();
}

__host__ __device__ inline int plane_stride(int nx) { return nx + 5; }
__host__ __device__ inline int odd_offset(int nx) { return nx / 2 + 4; }

template <bool INV> __device__ __forceinline__ void plane_rows(dc* P, int nx, int ny, int lx, const Tw* tw)
{
    const int ll = 30 - __clz(ny), lines = ny >> 1, S = plane_stride(nx);     // log2(ny / 2)
    lines64<INV>(P, lines * (nx >> 2), lx, tw,
                 [=](int i, int& l, int& t) { l = i & (lines - 1); t = i >> ll; },
                 [=](int l, int j) { return l * S + j; });
}
template <bool INV> __device__ __forceinline__ void plane_cols(dc* P, int nx, int ny, int ly, const Tw* tw)
{
    const int ll = 30 - __clz(nx), lines = nx >> 1, S = plane_stride(nx), H = odd_offset(nx);
    lines64<INV>(P, lines * (ny >> 2), ly, tw,
                 [=](int i, int& l, int& t) { l = i & (lines - 1); t = i >> ll; },
                 [=](int l, int y) { return (y >> 1) * S + ((y & 1) ? H : 0) + l; });
}

}  // namespace

// Pass A: right-hand side and 2-D R2C transform of one (box, component, z) plane.  Half of the
// Laplacian's neighbours (z and the outer y) and -6 times the centre are summed on the FP64 pipe, six
// instructions a row pair, while the FP32 pipes convert and add the rest in double-float: all of it
// in FP64 would hold this phase for 41k cycles a 128 x 128 plane, all of it in double-float for 24k.
// The centre goes in before the sum is scaled: with a weight of rho/dt - 3 eta/h^2 for the centre
// instead, the roundings of the weights did not cancel on smooth fields and scaled every low mode
// the same way each step (1.2e-12 at eta dt / (rho h^2) = 183; 4e-15 to 2e-14 now, for 8 us of a dense 128^3 step of 900).
__global__ void __launch_bounds__(1024, 1)
k_plane_fwd64(FluidArgs<double> a, GridGeo g)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int nx = g.n[0], ny = g.n[1], nz = g.n[2], nxh = nx / 2 + 1;
    const int lx = 31 - __clz(nx), ly = 31 - __clz(ny);
    const int S = plane_stride(nx), H = odd_offset(nx);
    dc* P = reinterpret_cast<dc*>(smem_raw);
    Tw* twx = reinterpret_cast<Tw*>(P + (ny / 2) * S);
    Tw* twy = twx + nx;
    load_tw(twx, a.twk[0], nx);
    load_tw(twy, a.twk[1], ny);
    dep_wait();
    dep_release();
    const int z = blockIdx.x, bc = blockIdx.y, comp = bc % 3;
    const size_t plane = (size_t)ny * nx;
    const double* vz = a.v + (size_t)bc * g.N + z * plane;
    const double* vzp = a.v + (size_t)bc * g.N + ((z + 1) & (nz - 1)) * plane;
    const double* vzm = a.v + (size_t)bc * g.N + ((z - 1) & (nz - 1)) * plane;
    const double* f = a.f ? a.f + (size_t)bc * g.N + z * plane : nullptr;
    double* fclr = a.f_clear && f ? a.f_clear + (size_t)bc * g.N + z * plane : nullptr;
    const bool body = a.body_prof && comp == a.body_axis;
    const dfloat rho_dt(a.rho_dt), beta(a.half_eta * a.inv_h2);
    for (int i = threadIdx.x; i < (ny / 2) * nx; i += blockDim.x) {
        const int x = i & (nx - 1), p = i >> lx;
        const int o0 = 2 * p * nx + x, o1 = o0 + nx;
        double r0 = 0.0, r1 = 0.0;
        if (f) {
            r0 = f[o0];
            r1 = f[o1];
        }
        if (body) {
            r0 += a.body_prof[a.body_dir == 0 ? x : (a.body_dir == 1 ? 2 * p : z)];
            r1 += a.body_prof[a.body_dir == 0 ? x : (a.body_dir == 1 ? 2 * p + 1 : z)];
        }
        if (a.no_v) {                     // Stokes limit: the force density alone
            P[p * S + x] = dc_make(dfloat(r0), dfloat(r1));
            continue;
        }
        const int xm = ((x - 1) & (nx - 1)) - x, xp = ((x + 1) & (nx - 1)) - x;
        const int om = ((2 * p - 1) & (ny - 1)) * nx + x, op = ((2 * p + 2) & (ny - 1)) * nx + x;
        const double c0 = vz[o0], c1 = vz[o1];
        const double s0 = fma(-6.0, c0, (vzp[o0] + vzm[o0]) + vz[om]);
        const double s1 = fma(-6.0, c1, (vzp[o1] + vzm[o1]) + vz[op]);
        const dc cc = dc_make(dfloat(c0), dfloat(c1));
        // the row pair's other row: c1 is a neighbour of row 0, c0 of row 1
        dc lap = cadd(dc_make(dfloat(s0), dfloat(s1)), cswap(cc));
        lap = cadd(lap, cadd(dc_make(dfloat(vz[o0 + xm]), dfloat(vz[o1 + xm])),
                             dc_make(dfloat(vz[o0 + xp]), dfloat(vz[o1 + xp]))));
        dc v = cadd(cscale(cc, dr_make(rho_dt)), cscale(lap, dr_make(beta)));
        if (f || body) v = cadd(v, dc_make(dfloat(r0), dfloat(r1)));
        P[p * S + x] = v;
    }
    __syncthreads();
    // leave f zeroed for the next accumulation (after the plane's loads: stores between them
    // held them back, 410 against 165 us at 128^3)
    if (fclr)
        for (int i = threadIdx.x; i < ny * nx / 2; i += blockDim.x)
            reinterpret_cast<double2*>(fclr)[i] = make_double2(0.0, 0.0);
    plane_rows<false>(P, nx, ny, lx, twx);
    // the two real rows of each packed row, one warp per row, in place: X_2p[k] = (Z_k +
    // conj Z_-k)/2 to slot k, X_2p+1[k] = -i (Z_k - conj Z_-k)/2 to slot H + k, k < nx/2.
    // Columns 0 and nx/2 are real: column 0 carries X[0] + i X[nx/2]
    {
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
        for (int p = warp; p < ny / 2; p += nw) {
            dc* row = P + p * S;
            dc ev[2], od[2];
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                const int k = lane + 32 * r;
                if (k >= nx / 2) continue;
                const dc Z = row[pos_of(k, lx)], Zr = row[pos_of(k == 0 ? nx / 2 : nx - k, lx)];
                if (k == 0) {
                    ev[r] = dc_make(dc_x(Z), dc_x(Zr));
                    od[r] = dc_make(dc_y(Z), dc_y(Zr));
                } else {
                    const dc c0 = cconj(Zr);
                    ev[r] = chalf(cadd(Z, c0));
                    const dc d = crot(chalf(csub(c0, Z)));       // -i (Z - conj Zr) / 2
                    od[r] = d;
                }
            }
            __syncwarp();
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                const int k = lane + 32 * r;
                if (k >= nx / 2) continue;
                row[k] = ev[r];
                row[H + k] = od[r];
            }
        }
    }
    __syncthreads();
    plane_cols<false>(P, nx, ny, ly, twy);
    dc* out = reinterpret_cast<dc*>(a.spec) + ((size_t)bc * nz + z) * (size_t)nxh * ny;
    auto elem = [=](int k, int y) { return P[(y >> 1) * S + ((y & 1) ? H : 0) + k]; };
    for (int i = threadIdx.x; i < nxh * ny; i += blockDim.x) {
        const int k = i >> ly, y = i & (ny - 1);         // y: position of the frequency
        dc v;
        if (k == 0 || k == nx / 2) {
            // A = FFT X[0] = (Z_k + conj Z_-k) / 2,  B = FFT X[nx/2] = (Z_k - conj Z_-k) / (2i)
            const dc Z = elem(0, y);
            const dc Zr = cconj(elem(0, pos_of((ny - freq_of(y, ly)) & (ny - 1), ly)));
            v = k == 0 ? chalf(cadd(Z, Zr)) : crot(chalf(csub(Zr, Z)));
        } else {
            v = elem(k, y);
        }
        out[i] = v;
    }
}

// Pass B: FFT along z of all three components, divide, projection, k = 0 mode, inverse FFT along
// z; C columns (positions of ky) at one kx of one box.
template <int C>
__global__ void __launch_bounds__(384, 2)
k_zsolve64(FluidArgs<double> a, GridGeo g)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int nx = g.n[0], ny = g.n[1], nz = g.n[2], nxh = nx / 2 + 1;
    const int lz = 31 - __clz(nz), ly = 31 - __clz(ny);
    constexpr int LC = C == 8 ? 3 : 2;
    dc* Bf = reinterpret_cast<dc*>(smem_raw);              // [3][nz][C]
    Tw* twz = reinterpret_cast<Tw*>(Bf + 3 * nz * C);
    load_tw(twz, a.twk[2], nz);
    dep_wait();
    dep_release();
    const int yp0 = blockIdx.x * C, kx = blockIdx.y, box = blockIdx.z;
    const size_t zstride = (size_t)nxh * ny, cstride = (size_t)nz * zstride;
    dc* base = reinterpret_cast<dc*>(a.spec) + (size_t)(box * 3) * cstride + (size_t)kx * ny + yp0;
    const int total = 3 * nz * C;
    for (int i = threadIdx.x; i < total; i += blockDim.x) {
        const int k = i & (C - 1), z = (i >> LC) & (nz - 1), c = i >> (LC + lz);
        const unsigned d = (unsigned)__cvta_generic_to_shared(Bf + i);
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d),
                     "l"(base + c * cstride + (size_t)z * zstride + k) : "memory");
    }
    async_wait_all();
    __syncthreads();
    // line l = (component, column): consecutive lanes take the C columns of one z
    auto line = [=](int i, int& l, int& t) {
        const int r = i >> LC;
        l = (i & (C - 1)) | ((r % 3) << LC);
        t = r / 3;
    };
    auto at = [=](int l, int z) { return (((l >> LC) * nz + z) << LC) + (l & (C - 1)); };
    lines64<false>(Bf, 3 * C * (nz >> 2), lz, twz, line, at);
    const float2* sym = reinterpret_cast<const float2*>(a.symk);    // [9][256] cos, sin, lambda
    auto S = [=](int t, int k) { const float2 s = __ldg(sym + t * 256 + k); return dfloat(s.x, s.y); };
    const dfloat ih(a.inv_h), rho_dt(a.rho_dt), half_eta(a.half_eta), one(1.0f, 0.0f);
    for (int i = threadIdx.x; i < nz * C; i += blockDim.x) {
        const int k = i & (C - 1), zp = i >> LC;
        const int kz = freq_of(zp, lz), ky = freq_of(yp0 + k, ly);
        const dfloat lam = S(2, kx) + S(5, ky) + S(8, kz);
        const bool zero = kx == 0 && ky == 0 && kz == 0;
        dc W[3];
        const dr cinv = dr_make(recip(rho_dt + half_eta * lam));
#pragma unroll
        for (int c = 0; c < 3; ++c) W[c] = cscale(Bf[((c * nz + zp) << LC) + k], cinv);
        if (zero) {
            for (int c = 0; c < 3; ++c) {
                if (a.mean_state) {              // the only thread of this box at k = 0
                    double m = a.mean_state[3 * box + c];
                    if (a.mean_force) m += a.mean_scale * a.mean_force[3 * box + c];
                    a.mean_state[3 * box + c] = m;
                    W[c] = dc_make(dfloat((double)g.N * m), dfloat(0.0f, 0.0f));
                } else if (a.mean_override) {
                    W[c] = dc_make(dfloat((double)g.N * a.mean_override[3 * box + c]),
                                   dfloat(0.0f, 0.0f));
                } else if (a.mean_mode == 1) {
                    W[c] = dc{0ull, 0ull};
                }
            }
        } else {
            // D_a = (e^{i th} - 1)/h, G_a = (1 - e^{-i th})/h = -conj(D_a), D.G = -lambda:
            // P W = W + G (D.W) / lambda
            const int kk[3] = {kx, ky, kz};
            dr Dr[3], Di[3];
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                Dr[c] = dr_make((S(3 * c, kk[c]) - one) * ih);
                Di[c] = dr_make(S(3 * c + 1, kk[c]) * ih);
            }
            dc d = cadd(cadd(cmul(W[0], Dr[0], Di[0]), cmul(W[1], Dr[1], Di[1])),
                        cmul(W[2], Dr[2], Di[2]));
            d = cscale(d, dr_make(recip(lam)));
#pragma unroll
            for (int c = 0; c < 3; ++c) W[c] = csub(W[c], cmulc(d, Dr[c], Di[c]));
        }
#pragma unroll
        for (int c = 0; c < 3; ++c) Bf[((c * nz + zp) << LC) + k] = W[c];
    }
    __syncthreads();
    lines64<true>(Bf, 3 * C * (nz >> 2), lz, twz, line, at);
    for (int i = threadIdx.x; i < total; i += blockDim.x) {
        const int k = i & (C - 1), z = (i >> LC) & (nz - 1), c = i >> (LC + lz);
        base[c * cstride + (size_t)z * zstride + k] = Bf[i];
    }
}

// Pass C: 2-D C2R inverse of one plane, scaled by 1/N.
__global__ void __launch_bounds__(1024, 1)
k_plane_inv64(FluidArgs<double> a, GridGeo g)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int nx = g.n[0], ny = g.n[1], nz = g.n[2], nxh = nx / 2 + 1;
    const int lx = 31 - __clz(nx), ly = 31 - __clz(ny);
    const int S = plane_stride(nx), H = odd_offset(nx);
    dc* P = reinterpret_cast<dc*>(smem_raw);
    Tw* twx = reinterpret_cast<Tw*>(P + (ny / 2) * S);
    Tw* twy = twx + nx;
    load_tw(twx, a.twk[0], nx);
    load_tw(twy, a.twk[1], ny);
    dep_wait();
    dep_release();
    const int z = blockIdx.x, bc = blockIdx.y;
    const dc* in = reinterpret_cast<const dc*>(a.spec) + ((size_t)bc * nz + z) * (size_t)nxh * ny;
    for (int i = threadIdx.x + ny; i < (nx / 2) * ny; i += blockDim.x) {
        const int k = i >> ly, y = i & (ny - 1);
        const unsigned d = (unsigned)__cvta_generic_to_shared(P + (y >> 1) * S + ((y & 1) ? H : 0) + k);
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(in + i) : "memory");
    }
    // columns 0 and nx/2 invert to real sequences: their Hermitian parts as one complex column,
    // herm(A) + i herm(B)
    for (int y = threadIdx.x; y < ny; y += blockDim.x) {
        const int yr = pos_of((ny - freq_of(y, ly)) & (ny - 1), ly);
        const dc ha = chalf(cadd(in[y], cconj(in[yr])));
        const dc* b = in + (nx / 2) * ny;
        const dc hb = chalf(cadd(b[y], cconj(b[yr])));
        P[(y >> 1) * S + ((y & 1) ? H : 0)] = cadd(ha, crot(hb));
    }
    async_wait_all();
    __syncthreads();
    plane_cols<true>(P, nx, ny, ly, twy);
    // Z = X_2p + i X_2p+1 with the Hermitian extension, to the frequencies' positions, one warp
    // per packed row
    {
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
        for (int p = warp; p < ny / 2; p += nw) {
            dc* row = P + p * S;
            dc zk[2], zr[2];
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                const int k = lane + 32 * r;
                if (k >= nx / 2) continue;
                const dc e = row[k], o = row[H + k];
                if (k == 0) {              // X[0] + i X[nx/2] of both rows
                    zk[r] = dc_make(dc_x(e), dc_x(o));
                    zr[r] = dc_make(dc_y(e), dc_y(o));
                } else {
                    zk[r] = cadd(e, crot(o));
                    zr[r] = cadd(cconj(e), crot(cconj(o)));
                }
            }
            __syncwarp();
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                const int k = lane + 32 * r;
                if (k >= nx / 2) continue;
                row[pos_of(k, lx)] = zk[r];
                row[pos_of(k == 0 ? nx / 2 : nx - k, lx)] = zr[r];
            }
        }
    }
    __syncthreads();
    plane_rows<true>(P, nx, ny, lx, twx);
    const dr scale = dr_make(dfloat(a.inv_n));       // a power of two: exact
    const size_t at = (size_t)bc * g.N + (size_t)z * ny * nx;
    double* out = a.v_out + at;
    const double* base = a.v_sum_out ? a.v_sum_base + at : nullptr;
    double* sum = a.v_sum_out + (base ? at : 0);
    for (int i = threadIdx.x; i < (ny / 2) * nx; i += blockDim.x) {
        const int x = i & (nx - 1), p = i >> lx;
        const dc v = P[p * S + x];
        const dc w = dc{mul2(v.hi, scale.hi), mul2(v.lo, scale.hi)};
        const double u0 = (double)dc_x(w), u1 = (double)dc_y(w);
        const int o = 2 * p * nx + x;
        out[o] = u0;
        out[o + nx] = u1;
        if (base) {                          // v^n + v^{n+1} for the corrector's single gather
            sum[o] = __ldg(base + o) + u0;
            sum[o + nx] = __ldg(base + o + nx) + u1;
        }
    }
}

template <>
cudaError_t launch_fluid3<double>(Chain st, int B, const GridGeo& g,
                                  const FluidArgs<double>& a_in, cudaEvent_t* marks)
{
    const FluidArgs<double> a = with_derived(a_in, g);
    const int nx = g.n[0], ny = g.n[1], nz = g.n[2], nxh = nx / 2 + 1;
    static std::atomic<unsigned> attr{0};
    if (first_on_device(attr)) {
        const int lim = 200 * 1024;
        cudaFuncSetAttribute(k_plane_fwd64, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
        cudaFuncSetAttribute(k_zsolve64<8>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
        cudaFuncSetAttribute(k_zsolve64<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
        cudaFuncSetAttribute(k_plane_inv64, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
    }
    // one thread for every four points of a plane (a stage's butterflies), whole warps
    auto threads = [](int items, int most) {
        const int t = ((items + 31) / 32) * 32;
        return t < most ? t : most;
    };
    const int tp = threads(nx * ny / 8, 1024);
    const size_t smem_p = (size_t)(ny / 2) * plane_stride(nx) * sizeof(dc) + (size_t)(nx + ny) * sizeof(Tw);
    const int C = ny >= 8 ? 8 : 4;
    const int tz = threads(3 * C * nz / 4, 384);
    const size_t smem_z = (size_t)3 * nz * C * sizeof(dc) + nz * sizeof(Tw);
    auto mark = [&](int i) { if (marks) cudaEventRecord(marks[i], st.st); };
    mark(0);
    const dim3 gp(nz, 3 * B), gz(ny / C, nxh, B);
    cudaError_t e = launch_on(st, k_plane_fwd64, gp, dim3(tp), smem_p, a, g);
    if (e != cudaSuccess) return e;
    mark(1);
    mark(2);
    e = C == 8 ? launch_on(st, k_zsolve64<8>, gz, dim3(tz), smem_z, a, g)
               : launch_on(st, k_zsolve64<4>, gz, dim3(tz), smem_z, a, g);
    if (e != cudaSuccess) return e;
    mark(3);
    mark(4);
    e = launch_on(st, k_plane_inv64, gp, dim3(tp), smem_p, a, g);
    if (e != cudaSuccess) return e;
    mark(5);
    return cudaGetLastError();
}

}  // namespace mbk
