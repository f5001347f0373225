// Blob-side kernels: interpolation J, cell binning, blob forces, tiled spreading S,
// particle velocities.
#include "mb_internal.cuh"
#include "peskin.cuh"

namespace mbk {

// ==========================================================================================
// Launch shapes of the FP64 blob kernels.  GB300 issues two FP64 lanes a cycle and SM, so these
// kernels are bound by that pipe on every SM they reach, and below a few thousand blobs by the
// latency of one thread's chain: few blobs are spread over as many SMs as there are warps.
// Blocks of 32 threads up to 16384 blobs (512 blocks, over three for each SM), larger ones
// after that; a thread per blob and component (split) up to 4096 blobs, where the 3 x 128
// warps still fit one or two an SM: 832 blobs at 64^3, predictor 26.8 -> 5.0 us.
inline int blob_block(int64_t nb) { return nb <= 16384 ? 32 : 128; }
inline bool split_components(int64_t nb) { return nb <= 4096; }
inline unsigned blocks_of(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }

__device__ __forceinline__ int bin_coord(double x, double inv_w, int nc)
{
    int c = (int)floor(x * inv_w);
    if (c >= nc) c -= nc;
    if (c < 0) c += nc;
    if (c < 0 || c >= nc) c = 0;   // non-finite position: keep every index in bounds
    return c;
}

// Counts a blob at p into its bin cell; its rank there is its place in the cell.
__device__ __forceinline__ void count_blob(const BinCount& c, int64_t b, int box, const double* p)
{
    const int cx = bin_coord(p[0], c.bg.inv_w, c.bg.nc[0]);
    const int cy = bin_coord(p[1], c.bg.inv_w, c.bg.nc[1]);
    const int cz = bin_coord(p[2], c.bg.inv_w, c.bg.nc[2]);
    const int cell = (int)(box * c.bg.ncell + ((int64_t)cz * c.bg.nc[1] + cy) * c.bg.nc[0] + cx);
    c.blob_cell[b] = cell;
    c.blob_rank[b] = atomicAdd(c.count + cell, 1);
}

// Sum over a blob's 27 nodes of the weights times c0 (+ c1 with TWO).
template <bool TWO, typename R>
__device__ __forceinline__ R window_sum(const R* __restrict__ c0, const R* __restrict__ c1,
                                        const Win<R>& wx, const Win<R>& wy, const Win<R>& wz)
{
    R acc = R(0);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        R plane = R(0);
#pragma unroll
        for (int bb = 0; bb < 3; ++bb) {
            const int row = wz.o[c] + wy.o[bb];
            R r = R(0);
#pragma unroll
            for (int aa = 0; aa < 3; ++aa) {
                R val = __ldg(c0 + (row + wx.o[aa]));
                if (TWO) val += __ldg(c1 + (row + wx.o[aa]));
                r += wx.w[aa] * val;
            }
            // FP64: products summed by rows and planes (39 instructions instead of 45)
            if constexpr (sizeof(R) == 8) plane += wy.w[bb] * r;
            else acc += wy.w[bb] * wz.w[c] * r;
        }
        if constexpr (sizeof(R) == 8) acc += wz.w[c] * plane;
    }
    return acc;
}

// Interpolation J (Eq. ju): u_a = sum over the 3x3x3 window of Phi Phi Phi v_a(node), each
// component on its own staggered grid.  One thread per blob, its windows at both MAC shifts
// computed once per dimension (6 instead of 9); with SPLIT one per blob and component, three
// windows each.  TWO: the sum of v0 and v1, otherwise v0 alone, times `scale`.  WRAP: positions from
// anywhere.  With `count` the new position is counted into its bin cell.
struct InterpArgs {
    int64_t nb;
    const double* q;
    const double* q_base;
    const int32_t* box_of;
    double dt;
    double scale;              // of the gathered sums
    double* u_out;
    double* q_out;
    BinCount bin;
};

template <typename R, int MODE, bool SPLIT, bool WRAP, bool TWO>
__global__ void __launch_bounds__(128)
k_interp(InterpArgs a, const R* __restrict__ v0, const R* __restrict__ v1, GridGeo g)
{
    dep_wait();
    dep_release();
    __shared__ double moved[MODE == 1 && SPLIT ? 96 : 1];       // [32 blobs][3]
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    int64_t b = SPLIT ? t / 3 : t;
    const int mine = SPLIT ? (int)(t - 3 * b) : 0;
    const bool live = b < a.nb;
    if (!live) {
        if (!(MODE == 1 && SPLIT)) return;
        b = a.nb - 1;                      // stays for the block's barrier, stores nothing
    }
    const int box = a.box_of ? a.box_of[b] : 0;
    double p[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        p[d] = a.q[3 * b + d];
        if (WRAP) p[d] = wrap_any(p[d], g.L[d]);
    }
    const int nx = g.n[0], ny = g.n[1], nz = g.n[2];
    const int mask[3] = {nx - 1, ny - 1, nz - 1}, stride[3] = {1, nx, ny * nx};
    double u[3] = {0.0, 0.0, 0.0};
    const double unit = a.scale * Win<R>::UNIT;
    if (SPLIT) {
        Win<R> w[3];
#pragma unroll
        for (int d = 0; d < 3; ++d)
            w[d].set(p[d] * g.inv_h - (d == mine ? 0.0 : 0.5), mask[d], stride[d]);
        const size_t base = ((size_t)box * 3 + mine) * (size_t)g.N;
        const R acc = window_sum<TWO>(v0 + base, TWO ? v1 + base : nullptr, w[0], w[1], w[2]);
        u[0] = unit * (double)acc;
    } else {
        Win<R> own[3], across[3];
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            own[d].set(p[d] * g.inv_h - 0.0, mask[d], stride[d]);
            across[d].set(p[d] * g.inv_h - 0.5, mask[d], stride[d]);
        }
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const size_t base = ((size_t)box * 3 + c) * (size_t)g.N;
            const R acc = window_sum<TWO>(v0 + base, TWO ? v1 + base : nullptr,
                                          c == 0 ? own[0] : across[0], c == 1 ? own[1] : across[1],
                                          c == 2 ? own[2] : across[2]);
            u[c] = unit * (double)acc;
        }
    }
    // position updates round like the plain expression q + (c dt) u (no contraction)
    double nq[3] = {0.0, 0.0, 0.0};
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        if ((SPLIT && c > 0) || !live) break;
        const int d = SPLIT ? mine : c;
        if (a.u_out) a.u_out[3 * b + d] = u[c];
        if (MODE == 0) continue;
        const double base = MODE == 1 ? (SPLIT ? (mine == 0 ? p[0] : mine == 1 ? p[1] : p[2]) : p[c])
                                      : a.q_base[3 * b + d];
        nq[c] = wrap_position(__dadd_rn(base, __dmul_rn(MODE == 1 ? 0.5 * a.dt : a.dt, u[c])), g.L[d]);
        a.q_out[3 * b + d] = nq[c];
    }
    if (MODE == 1 && a.bin.count) {
        if constexpr (SPLIT) {
            moved[threadIdx.x] = nq[0];
            __syncthreads();
            const int64_t mb = (int64_t)blockIdx.x * 32 + threadIdx.x;
            if (threadIdx.x < 32 && mb < a.nb)
                count_blob(a.bin, mb, a.box_of ? a.box_of[mb] : 0, moved + 3 * threadIdx.x);
        } else {
            count_blob(a.bin, b, box, nq);
        }
    }
}

template <typename R>
cudaError_t launch_interp(Chain st, int mode, int64_t nb, const double* q,
                          const double* q_base, const R* v0, const R* v1,
                          const int32_t* box_of, const GridGeo& g, double dt, double* u_out,
                          double* q_out, bool wrap, const BinCount* bin, double scale)
{
    if (nb <= 0) return cudaSuccess;
    InterpArgs a{nb, q, q_base, box_of, dt, scale, u_out, q_out, bin ? *bin : BinCount{}};
    const bool split = split_components(nb);
    const int T = split ? 96 : blob_block(nb);           // split: 32 blobs a block
    const unsigned blocks = blocks_of(split ? 3 * nb : nb, T);
    auto go = [&](auto k) { return launch_on(st, k, dim3(blocks), dim3(T), 0, a, v0, v1, g); };
    if (mode == 0) {
        if (wrap) return split ? go(k_interp<R, 0, true, true, false>) : go(k_interp<R, 0, false, true, false>);
        return split ? go(k_interp<R, 0, true, false, false>) : go(k_interp<R, 0, false, false, false>);
    }
    if constexpr (sizeof(R) == 4) {
        return cudaErrorInvalidValue;                    // FP32 grids move blobs in kernels_blob32.cu
    } else {
        if (mode == 1) {
            if (wrap) return split ? go(k_interp<R, 1, true, true, false>) : go(k_interp<R, 1, false, true, false>);
            return split ? go(k_interp<R, 1, true, false, false>) : go(k_interp<R, 1, false, false, false>);
        }
        if (v1) return split ? go(k_interp<R, 2, true, false, true>) : go(k_interp<R, 2, false, false, true>);
        return split ? go(k_interp<R, 2, true, false, false>) : go(k_interp<R, 2, false, false, false>);
    }
}
template cudaError_t launch_interp<float>(Chain, int, int64_t, const double*,
                                          const double*, const float*, const float*,
                                          const int32_t*, const GridGeo&, double, double*,
                                          double*, bool, const BinCount*, double);
template cudaError_t launch_interp<double>(Chain, int, int64_t, const double*,
                                           const double*, const double*, const double*,
                                           const int32_t*, const GridGeo&, double, double*,
                                           double*, bool, const BinCount*, double);

// ==========================================================================================
// Cell binning (counting sort of blobs by bin cell, box-major): counts (by the predictor or
// k_bin_count), the scan of kernels_blob32.cu, and the placement.
__global__ void k_bin_count(int64_t nb, const double* __restrict__ q,
                            const int32_t* __restrict__ box_of, BinCount c)
{
    dep_wait();
    dep_release();
    const int64_t b = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (b >= nb) return;
    const double p[3] = {q[3 * b], q[3 * b + 1], q[3 * b + 2]};
    count_blob(c, b, box_of ? box_of[b] : 0, p);
}

// The position of blob b (of bin cell `cell`) relative to the lower corner of its cell (FP32,
// |x| < cell side) and its particle id, for the FP32 prefilter of the pair search.
__device__ __forceinline__ float4 cell_local(int b, int cell, const double* __restrict__ q,
                                             const int32_t* __restrict__ pid, const BinGeo& bg)
{
    const int local = (int)(cell % bg.ncell);
    const int c[3] = {local % bg.nc[0], (local / bg.nc[0]) % bg.nc[1],
                      local / (bg.nc[0] * bg.nc[1])};
    float r[3];
    for (int d = 0; d < 3; ++d) r[d] = (float)(q[3 * b + d] - c[d] * bg.w);
    return make_float4(r[0], r[1], r[2], __int_as_float(pid ? pid[b] : 0));
}

// Cell starts from the scan's two levels, and every blob's slot.
__global__ void __launch_bounds__(256)
k_bin_place(int64_t nb, int64_t ncells, const int32_t* __restrict__ local,
            const int32_t* __restrict__ tile_off, int32_t* __restrict__ cell_start,
            const int32_t* __restrict__ blob_cell, const int32_t* __restrict__ blob_rank,
            int32_t* __restrict__ sorted, const double* __restrict__ q,
            const int32_t* __restrict__ pid, BinGeo bg, float4* __restrict__ loc)
{
    dep_wait();
    dep_release();
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < ncells) cell_start[i] = local[i] + tile_off[i >> BIN_SCAN_LOG];
    if (i < nb) {
        const int cell = blob_cell[i];
        const int slot = local[cell] + tile_off[cell >> BIN_SCAN_LOG] + blob_rank[i];
        sorted[slot] = (int32_t)i;
        if (loc) loc[slot] = cell_local((int)i, cell, q, pid, bg);
    }
}

// Deterministic order inside each cell: ascending blob index (cells hold a handful of blobs),
// then the cell-local coordinates in that order.
__global__ void k_cell_order(int64_t ncells, const int32_t* __restrict__ cell_start,
                             int32_t* __restrict__ sorted, const double* __restrict__ q,
                             const int32_t* __restrict__ pid, BinGeo bg, float4* __restrict__ loc)
{
    dep_wait();
    dep_release();
    const int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (c >= ncells) return;
    const int s = cell_start[c], e = cell_start[c + 1];
    for (int i = s + 1; i < e; ++i) {
        const int32_t key = sorted[i];
        int j = i - 1;
        while (j >= s && sorted[j] > key) {
            sorted[j + 1] = sorted[j];
            --j;
        }
        sorted[j + 1] = key;
    }
    for (int i = s; i < e; ++i) loc[i] = cell_local(sorted[i], (int)c, q, pid, bg);
}

cudaError_t launch_bin(Chain st, int64_t nb, const double* q, const int32_t* box_of,
                       int B, const BinCount& c, int32_t* cell_start, int32_t* sorted,
                       int32_t* scan_tmp, bool ordered, const int32_t* pid, float4* loc,
                       bool counted)
{
    const BinGeo& bg = c.bg;
    const int64_t ncells = (int64_t)B * bg.ncell;
    cudaError_t e;
    if (!counted) {
        e = cudaMemsetAsync(c.count, 0, sizeof(int32_t) * ncells, st.st);
        if (e != cudaSuccess) return e;
        if (nb > 0) {
            e = launch_on(st, k_bin_count, dim3(blocks_of(nb, 256)), dim3(256), 0, nb, q, box_of, c);
            if (e != cudaSuccess) return e;
        }
    }
    e = launch_bin_scan(st, c.count, ncells, scan_tmp, cell_start + ncells);
    if (e != cudaSuccess) return e;
    e = launch_on(st, k_bin_place, dim3(blocks_of(nb > ncells ? nb : ncells, 256)), dim3(256), 0,
                   nb, ncells, (const int32_t*)c.count, (const int32_t*)scan_tmp, cell_start,
                   (const int32_t*)c.blob_cell, (const int32_t*)c.blob_rank, sorted, q, pid, bg,
                   ordered ? (float4*)nullptr : loc);
    if (e == cudaSuccess && ordered)
        e = launch_on(st, k_cell_order, dim3(blocks_of(ncells, 256)), dim3(256), 0, ncells,
                       (const int32_t*)cell_start, sorted, q, pid, bg, loc);
    return e;
}

// ==========================================================================================
// Blob forces (FP64): harmonic bonds from a per-blob adjacency list, soft repulsion between
// blobs of different particles found through the bin cells, external forces.
// One thread per sorted slot; the grid is (chunks, boxes) so block partial sums stay per box.

__device__ __forceinline__ void block_sum3(double v[3], double* sh /*[3][32]*/)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        double x = v[a];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
        if (lane == 0) sh[a * 32 + warp] = x;
    }
    __syncthreads();
    if (warp == 0) {
        const int nw = blockDim.x >> 5;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            double x = lane < nw ? sh[a * 32 + lane] : 0.0;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
            if (lane == 0) v[a] = x;
        }
    }
}

// The nearest image of a difference beyond half the box: one box on, or more where a midpoint moved
// by more than the box.  Not inlined: as predicated instructions its comparisons and additions
// would take the FP64 pipe for every bond.
__device__ __noinline__ double other_image(double x, double L)
{
    const double half = 0.5 * L;
    if (fabs(x) >= L) return __dsub_rn(x, __dmul_rn(L, rint(__ddiv_rn(x, L))));
    return x > half ? __dsub_rn(x, L) : (x < -half ? __dadd_rn(x, L) : x);
}

// Spring force on blob b from bond (b, j): -k (|r| - r0) r/|r|, r = q_b - q_j (minimum image),
// in FP64 with the operations in the plain order and no contraction, so that a blob's spring
// force is the same bits however the work is scheduled.
__device__ __forceinline__ void spring_force(const double* __restrict__ qb,
                                             const double* __restrict__ qj, double r0, double k,
                                             const double L[3], double f[3])
{
    double r[3];
    for (int d = 0; d < 3; ++d) {
        double x = __dsub_rn(qb[d], qj[d]);
        // beyond half the box (by the high words; exactly below): the other image
        if ((__double2hiint(x) & 0x7fffffff) >= __double2hiint(L[d]) - (1 << 20))
            x = other_image(x, L[d]);
        r[d] = x;
    }
    const Length l(__dadd_rn(__dadd_rn(__dmul_rn(r[0], r[0]), __dmul_rn(r[1], r[1])),
                             __dmul_rn(r[2], r[2])));
    const double mag = l.divide(__dmul_rn(-k, __dsub_rn(l.len, r0)));
    for (int d = 0; d < 3; ++d) f[d] = __dmul_rn(mag, r[d]);
}

// Repulsion k_rep (r_cut - |r|) r/|r| for |r| < r_cut, r = q_b - q_j.
__device__ __forceinline__ void pair_term(const double qb[3], const double* __restrict__ qj,
                                          double k_rep, double r_cut, const double L[3],
                                          double Fp[3])
{
    double r[3];
    for (int d = 0; d < 3; ++d) r[d] = min_image(__dsub_rn(qb[d], qj[d]), L[d]);
    const double r2 = __dadd_rn(__dadd_rn(__dmul_rn(r[0], r[0]), __dmul_rn(r[1], r[1])),
                                __dmul_rn(r[2], r[2]));
    if (r2 >= r_cut * r_cut || r2 == 0.0) return;
    const Length l(r2);
    const double mag = l.divide(__dmul_rn(k_rep, __dsub_rn(r_cut, l.len)));
    for (int d = 0; d < 3; ++d) Fp[d] = __dadd_rn(Fp[d], __dmul_rn(mag, r[d]));
}

// FP64 springs of a bond pattern shared by all particles (launch_springs64).  A block holds
// whole particles.  Their bonds are spread evenly over its threads (an icosahedron's 42 over 13
// threads' worth: evaluated at the blobs, the fullest one's four set the pace), each evaluated
// once, as the force on its first end, into shared memory; after a barrier one thread per blob
// and component sums ext and its bonds in adjacency order, negated where it is the other end.  Negation is
// exact and the evaluation of a bond from the other end gives the negated bits, so every sum
// equals the per-blob adjacency sum of k_forces bit for bit.
__global__ void __launch_bounds__(256)
k_springs64(int np, int m, int nbond, int ppb, const double* __restrict__ q,
            const double* __restrict__ ext, const int4* __restrict__ tmpl,
            const int32_t* __restrict__ tstart, const int32_t* __restrict__ box_of,
            const double* __restrict__ box_par, GridGeo g, double* __restrict__ Fout)
{
    dep_wait();
    dep_release();
    extern __shared__ double bond_f[];                   // [ppb][nbond][3]
    const int p0 = blockIdx.x * ppb, here = min(ppb, np - p0);
    for (int i = threadIdx.x; i < here * nbond; i += blockDim.x) {
        const int p = i / nbond;
        const int4 bd = __ldg(tmpl + (i - p * nbond));
        const int base = (p0 + p) * m, a = base + (bd.x & 0xffff), b = base + (bd.x >> 16);
        const double k_spring = box_par[3 * (box_of ? box_of[a] : 0)];
        spring_force(q + 3 * a, q + 3 * b, __hiloint2double(bd.z, bd.y), k_spring, g.L, bond_f + 3 * i);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < 3 * here * m; i += blockDim.x) {      // a component of a blob
        const int j = i / 3, d = i - 3 * j, p = j / m, l = j - p * m;
        const int64_t at = 3 * (int64_t)p0 * m + i;
        double F = ext ? ext[at] : 0.0;
        const int c0 = __ldg(tstart + l), c1 = __ldg(tstart + l + 1);
        for (int e = c0; e < c1; ++e) {
            const int4 ad = __ldg(tmpl + e);
            const double v = bond_f[3 * (p * nbond + ad.x) + d];
            F = __dadd_rn(F, ad.y > 0 ? v : -v);
        }
        Fout[at] = F;
    }
}

cudaError_t launch_springs64(Chain st, int64_t nb, int m, int nbond, const double* q,
                             const double* ext, const int4* tmpl, const int32_t* tstart,
                             const int32_t* box_of, const double* box_par, const GridGeo& g,
                             double* Fout)
{
    if (nb <= 0) return cudaSuccess;
    // about a warp of blobs a block while there are few, eight warps otherwise, within the
    // 48 KiB of shared memory that need no opt-in (SPRINGS64_MAX_BONDS for one particle)
    const int most = blob_block(nb) < 128 ? 32 : 256;
    const int fit = SPRINGS64_MAX_BONDS / (nbond > 0 ? nbond : 1);
    int ppb = most / m > 1 ? most / m : 1;
    if (ppb > fit) ppb = fit;
    const int np = (int)(nb / m);
    const int threads = most == 32 ? 64 : 256;
    return launch_on(st, k_springs64, dim3(blocks_of(np, ppb)), dim3(threads),
                      sizeof(double) * 3 * (size_t)ppb * (nbond > 0 ? nbond : 1), np, m, nbond,
                      ppb, q, ext, tmpl, tstart, box_of, box_par, g, Fout);
}

// Blob forces in slot order (blob order without bins: no repulsion then).
__global__ void __launch_bounds__(256)
k_forces(ForceArgs a, GridGeo g, BinGeo bg)
{
    dep_wait();
    dep_release();
    __shared__ double sh[96];
    __shared__ bool last;
    const int box = blockIdx.y;
    const int64_t s0 = a.box_off[box], cnt = a.box_off[box + 1] - s0;
    const int64_t local = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    double F[3] = {0.0, 0.0, 0.0};
    if (local < cnt) {
        const int64_t slot = s0 + local;
        const int b = a.sorted ? a.sorted[slot] : (int)slot;
        const double qb[3] = {a.q[3 * b], a.q[3 * b + 1], a.q[3 * b + 2]};
        const double k_rep = a.box_par[3 * box + 1];
        const double r_cut = a.box_par[3 * box + 2];
        if (a.Fpre) {
            for (int d = 0; d < 3; ++d) F[d] = a.Fpre[3 * b + d];
        } else {
            if (a.ext) {
                F[0] = a.ext[3 * b];
                F[1] = a.ext[3 * b + 1];
                F[2] = a.ext[3 * b + 2];
            }
            const double k_spring = a.box_par[3 * box];
            for (int e = a.adj_start[b]; e < a.adj_start[b + 1]; ++e)
            {
                double f[3];
                spring_force(qb, a.q + 3 * a.adj_j[e], a.adj_rest[e], k_spring, g.L, f);
                for (int d = 0; d < 3; ++d) F[d] = __dadd_rn(F[d], f[d]);
            }
        }
        if (a.sorted && k_rep != 0.0 && r_cut > 0.0) {
            double Fp[3] = {0.0, 0.0, 0.0};
            const float4 lb = a.loc[slot];
            const int pb = __float_as_int(lb.w);
            const int cell = a.blob_cell[b] - (int)(box * bg.ncell);
            const int c[3] = {cell % bg.nc[0], (cell / bg.nc[0]) % bg.nc[1],
                              cell / (bg.nc[0] * bg.nc[1])};
            const float w = bg.w32;
            const float rcf = (float)r_cut;
            const float pre = rcf * rcf * 1.0001f + 1e-6f;     // conservative FP32 prefilter
            const bool wide = bg.nc[0] >= 3 && bg.nc[1] >= 3 && bg.nc[2] >= 3;
            // neighbour cells along each axis; in the wide case only those on whose side the
            // blob is within the prefilter's reach (the margin covers the rounding of loc), in
            // the order of the full search: the partners met are the same
            const float reach = sqrtf(pre) + 1e-3f * w, mine[3] = {lb.x, lb.y, lb.z};
            int lo[3], hi[3];
            for (int d = 0; d < 3; ++d) {
                if (wide) {
                    lo[d] = mine[d] < reach ? -1 : 0;
                    hi[d] = mine[d] > w - reach ? 1 : 0;
                } else if (bg.nc[d] >= 3) {
                    lo[d] = -1;
                    hi[d] = 1;
                } else {
                    lo[d] = 0;
                    hi[d] = bg.nc[d] - 1;
                }
            }
            auto nbr = [](int c0, int d, int nc) {
                if (nc < 3) return d;
                int x = c0 + d;
                x += x < 0 ? nc : 0;
                x -= x >= nc ? nc : 0;
                return x;
            };
            for (int dz = lo[2]; dz <= hi[2]; ++dz) {
                const int cz = nbr(c[2], dz, bg.nc[2]);
                for (int dy = lo[1]; dy <= hi[1]; ++dy) {
                    const int cy = nbr(c[1], dy, bg.nc[1]);
                    const int row = (int)(box * bg.ncell) + (cz * bg.nc[1] + cy) * bg.nc[0];
                    for (int dx = lo[0]; dx <= hi[0]; ++dx) {
                        const int cc = row + nbr(c[0], dx, bg.nc[0]);
                        const float ox = dx * w, oy = dy * w, oz = dz * w;
                        for (int t = a.cell_start[cc]; t < a.cell_start[cc + 1]; ++t) {
                            if (t == slot) continue;
                            const float4 lj = a.loc[t];
                            if (__float_as_int(lj.w) == pb) continue;
                            const float rf[3] = {lb.x - lj.x - ox, lb.y - lj.y - oy, lb.z - lj.z - oz};
                            if (wide && rf[0] * rf[0] + rf[1] * rf[1] + rf[2] * rf[2] > pre) continue;
                            pair_term(qb, a.q + 3 * a.sorted[t], k_rep, r_cut, g.L, Fp);
                        }
                    }
                }
            }
            for (int d = 0; d < 3; ++d) F[d] = __dadd_rn(F[d], Fp[d]);
        }
        for (int d = 0; d < 3; ++d) a.F[3 * b + d] = F[d];
    }
    if (!a.vbar) return;
    // the net force: one partial sum a block; the last block of the box to finish (atomic ticket
    // after a fence; no block waits for another) adds them in a fixed order and advances the
    // mean velocity
    block_sum3(F, sh);
    if (threadIdx.x == 0) {
        for (int d = 0; d < 3; ++d) a.partial[((int64_t)box * gridDim.x + blockIdx.x) * 3 + d] = F[d];
        __threadfence();
        last = atomicAdd(a.ticket + box, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    double s[3] = {0.0, 0.0, 0.0};
    for (int c = threadIdx.x; c < (int)gridDim.x; c += blockDim.x)
        for (int d = 0; d < 3; ++d) s[d] += __ldcg(a.partial + ((int64_t)box * gridDim.x + c) * 3 + d);
    block_sum3(s, sh);
    if (threadIdx.x == 0) {
        for (int d = 0; d < 3; ++d)
            a.vbar[3 * box + d] = a.mean_mode == 0 ? a.vbar[3 * box + d] + a.mean_scale * s[d] : 0.0;
        a.ticket[box] = 0u;
    }
}

int force_chunks(int64_t nb, int64_t max_box_blobs)
{
    const int T = blob_block(nb);
    return (int)((max_box_blobs + T - 1) / T);
}

cudaError_t launch_forces(Chain st, int B, int64_t nb, int64_t max_box_blobs,
                          const ForceArgs& a, const GridGeo& g, const BinGeo& bg)
{
    const int chunks = force_chunks(nb, max_box_blobs);
    if (chunks <= 0) return cudaSuccess;
    return launch_on(st, k_forces, dim3((unsigned)chunks, (unsigned)B), dim3(blob_block(nb)), 0, a,
                      g, bg);
}

// ==========================================================================================
// Deterministic spreading (FP64 grids): tile-owner accumulation in 64-bit fixed point.  Each CTA
// owns a TX x TY x TZ block of nodes of all three components and gathers every blob whose 3x3x3
// window can reach it from the bin cells of the block plus its halo.

__host__ __device__ __forceinline__ int floor_div(int a, int b)
{
    return a >= 0 ? a / b : -((-a + b - 1) / b);
}

__host__ __device__ __forceinline__ int wrap_cell(int c, int n)
{
    c %= n;
    return c < 0 ? c + n : c;
}

// Bin-cell window [lo, lo + cnt) along one dimension holding every blob that can touch nodes
// [T0, T0 + T): blob positions q/h in [T0 - 3/2, T0 + T + 1) (union of both MAC shifts).
__host__ __device__ __forceinline__ void halo_cells(int T0, int T, int bs, int nc, int& lo,
                                                    int& cnt)
{
    lo = floor_div(2 * T0 - 3, 2 * bs);
    const int hi = floor_div(T0 + T + 1 + bs - 1, bs) - 1;
    cnt = hi - lo + 1;
    if (cnt >= nc) {
        lo = 0;
        cnt = nc;
    }
}

// Blob-owner spreading with global atomics, straight from the caller's order: each blob adds its
// 81 node contributions into f (zeroed beforehand) with the native FP64 global atomic add, or on
// FP32 grids with two aligned 8-byte vector adds a row of three nodes (the spare node gets zero;
// nx is even, so a pair never wraps).  One thread per blob, or with SPLIT one per blob and
// component.
template <typename R, bool SPLIT, bool WRAP>
__global__ void __launch_bounds__(128)
k_spread_atomic(int64_t nb, const double* __restrict__ q, const double* __restrict__ F,
                const int32_t* __restrict__ box_of, GridGeo g, double scale, R* __restrict__ f)
{
    dep_wait();
    dep_release();
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int64_t b = SPLIT ? t / 3 : t;
    if (b >= nb) return;
    const int mine = SPLIT ? (int)(t - 3 * b) : 0;
    const int nx = g.n[0], ny = g.n[1], nz = g.n[2];
    const int mask[3] = {nx - 1, ny - 1, nz - 1}, stride[3] = {1, nx, ny * nx};
    R* fb = f + (size_t)(box_of ? box_of[b] : 0) * 3 * (size_t)g.N;
    double x[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        x[d] = q[3 * b + d];
        if (WRAP) x[d] = wrap_any(x[d], g.L[d]);
    }
    auto add = [&](int comp, const Win<R>& wx, const Win<R>& wy, const Win<R>& wz) {
        const R Fa = static_cast<R>(F[3 * b + comp] * scale);
        R* fa = fb + comp * (int)g.N;
        const bool odd = (wx.o[0] & 1) != 0;
        const int a0 = wx.o[0] & ~1, a1 = (a0 + 2) & (nx - 1);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
#pragma unroll
            for (int bb = 0; bb < 3; ++bb) {
                const R wyz = wy.w[bb] * wz.w[c] * Fa;
                R* row = fa + (wz.o[c] + wy.o[bb]);
                if constexpr (sizeof(R) == 4) {
                    const float v0 = wx.w[0] * wyz, v1 = wx.w[1] * wyz, v2 = wx.w[2] * wyz;
                    atomicAdd(reinterpret_cast<float2*>(row + a0),
                              odd ? make_float2(0.0f, v0) : make_float2(v0, v1));
                    atomicAdd(reinterpret_cast<float2*>(row + a1),
                              odd ? make_float2(v1, v2) : make_float2(v2, 0.0f));
                } else {
#pragma unroll
                    for (int aa = 0; aa < 3; ++aa) atomicAdd(row + wx.o[aa], wx.w[aa] * wyz);
                }
            }
        }
    };
    if (SPLIT) {
        Win<R> w[3];
#pragma unroll
        for (int d = 0; d < 3; ++d)
            w[d].set(x[d] * g.inv_h - (d == mine ? 0.0 : 0.5), mask[d], stride[d]);
        add(mine, w[0], w[1], w[2]);
    } else {
        Win<R> own[3], across[3];
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            own[d].set(x[d] * g.inv_h - 0.0, mask[d], stride[d]);
            across[d].set(x[d] * g.inv_h - 0.5, mask[d], stride[d]);
        }
#pragma unroll
        for (int c = 0; c < 3; ++c)
            add(c, c == 0 ? own[0] : across[0], c == 1 ? own[1] : across[1],
                c == 2 ? own[2] : across[2]);
    }
}

template <typename R>
cudaError_t launch_spread_atomic(Chain st, int B, int64_t nb, const double* q,
                                 const double* F, const int32_t* box_of, const GridGeo& g, R* f,
                                 bool zeroed, bool wrap, double scale)
{
    if (!zeroed) {
        const cudaError_t e = cudaMemsetAsync(f, 0, sizeof(R) * 3 * (size_t)B * g.N, st.st);
        if (e != cudaSuccess) return e;
    }
    if (nb <= 0) return cudaSuccess;
    const bool split = split_components(nb);
    const int T = split ? 96 : blob_block(nb);
    const unsigned blocks = blocks_of(split ? 3 * nb : nb, T);
    scale *= Win<R>::UNIT;
    auto go = [&](auto k) {
        return launch_on(st, k, dim3(blocks), dim3(T), 0, nb, q, F, box_of, g, scale, f);
    };
    if (wrap) return split ? go(k_spread_atomic<R, true, true>) : go(k_spread_atomic<R, false, true>);
    return split ? go(k_spread_atomic<R, true, false>) : go(k_spread_atomic<R, false, false>);
}
template cudaError_t launch_spread_atomic<double>(Chain, int, int64_t, const double*,
                                                  const double*, const int32_t*, const GridGeo&,
                                                  double*, bool, bool, double);
template cudaError_t launch_spread_atomic<float>(Chain, int, int64_t, const double*,
                                                 const double*, const int32_t*, const GridGeo&,
                                                 float*, bool, bool, double);

// The sums are 64-bit fixed point
// (shared-memory integer atomics are associative, so the sums do not depend on the order in
// which threads add).  The tile's scale is a power of two chosen from its largest force so that
// no node can overflow: 2^62 over (candidates x max weight product x max |F| / h^3).
__global__ void __launch_bounds__(256)
k_spread_det(const double* __restrict__ q, const double* __restrict__ F,
             const int32_t* __restrict__ sorted, const int32_t* __restrict__ cell_start, GridGeo g,
             BinGeo bg, int TX, int TY, int TZ, int max_ranges, double* __restrict__ f)
{
    dep_wait();
    dep_release();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int tileN = TX * TY * TZ;
    unsigned long long* acc = reinterpret_cast<unsigned long long*>(smem_raw);
    int32_t* rbeg = reinterpret_cast<int32_t*>(acc + 3 * tileN);
    int32_t* rpre = rbeg + max_ranges;
    __shared__ double fmax_sh[32];
    const int nx = g.n[0], ny = g.n[1], nz = g.n[2];
    const int box = blockIdx.y;
    const int ntx = nx / TX, nty = ny / TY;
    const int tid = blockIdx.x;
    const int T0[3] = {(tid % ntx) * TX, ((tid / ntx) % nty) * TY, (tid / (ntx * nty)) * TZ};
    const int T[3] = {TX, TY, TZ};
    for (int i = threadIdx.x; i < 3 * tileN; i += blockDim.x) acc[i] = 0ull;
    int lo[3], cnt[3];
    for (int d = 0; d < 3; ++d) halo_cells(T0[d], T[d], bg.bs, bg.nc[d], lo[d], cnt[d]);
    const int rows = cnt[1] * cnt[2];
    const int nr = 2 * rows;
    for (int r = threadIdx.x; r < rows; r += blockDim.x) {
        const int cz = wrap_cell(lo[2] + r / cnt[1], bg.nc[2]);
        const int cy = wrap_cell(lo[1] + r % cnt[1], bg.nc[1]);
        const int64_t rowbase = box * bg.ncell + ((int64_t)cz * bg.nc[1] + cy) * bg.nc[0];
        const int sx = wrap_cell(lo[0], bg.nc[0]);
        const int ex = sx + cnt[0];
        const int a1 = ex <= bg.nc[0] ? ex : bg.nc[0];
        const int s0 = cell_start[rowbase + sx];
        rbeg[2 * r] = s0;
        rpre[2 * r] = cell_start[rowbase + a1] - s0;
        if (ex > bg.nc[0]) {
            const int t0 = cell_start[rowbase];
            rbeg[2 * r + 1] = t0;
            rpre[2 * r + 1] = cell_start[rowbase + (ex - bg.nc[0])] - t0;
        } else {
            rbeg[2 * r + 1] = 0;
            rpre[2 * r + 1] = 0;
        }
    }
    __syncthreads();
    if (threadIdx.x < 32) {       // exclusive prefix of the lengths (one warp)
        const int lane = threadIdx.x;
        int carry = 0;
        for (int c0 = 0; c0 < nr; c0 += 32) {
            const int i = c0 + lane;
            const int len = i < nr ? rpre[i] : 0;
            int x = len;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, x, o);
                if (lane >= o) x += y;
            }
            if (i < nr) rpre[i] = carry + x - len;
            carry += __shfl_sync(0xffffffffu, x, 31);
        }
        if (lane == 0) rpre[nr] = carry;
    }
    __syncthreads();
    const int total = rpre[nr];
    auto blob_of = [&](int t) {
        int a = 0, b = nr - 1;
        while (a < b) {
            const int m = (a + b + 1) >> 1;
            if (rpre[m] <= t) a = m; else b = m - 1;
        }
        return 3 * (int64_t)sorted[rbeg[a] + (t - rpre[a])];      // its offset in q and F
    };
    // tile scale from the largest force component among the candidates
    double fm = 0.0;
    for (int t = threadIdx.x; t < total; t += blockDim.x) {
        const double* Fb = F + blob_of(t);
        fm = fmax(fm, fmax(fabs(Fb[0]), fmax(fabs(Fb[1]), fabs(Fb[2]))));
    }
    for (int o = 16; o > 0; o >>= 1) fm = fmax(fm, __shfl_down_sync(0xffffffffu, fm, o));
    if ((threadIdx.x & 31) == 0) fmax_sh[threadIdx.x >> 5] = fm;
    __syncthreads();
    if (threadIdx.x == 0) {
        double m = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) m = fmax(m, fmax_sh[w]);
        fmax_sh[0] = m;
    }
    __syncthreads();
    const double inv_h3 = g.inv_h * g.inv_h * g.inv_h;
    const double bound = fmax(fmax_sh[0] * inv_h3 * (8.0 / 27.0) * (double)(total + 1), 1e-300);
    int ex2;
    frexp(bound, &ex2);                      // bound < 2^ex2
    const double scale = ldexp(1.0, 62 - max(ex2, -900));   // finite even for a zero tile
    // one thread per blob and component, or per plane of its window too when the tile has few
    // blobs (a thread's chain of roots and conversions sets the time then)
    const int parts = 9 * total <= (int)blockDim.x ? 9 : 3;
    for (int i = threadIdx.x; i < parts * total; i += blockDim.x) {
        const int t = i / parts, part = i - t * parts;
        const int a = part % 3, c0 = part / 3, c1 = parts == 9 ? c0 + 1 : 3;
        const int64_t at = blob_of(t);
        const double* rr = q + at;
        const double Fa = F[at + a] * inv_h3;
        double wx[3], wy[3], wz[3];
        const int ix = peskin_window<double>(rr[0] * g.inv_h - mac_shift(a, 0), wx) - T0[0];
        const int iy = peskin_window<double>(rr[1] * g.inv_h - mac_shift(a, 1), wy) - T0[1];
        const int iz = peskin_window<double>(rr[2] * g.inv_h - mac_shift(a, 2), wz) - T0[2];
        unsigned long long* acc_a = acc + a * tileN;
        for (int c = c0; c < c1; ++c) {
            const int rz = (iz + c) & (nz - 1);
            if (rz >= TZ) continue;
            const double wzc = c == 0 ? wz[0] : (c == 1 ? wz[1] : wz[2]);
            for (int bb = 0; bb < 3; ++bb) {
                const int ry = (iy + bb) & (ny - 1);
                if (ry >= TY) continue;
                const double wyz = wy[bb] * wzc * Fa;
                for (int aa = 0; aa < 3; ++aa) {
                    const int rx = (ix + aa) & (nx - 1);
                    if (rx < TX) {
                        const long long v = llrint(wx[aa] * wyz * scale);
                        atomicAdd(acc_a + (rz * TY + ry) * TX + rx, (unsigned long long)v);
                    }
                }
            }
        }
    }
    __syncthreads();
    const double inv_scale = 1.0 / scale;
    const int lx = 31 - __clz(TX), lxy = lx + 31 - __clz(TY), lt = 31 - __clz(tileN);   // powers of two
    for (int i = threadIdx.x; i < 3 * tileN; i += blockDim.x) {
        const int a = i >> lt, rem = i & (tileN - 1);
        const int rz = rem >> lxy, ry = (rem >> lx) & (TY - 1), rx = rem & (TX - 1);
        f[((size_t)box * 3 + a) * (size_t)g.N +
          ((size_t)(T0[2] + rz) * ny + (T0[1] + ry)) * nx + (T0[0] + rx)] =
            (double)(long long)acc[i] * inv_scale;
    }
}

cudaError_t launch_spread_det(Chain st, int B, const double* q, const double* F,
                              const int32_t* sorted, const int32_t* cell_start, const GridGeo& g,
                              const BinGeo& bg, const int tile_in[3], double* f)
{
    // small grids: tiles halved along their longest side (whole bin cells, at least four nodes)
    // until there are two blocks for each SM; a block's clearing and writing of its nodes, not
    // its blobs, sets the time there
    int tile[3] = {tile_in[0], tile_in[1], tile_in[2]};
    const int least = bg.bs > 4 ? bg.bs : 4;
    auto tiles = [&] { return (int64_t)(g.n[0] / tile[0]) * (g.n[1] / tile[1]) * (g.n[2] / tile[2]); };
    while (tiles() * B < 304) {
        int d = 0;
        for (int e = 1; e < 3; ++e)
            if (tile[e] > tile[d]) d = e;
        if (tile[d] / 2 < least) break;
        tile[d] /= 2;
    }
    const int TX = tile[0], TY = tile[1], TZ = tile[2];
    int max_rows = 1;
    for (int d = 1; d < 3; ++d) {
        int most = 0;
        for (int T0 = 0; T0 < g.n[d]; T0 += tile[d]) {
            int lo, cnt;
            halo_cells(T0, tile[d], bg.bs, bg.nc[d], lo, cnt);
            most = cnt > most ? cnt : most;
        }
        max_rows *= most;
    }
    const int max_ranges = 2 * max_rows;
    const size_t smem = 3 * (size_t)TX * TY * TZ * 8 + sizeof(int32_t) * (2 * max_ranges + 1);
    static std::atomic<unsigned> attr{0};
    if (first_on_device(attr))
        cudaFuncSetAttribute(k_spread_det, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
    return launch_on(st, k_spread_det, dim3((unsigned)tiles(), (unsigned)B), dim3(256), smem, q, F,
                     sorted, cell_start, g, bg, TX, TY, TZ, max_ranges, f);
}

// ==========================================================================================
// Particle velocities: U0 = mean blob velocity; Omega from the least-squares rigid rotation,
// I0 Omega = sum s x (u - U0) with I0 = sum (s.s 1 - s s) and s relative to the baricentre.
// One warp per particle, its blobs over the lanes (a thread per particle took 60 us for 64
// particles, one chain of FP64 sums and image searches each).
__device__ __forceinline__ double warp_sum(double x)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    return x;
}

__global__ void __launch_bounds__(128)
k_particle_reduce(int64_t np, const int32_t* __restrict__ part_start,
                  const int32_t* __restrict__ part_blobs, const double* __restrict__ q,
                  const double* __restrict__ u, GridGeo g, double* __restrict__ U,
                  double* __restrict__ Omega)
{
    const int64_t p = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (p >= np) return;
    const int s = part_start[p], e = part_start[p + 1];
    double Um[3] = {0, 0, 0}, Om[3] = {0, 0, 0};
    if (e > s) {
        const int b0 = part_blobs[s];
        const double inv = 1.0 / (double)(e - s);
        double cm[3] = {0, 0, 0}, q0[3];
        for (int d = 0; d < 3; ++d) q0[d] = q[3 * b0 + d];
        for (int i = s + lane; i < e; i += 32) {
            const int b = part_blobs[i];
            for (int d = 0; d < 3; ++d) {
                Um[d] += u[3 * b + d];
                cm[d] += min_image(q[3 * b + d] - q0[d], g.L[d]);
            }
        }
        for (int d = 0; d < 3; ++d) {
            Um[d] = warp_sum(Um[d]) * inv;
            cm[d] = warp_sum(cm[d]) * inv;
        }
        if (Omega) {
            double I[6] = {0, 0, 0, 0, 0, 0};   // xx, yy, zz, xy, xz, yz
            double tq[3] = {0, 0, 0};
            for (int i = s + lane; i < e; i += 32) {
                const int b = part_blobs[i];
                double sv[3], w[3];
                for (int d = 0; d < 3; ++d) {
                    sv[d] = min_image(q[3 * b + d] - q0[d], g.L[d]) - cm[d];
                    w[d] = u[3 * b + d] - Um[d];
                }
                const double s2 = sv[0] * sv[0] + sv[1] * sv[1] + sv[2] * sv[2];
                I[0] += s2 - sv[0] * sv[0];
                I[1] += s2 - sv[1] * sv[1];
                I[2] += s2 - sv[2] * sv[2];
                I[3] -= sv[0] * sv[1];
                I[4] -= sv[0] * sv[2];
                I[5] -= sv[1] * sv[2];
                tq[0] += sv[1] * w[2] - sv[2] * w[1];
                tq[1] += sv[2] * w[0] - sv[0] * w[2];
                tq[2] += sv[0] * w[1] - sv[1] * w[0];
            }
            for (int k = 0; k < 6; ++k) I[k] = warp_sum(I[k]);
            for (int k = 0; k < 3; ++k) tq[k] = warp_sum(tq[k]);
            // symmetric 3x3 inverse through the adjugate
            const double a = I[0], bq = I[1], c = I[2], xy = I[3], xz = I[4], yz = I[5];
            const double A00 = bq * c - yz * yz, A01 = xz * yz - xy * c, A02 = xy * yz - xz * bq;
            const double A11 = a * c - xz * xz, A12 = xy * xz - a * yz, A22 = a * bq - xy * xy;
            const double det = a * A00 + xy * A01 + xz * A02;
            const double tr = a + bq + c;
            if (tr > 0.0 && fabs(det) > 1e-12 * tr * tr * tr) {
                const double id = 1.0 / det;
                Om[0] = (A00 * tq[0] + A01 * tq[1] + A02 * tq[2]) * id;
                Om[1] = (A01 * tq[0] + A11 * tq[1] + A12 * tq[2]) * id;
                Om[2] = (A02 * tq[0] + A12 * tq[1] + A22 * tq[2]) * id;
            }
        }
    }
    if (lane != 0) return;
    for (int d = 0; d < 3; ++d) {
        if (U) U[3 * p + d] = Um[d];
        if (Omega) Omega[3 * p + d] = Om[d];
    }
}

cudaError_t launch_particle_reduce(cudaStream_t st, int64_t np, const int32_t* part_start,
                                   const int32_t* part_blobs, const double* q, const double* u,
                                   const GridGeo& g, double* U, double* Omega)
{
    if (np <= 0) return cudaSuccess;
    k_particle_reduce<<<blocks_of(np, 4), 128, 0, st>>>(np, part_start, part_blobs, q, u, g, U,
                                                        Omega);
    return cudaGetLastError();
}

// Transpose of the particle mean U0 = (1/N_p) sum_{i in p} u_i (Sec. 2): every blob of particle
// p receives gU_p / N_p.  One thread per particle; blobs belong to one particle each, so the
// writes are disjoint.
__global__ void k_particle_mean_adjoint(int64_t np, const int32_t* __restrict__ part_start,
                                        const int32_t* __restrict__ part_blobs,
                                        const double* __restrict__ gU, double* __restrict__ gu)
{
    const int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (p >= np) return;
    const int s = part_start[p], e = part_start[p + 1];
    if (e <= s) return;
    const double inv = 1.0 / (double)(e - s);
    const double g0 = gU[3 * p] * inv, g1 = gU[3 * p + 1] * inv, g2 = gU[3 * p + 2] * inv;
    for (int i = s; i < e; ++i) {
        const int b = part_blobs[i];
        gu[3 * b] = g0;
        gu[3 * b + 1] = g1;
        gu[3 * b + 2] = g2;
    }
}

cudaError_t launch_particle_mean_adjoint(cudaStream_t st, int64_t np, const int32_t* part_start,
                                         const int32_t* part_blobs, const double* gU, double* gu)
{
    if (np <= 0) return cudaSuccess;
    k_particle_mean_adjoint<<<(unsigned)((np + 127) / 128), 128, 0, st>>>(np, part_start,
                                                                         part_blobs, gU, gu);
    return cudaGetLastError();
}

// ==========================================================================================
// Mean of each component grid (FP64 accumulation, fixed order): partial sums of equal chunks,
// then their sum.  (One block a component took 1.5 ms at 128^3.)
__device__ __forceinline__ double block_sum(double s, double* sh)
{
    sh[threadIdx.x] = s;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w) sh[threadIdx.x] += sh[threadIdx.x + w];
        __syncthreads();
    }
    return sh[0];
}

template <typename R>
__global__ void __launch_bounds__(256)
k_grid_partial(GridGeo g, const R* __restrict__ v, double* __restrict__ partial)
{
    __shared__ double sh[256];
    const R* c = v + (size_t)blockIdx.y * g.N;
    double s = 0.0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < g.N;
         i += (int64_t)gridDim.x * blockDim.x)
        s += (double)c[i];
    s = block_sum(s, sh);
    if (threadIdx.x == 0) partial[(size_t)blockIdx.y * gridDim.x + blockIdx.x] = s;
}

__global__ void __launch_bounds__(256)
k_grid_mean(int chunks, int64_t N, const double* __restrict__ partial, double* __restrict__ mean_out)
{
    __shared__ double sh[256];
    double s = 0.0;
    for (int i = threadIdx.x; i < chunks; i += blockDim.x) s += partial[(size_t)blockIdx.x * chunks + i];
    s = block_sum(s, sh);
    if (threadIdx.x == 0) mean_out[blockIdx.x] = s / (double)N;
}

int grid_mean_chunks(int64_t N) { return (int)((N + 16383) / 16384); }

template <typename R>
cudaError_t launch_grid_mean(cudaStream_t st, int B, const GridGeo& g, const R* v,
                             double* mean_out, double* partial)
{
    const int chunks = grid_mean_chunks(g.N);
    for (int b0 = 0; b0 < 3 * B; b0 += 65535) {                 // the grid's y limit
        const int nc = 3 * B - b0 < 65535 ? 3 * B - b0 : 65535;
        k_grid_partial<R><<<dim3((unsigned)chunks, (unsigned)nc), 256, 0, st>>>(
            g, v + (size_t)b0 * g.N, partial + (size_t)b0 * chunks);
    }
    k_grid_mean<<<B * 3, 256, 0, st>>>(chunks, g.N, partial, mean_out);
    return cudaGetLastError();
}
template cudaError_t launch_grid_mean<float>(cudaStream_t, int, const GridGeo&, const float*,
                                             double*, double*);
template cudaError_t launch_grid_mean<double>(cudaStream_t, int, const GridGeo&, const double*,
                                              double*, double*);

}  // namespace mbk
