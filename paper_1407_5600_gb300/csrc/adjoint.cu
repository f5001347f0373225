// Kernels of the adjoint (reverse-mode derivative) of the ICM step, FP64.
//
// The step's position dependence enters through the kernel weights of J and S and through the
// blob forces.  Their transposes are
//   d/dq_i [ sum_a c_ia J_i(q) w_a ]          = sum_a c_ia sum_nodes grad_q(prod Phi) w_a(node)
//   d/dq_i [ <g, S(q) F> ]                    = h^-3 sum_a F_ia sum_nodes grad_q(prod Phi) g_a(node)
// (gradient interpolation with the kernel derivative Phi', continuous because Phi is C^1), and
// the force Jacobian-vector product (dF/dq)^T g = (dF/dq) g (forces derive from a potential),
// bond by bond: J_f (g_i - g_j) with J_f = df/dr.
#include "mb_internal.cuh"
#include "peskin.cuh"

namespace mbk {

namespace {

// Sums over the 27 nodes of a window of one grid (+ a second one): the interpolated value and
// the sums with the weights' derivatives along x, y, z, taken by rows and planes (90 products
// a component instead of 243).
struct WinD {
    double w[3], d[3];
    int o[3];
    __device__ __forceinline__ void set(double x, int mask, int stride)
    {
        const int i = peskin_window_d(x, w, d);
#pragma unroll
        for (int k = 0; k < 3; ++k) o[k] = ((i + k) & mask) * stride;
    }
};
__device__ __forceinline__ void window_grad(const double* __restrict__ c0,
                                            const double* __restrict__ c1, const WinD& wx,
                                            const WinD& wy, const WinD& wz, double& val,
                                            double gr[3])
{
    val = gr[0] = gr[1] = gr[2] = 0.0;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        double pv = 0.0, px = 0.0, py = 0.0;
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            const int row = wz.o[c] + wy.o[b];
            double rv = 0.0, rx = 0.0;
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                double v = __ldg(c0 + (row + wx.o[a]));
                if (c1) v += __ldg(c1 + (row + wx.o[a]));
                rv += wx.w[a] * v;
                rx += wx.d[a] * v;
            }
            pv += wy.w[b] * rv;
            px += wy.w[b] * rx;
            py += wy.d[b] * rv;
        }
        val += wz.w[c] * pv;
        gr[0] += wz.w[c] * px;
        gr[1] += wz.w[c] * py;
        gr[2] += wz.d[c] * pv;
    }
}

// The windows of component `comp` at position x (in mesh units, x h = q).
__device__ __forceinline__ void windows_of(int comp, const double x[3], const GridGeo& g, WinD w[3])
{
    w[0].set(x[0] - (comp == 0 ? 0.0 : 0.5), g.n[0] - 1, 1);
    w[1].set(x[1] - (comp == 1 ? 0.0 : 0.5), g.n[1] - 1, g.n[0]);
    w[2].set(x[2] - (comp == 2 ? 0.0 : 0.5), g.n[2] - 1, g.n[0] * g.n[1]);
}

// These two kernels take one thread per blob and component, 32 blobs a block: the component
// sums of a blob's gradient meet in shared memory.
constexpr int ADJ_BLOBS = 32, ADJ_THREADS = 3 * ADJ_BLOBS;

__device__ __forceinline__ double component_sum(const double gr[3], double (*sh)[3], int mine)
{
    for (int d = 0; d < 3; ++d) sh[threadIdx.x][d] = gr[d];
    __syncthreads();
    const int j = (int)threadIdx.x - mine;
    return sh[j][mine] + sh[j + 1][mine] + sh[j + 2][mine];
}

// At the midpoints q: with gf = T dL/dv^{n+1} (the transpose of the fluid update in f),
//   gF  = S^T gf = h^-3 J gf
//   gqh = d/dq [ <gf, S(q) F> + sum dt gq . J(q) (v0 + v1)/2 ]
__global__ void __launch_bounds__(ADJ_THREADS)
k_adjoint_midpoint(int64_t nb, const double* __restrict__ q, const double* __restrict__ gf,
                   const double* __restrict__ F, const double* __restrict__ v0,
                   const double* __restrict__ v1, const double* __restrict__ gq, double dt,
                   GridGeo g, double* __restrict__ gF, double* __restrict__ gqh)
{
    dep_wait();
    dep_release();
    __shared__ double sh[ADJ_THREADS][3];
    const int64_t t = blockIdx.x * (int64_t)ADJ_THREADS + threadIdx.x;
    const int64_t b = t / 3;
    const int mine = (int)(t - 3 * b);
    const bool live = b < nb;
    const double inv_h3 = g.inv_h * g.inv_h * g.inv_h;
    double gr[3] = {0.0, 0.0, 0.0};
    if (live) {
        const double x[3] = {q[3 * b] * g.inv_h, q[3 * b + 1] * g.inv_h, q[3 * b + 2] * g.inv_h};
        WinD w[3];
        windows_of(mine, x, g, w);
        const size_t base = (size_t)mine * g.N;
        double val, d1[3], d2[3];
        window_grad(gf + base, nullptr, w[0], w[1], w[2], val, d1);
        gF[t] = val * inv_h3;
        const double c1 = F[t] * inv_h3, c2 = 0.5 * dt * gq[t];
        window_grad(v0 + base, v1 + base, w[0], w[1], w[2], val, d2);
        for (int d = 0; d < 3; ++d) gr[d] = (c1 * d1[d] + c2 * d2[d]) * g.inv_h;
    }
    const double s = component_sum(gr, sh, mine);
    if (live) gqh[t] = s;
}

// Transpose of u = J(q) v with gradient gu = scale * gu_in:
//   out = base (+ base2) + (du/dq)^T gu,  gv += J(q)^T gu
__global__ void __launch_bounds__(ADJ_THREADS)
k_adjoint_velocity(int64_t nb, const double* __restrict__ q, const double* __restrict__ v,
                   const double* gu_in, double scale, const double* base, const double* base2,
                   GridGeo g, double* out, double* gv)
{
    dep_wait();
    dep_release();
    __shared__ double sh[ADJ_THREADS][3];
    const int64_t t = blockIdx.x * (int64_t)ADJ_THREADS + threadIdx.x;
    const int64_t b = t / 3;
    const int mine = (int)(t - 3 * b);
    const bool live = b < nb;
    double gr[3] = {0.0, 0.0, 0.0};
    double at = 0.0;
    if (live) {
        double x[3];
        for (int d = 0; d < 3; ++d) x[d] = wrap_any(q[3 * b + d], g.L[d]) * g.inv_h;
        const double gu = scale * gu_in[t];
        at = base2 ? base[t] + base2[t] : base[t];
        if (gu != 0.0) {
            WinD w[3];
            windows_of(mine, x, g, w);
            const size_t comp = (size_t)mine * g.N;
            double val;
            window_grad(v + comp, nullptr, w[0], w[1], w[2], val, gr);
            for (int d = 0; d < 3; ++d) gr[d] *= gu * g.inv_h;
            double* f = gv + comp;
#pragma unroll
            for (int c = 0; c < 3; ++c)
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    const double wyz = w[1].w[k] * w[2].w[c] * gu;
                    const int row = w[2].o[c] + w[1].o[k];
#pragma unroll
                    for (int a = 0; a < 3; ++a) atomicAdd(f + (row + w[0].o[a]), w[0].w[a] * wyz);
                }
        }
    }
    const double s = component_sum(gr, sh, mine);
    if (live) out[t] = at + s;
}

// (rho/dt + (eta/2) L) x: A = (rho/dt + (eta/2) L) T for the fluid update v' = A v + T f, all
// three diagonal in Fourier space, so that A^T g is this stencil of T g and needs no second
// solve.
__global__ void __launch_bounds__(256)
k_viscous_stencil(GridGeo g, const double* __restrict__ x, double a, double c, double* __restrict__ out)
{
    dep_wait();
    dep_release();
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= 3 * g.N) return;
    const int nx = g.n[0], ny = g.n[1], nz = g.n[2];
    const int comp = (int)(i / g.N), m = (int)(i - comp * g.N);
    const int ix = m & (nx - 1), row = m - ix, iy = (row / nx) & (ny - 1), iz = row / (nx * ny);
    const int plane = row - iy * nx, col = m - iz * nx * ny;
    const double* s = x + (size_t)comp * g.N;
    const double v = s[m];
    const double sum = (s[row + ((ix - 1) & (nx - 1))] + s[row + ((ix + 1) & (nx - 1))]) +
                       (s[plane + ((iy - 1) & (ny - 1)) * nx + ix] + s[plane + ((iy + 1) & (ny - 1)) * nx + ix]) +
                       (s[col + ((iz - 1) & (nz - 1)) * nx * ny] + s[col + ((iz + 1) & (nz - 1)) * nx * ny]);
    out[i] = a * v + c * (sum - 6.0 * v);
}

// Hessian-vector product of the blob forces and the spring-stiffness derivative.
//   out_b += sum_bonds J_s(r_bj) (g_b - g_j) + sum_pairs J_r(r_bj) (g_b - g_j)
//   J_s = -k [(1 - r0/|r|) I + (r0/|r|) rhat rhat^T]
//   J_r = k_rep [(r_cut/|r| - 1) I - (r_cut/|r|) rhat rhat^T]         (|r| < r_cut)
//   dL/dk += (1/2) sum_b sum_bonds (f_bond(r_bj)/k) . (g_b - g_j)    (each bond seen twice)
// Eight lanes a blob over its bonds and then its neighbour cells: the centre of an icosahedron
// has twelve bonds, which one thread took in turn (101 us for 832 blobs).
constexpr int JVP_LANES = 8, JVP_BLOCK = 128;

__global__ void __launch_bounds__(JVP_BLOCK)
k_force_jvp(int64_t nb, const double* __restrict__ q, const double* __restrict__ gF,
            const int32_t* __restrict__ pid, const int32_t* __restrict__ adj_start,
            const int32_t* __restrict__ adj_j, const double* __restrict__ adj_rest,
            double k_spring, double k_rep, double r_cut, const int32_t* __restrict__ cell_start,
            const int32_t* __restrict__ sorted, const int32_t* __restrict__ blob_cell,
            GridGeo g, BinGeo bg, double* __restrict__ out, double* __restrict__ gk)
{
    dep_wait();
    dep_release();
    __shared__ double sh[JVP_BLOCK / 32];
    const int lane = threadIdx.x % JVP_LANES;
    double dk = 0.0;
    for (int64_t b0 = blockIdx.x * (int64_t)(JVP_BLOCK / JVP_LANES); b0 < nb;
         b0 += (int64_t)gridDim.x * (JVP_BLOCK / JVP_LANES)) {
        const int64_t b = b0 + threadIdx.x / JVP_LANES;
        double acc[3] = {0.0, 0.0, 0.0};
        if (b < nb) {
            const double qb[3] = {q[3 * b], q[3 * b + 1], q[3 * b + 2]};
            const double gb[3] = {gF[3 * b], gF[3 * b + 1], gF[3 * b + 2]};
            for (int e = adj_start[b] + lane; e < adj_start[b + 1]; e += JVP_LANES) {
                const int j = adj_j[e];
                double r[3], dg[3];
                for (int d = 0; d < 3; ++d) {
                    r[d] = min_image(qb[d] - q[3 * j + d], g.L[d]);
                    dg[d] = gb[d] - gF[3 * j + d];
                }
                const Length l(r[0] * r[0] + r[1] * r[1] + r[2] * r[2]);
                const double dot = r[0] * dg[0] + r[1] * dg[1] + r[2] * dg[2];
                const double ratio = l.divide(adj_rest[e]);
                const double a0 = -k_spring * (1.0 - ratio);
                const double a1 = -k_spring * ratio * l.divide(l.divide(dot));
                for (int d = 0; d < 3; ++d) acc[d] += a0 * dg[d] + a1 * r[d];
                dk -= 0.5 * l.divide(l.len - adj_rest[e]) * dot;      // f_bond / k
            }
            if (k_rep != 0.0 && r_cut > 0.0) {
                const int cell = blob_cell[b];
                const int c[3] = {cell % bg.nc[0], (cell / bg.nc[0]) % bg.nc[1],
                                  cell / (bg.nc[0] * bg.nc[1])};
                int lo[3], cnt[3];
                for (int d = 0; d < 3; ++d) {
                    lo[d] = bg.nc[d] >= 3 ? -1 : 0;
                    cnt[d] = bg.nc[d] >= 3 ? 3 : bg.nc[d];
                }
                for (int k = lane; k < cnt[0] * cnt[1] * cnt[2]; k += JVP_LANES) {
                    const int dd[3] = {lo[0] + k % cnt[0], lo[1] + (k / cnt[0]) % cnt[1],
                                       lo[2] + k / (cnt[0] * cnt[1])};
                    int cc[3];
                    for (int d = 0; d < 3; ++d)
                        cc[d] = bg.nc[d] >= 3 ? (c[d] + dd[d] + bg.nc[d]) % bg.nc[d] : dd[d];
                    const int at = (cc[2] * bg.nc[1] + cc[1]) * bg.nc[0] + cc[0];
                    for (int t = cell_start[at]; t < cell_start[at + 1]; ++t) {
                        const int j = sorted[t];
                        if (j == b || pid[j] == pid[b]) continue;
                        double r[3], dg[3];
                        for (int d = 0; d < 3; ++d) r[d] = min_image(qb[d] - q[3 * j + d], g.L[d]);
                        const double r2 = r[0] * r[0] + r[1] * r[1] + r[2] * r[2];
                        if (r2 >= r_cut * r_cut || r2 == 0.0) continue;
                        const Length l(r2);
                        for (int d = 0; d < 3; ++d) dg[d] = gb[d] - gF[3 * j + d];
                        const double dot = r[0] * dg[0] + r[1] * dg[1] + r[2] * dg[2];
                        const double ratio = l.divide(r_cut);
                        const double a0 = k_rep * (ratio - 1.0);
                        const double a1 = -k_rep * ratio * l.divide(l.divide(dot));
                        for (int d = 0; d < 3; ++d) acc[d] += a0 * dg[d] + a1 * r[d];
                    }
                }
            }
        }
#pragma unroll
        for (int o = JVP_LANES / 2; o > 0; o >>= 1)
            for (int d = 0; d < 3; ++d) acc[d] += __shfl_xor_sync(0xffffffffu, acc[d], o);
        if (b < nb && lane == 0)
            for (int d = 0; d < 3; ++d) out[3 * b + d] += acc[d];
    }
    if (!gk) return;
    // block sum of dk, one double atomic per block
    for (int o = 16; o > 0; o >>= 1) dk += __shfl_down_sync(0xffffffffu, dk, o);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = dk;
    __syncthreads();
    if (threadIdx.x == 0) {
        double x = 0.0;
        for (int w = 0; w < JVP_BLOCK / 32; ++w) x += sh[w];
        atomicAdd(gk, x);
    }
}

inline unsigned nblk(int64_t n, int per) { return (unsigned)((n + per - 1) / per); }

}  // namespace

cudaError_t launch_adjoint_midpoint(Chain st, int64_t nb, const double* q, const double* gf,
                                    const double* F, const double* v0, const double* v1,
                                    const double* gq, double dt, const GridGeo& g, double* gF,
                                    double* gqh)
{
    if (nb <= 0) return cudaSuccess;
    return launch_on(st, k_adjoint_midpoint, dim3(nblk(nb, ADJ_BLOBS)), dim3(ADJ_THREADS), 0, nb, q, gf, F, v0, v1, gq, dt, g,
                                                                   gF, gqh);
}

cudaError_t launch_adjoint_velocity(Chain st, int64_t nb, const double* q, const double* v,
                                    const double* gu, double scale, const double* base,
                                    const double* base2, const GridGeo& g, double* out, double* gv)
{
    if (nb <= 0) return cudaSuccess;
    return launch_on(st, k_adjoint_velocity, dim3(nblk(nb, ADJ_BLOBS)), dim3(ADJ_THREADS), 0, nb, q, v, gu, scale, base, base2,
                                                                   g, out, gv);
}

cudaError_t launch_viscous_stencil(Chain st, const GridGeo& g, const double* x, double a,
                                   double c, double* out)
{
    return launch_on(st, k_viscous_stencil, dim3(nblk(3 * g.N, 256)), dim3(256), 0, g, x, a, c, out);
}

cudaError_t launch_force_jvp(Chain st, int64_t nb, const double* q, const double* gF,
                             const int32_t* pid, const int32_t* adj_start, const int32_t* adj_j,
                             const double* adj_rest, double k_spring, double k_rep, double r_cut,
                             const int32_t* cell_start, const int32_t* sorted,
                             const int32_t* blob_cell, const GridGeo& g, const BinGeo& bg,
                             double* out, double* gk)
{
    if (nb <= 0) return cudaSuccess;
    // at most 2048 blocks, so that as few atomics meet on gk
    const unsigned blocks = nblk(nb, JVP_BLOCK / JVP_LANES);
    return launch_on(st, k_force_jvp, dim3(blocks < 2048 ? blocks : 2048), dim3(JVP_BLOCK), 0, 
        nb, q, gF, pid, adj_start, adj_j, adj_rest, k_spring, k_rep, r_cut, cell_start, sorted,
        blob_cell, g, bg, out, gk);
}

}  // namespace mbk
