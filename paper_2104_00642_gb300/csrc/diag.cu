// diag.cu -- FP64 diagnostics: field energy, kinetic energy per species,
// live counts, the particle charge density averaged over the two half-step
// positions that bracket the integer step, and the Gauss residual
// max |div E - rho - rho_bg| (Eq. (1) in the units of Eq. (8)).
//
// Sums use a fixed reduction tree: blocks that each reduce a fixed strided set
// of elements in a fixed shuffle order into one partial, and the block that
// finishes last summing the partials in index order, so results do not depend
// on scheduling.  Nor on the number of blocks, which follows the host's bound
// on the elements: as long as it is below kRedBlocks a thread has one element
// at most, its block's partial is the same whatever the grid, and the blocks
// left out are those whose partials would be zero.
//
// FP64 runs at 1/73 of the FP32 rate here and bounds these kernels: the roots
// and quotients are Newton iterations from an FP32 seed, FP32 inputs become
// FP64 by moving their bits, and nothing is divided by dx per particle
// (charge density of 1,048,576 particles in 2D: 326 -> 212 us; species
// without charge deposit none).
#include <algorithm>

#include "diag.cuh"
#include "fp64_dev.cuh"
#include "push_dev.cuh"

namespace pic {

constexpr int kRedBlocks = 1024;
constexpr int kRedThreads = 256;

__device__ __forceinline__ double warp_sum(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}
__device__ __forceinline__ double warp_max(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_down_sync(0xffffffffu, v, o));
    return v;
}

template <int NV, bool MAX>
__device__ __forceinline__ void block_reduce_store(const double *v, double *to)
{
    __shared__ double sh[NV][kRedThreads / 32];
    int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    __syncthreads();
#pragma unroll
    for (int q = 0; q < NV; q++) {
        double x = MAX ? warp_max(v[q]) : warp_sum(v[q]);
        if (lane == 0) sh[q][warp] = x;
    }
    __syncthreads();
    if (threadIdx.x < 32) {
#pragma unroll
        for (int q = 0; q < NV; q++) {
            double x = lane < kRedThreads / 32 ? sh[q][lane] : 0.0;
            x = MAX ? warp_max(x) : warp_sum(x);
            if (lane == 0) to[q] = x;
        }
    }
}

// NV values per thread to the grid's totals in out: one partial per block,
// summed by the block that arrives last (*done counts the arrivals and is
// left zero; a second launch for the last sum cost 5 us)
template <int NV, bool MAX>
__device__ __forceinline__ void grid_reduce(const double *v, double *partial, unsigned *done, double *out)
{
    __shared__ bool last;
    block_reduce_store<NV, MAX>(v, partial + (size_t)blockIdx.x * NV);
    if (threadIdx.x == 0) {
        __threadfence();
        last = atomicAdd(done, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    double t[NV];
#pragma unroll
    for (int q = 0; q < NV; q++) t[q] = 0.0;
    for (int b = threadIdx.x; b < (int)gridDim.x; b += kRedThreads)
#pragma unroll
        for (int q = 0; q < NV; q++) {
            const double x = __ldcg(partial + (size_t)b * NV + q);
            t[q] = MAX ? fmax(t[q], x) : t[q] + x;
        }
    block_reduce_store<NV, MAX>(t, out);
    if (threadIdx.x == 0) *done = 0u;
}

// cell t of the interior, x fastest (the padded grid holds fewer than 2^31 cells)
__device__ __forceinline__ long long interior(const Grid &g, uint32_t t)
{
    const uint32_t r = t / (uint32_t)g.n[0];
    const int i = (int)(t - r * (uint32_t)g.n[0]);
    const int k = (int)(r / (uint32_t)g.n[1]);
    return goff(g, i, (int)(r - (uint32_t)k * (uint32_t)g.n[1]), k);
}

template <typename R>
__global__ void __launch_bounds__(kRedThreads) k_field_energy(const R *__restrict__ F, Grid g, double *partial,
                                                              unsigned *done, double *out)
{
    const uint32_t tot = (uint32_t)g.n[0] * g.n[1] * g.n[2];
    double v[2] = {0.0, 0.0};
    for (uint32_t t = blockIdx.x * kRedThreads + threadIdx.x; t < tot; t += gridDim.x * kRedThreads) {
        const long long o = interior(g, t);
#pragma unroll
        for (int c = 0; c < 3; c++) {
            const double e = widen(F[(EX + c) * g.vol + o]), b = widen(F[(BX + c) * g.vol + o]);
            v[0] += e * e;
            v[1] += b * b;
        }
    }
    grid_reduce<2, false>(v, partial, done, out);
}

// sum of (gamma - 1) = u^2 / (gamma + 1) per particle, or of |k| for photons
template <class P_t>
__global__ void __launch_bounds__(kRedThreads) k_kinetic(P_t P, int photon, double *partial, unsigned *done, double *out)
{
    double v[2] = {0.0, 0.0};
    long long live = 0;
    const long long n = *P.dn;
    for (long long p = (long long)blockIdx.x * kRedThreads + threadIdx.x; p < n; p += (long long)gridDim.x * kRedThreads) {
        if (P.cell[p] == kDead) continue;
        const double ux = widen(P.u[0][p]), uy = widen(P.u[1][p]), uz = widen(P.u[2][p]);
        const double uu = ux * ux + uy * uy + uz * uz;
        if (photon) {
            v[0] += sqrt(uu);
        } else {
            const double a = 1.0 + uu;
            if ((uint32_t)__double2hiint(a) >= 0x46000000u) v[0] += uu / (sqrt(a) + 1.0);
            else v[0] += uu * rcp_fp64(fma(a, rsqrt_fp64(a), 1.0));
        }
        live++;
    }
    v[1] = (double)live;
    grid_reduce<2, false>(v, partial, done, out);
}

// charge density of one species: q w W (W_2 or W_4, the shape the deposit
// uses) at x -/+ (dt/2) v, half each.  X: position in cells (a cell index and
// the offset from it)
template <int DIM, int ORDER>
__device__ __forceinline__ void rho_add(double *rho, const Grid &g, const int *c, const double *X, double qw2)
{
    constexpr int P = ORDER + 1, H = ORDER / 2;
    // a non-finite position has no node; the pushes remove particles whose
    // momentum became non-finite, so this only guards the index arithmetic
#pragma unroll
    for (int d = 0; d < DIM; d++)
        if (!isfinite(X[d])) return;
    int ic[3] = {0, 0, 0};
    double w[3][P];
#pragma unroll
    for (int d = 0; d < DIM; d++) {
        const double f = floor(X[d] + 0.5);
        ic[d] = c[d] + (int)f - H;
        if constexpr (ORDER == 4) w4<double>(X[d] - f, w[d]);
        else w2<double>(X[d] - f, w[d]);
    }
    double *base = rho + goff(g, ic[0], ic[1], ic[2]);
#pragma unroll
    for (int k = 0; k < (DIM > 2 ? P : 1); k++) {
        const double wz = DIM > 2 ? qw2 * w[2][k] : qw2;
#pragma unroll
        for (int b = 0; b < (DIM > 1 ? P : 1); b++) {
            const double wy = DIM > 1 ? wz * w[1][b] : wz;
#pragma unroll
            for (int a = 0; a < P; a++) atomicAdd(base + (k * g.sz + b * g.sy + a), wy * w[0][a]);
        }
    }
}

// the particle of a thread: a warp takes 256 consecutive particles in eight
// rounds, its lanes eight apart, so that the lanes of one atomic are on
// several cells (the particles are cell-sorted; lanes on one node queue up)
__device__ __forceinline__ long long rho_particle()
{
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    return (t & ~255ll) | ((t & 31) << 3) | ((t >> 5) & 7);
}

template <int DIM, int ORDER>
__global__ void __launch_bounds__(256) k_rho_f32(PartF32 P, Grid g, double hdt, double qw2, double *rho)
{
    const long long p = rho_particle();
    if (p >= *P.dn) return;
    const uint32_t cp = P.cell[p];
    if (cp == kDead) return;
    int c[3];
    unpack_cell(g, cp, c[0], c[1], c[2]);
    const double u[3] = {widen(P.u[0][p]), widen(P.u[1][p]), widen(P.u[2][p])};
    const double h = hdt * rsqrt_fp64(1.0 + u[0] * u[0] + u[1] * u[1] + u[2] * u[2]);
    double o[3] = {0, 0, 0}, d[3] = {0, 0, 0};
#pragma unroll
    for (int a = 0; a < DIM; a++) {
        o[a] = widen(P.off[a][p]);
        d[a] = h * u[a] * g.rdx_d[a];
    }
#pragma unroll
    for (int side = -1; side <= 1; side += 2) {
        const double X[3] = {o[0] + side * d[0], o[1] + side * d[1], o[2] + side * d[2]};
        rho_add<DIM, ORDER>(rho, g, c, X, qw2);
    }
}

template <int DIM, int ORDER>
__global__ void __launch_bounds__(256) k_rho_f64(PartF64 P, Grid g, double hdt, double qw2, double *rho)
{
    const long long p = rho_particle();
    if (p >= *P.dn) return;
    if (P.cell[p] == kDead) return;
    const double u[3] = {P.u[0][p], P.u[1][p], P.u[2][p]};
    const double h = hdt * rsqrt_fp64(1.0 + u[0] * u[0] + u[1] * u[1] + u[2] * u[2]);
    const int c[3] = {0, 0, 0};
#pragma unroll
    for (int side = -1; side <= 1; side += 2) {
        double X[3] = {0, 0, 0};
#pragma unroll
        for (int a = 0; a < DIM; a++) X[a] = (P.x[a][p] + side * (h * u[a])) * g.rdx_d[a];
        rho_add<DIM, ORDER>(rho, g, c, X, qw2);
    }
}

// max over interior nodes of |div E - rho - rho_bg|
// (and the tallies the diagnostics report with it: out[1] = *t1, out[2] = *t2)
template <typename R>
__global__ void __launch_bounds__(kRedThreads) k_gauss(const R *__restrict__ F, const double *__restrict__ rho, Grid g,
                                                       double rho_bg, double *partial, unsigned *done, double *out,
                                                       const double *t1, const double *t2)
{
    const uint32_t tot = (uint32_t)g.n[0] * g.n[1] * g.n[2];
    double v[1] = {0.0};
    const R *Ex = F + EX * g.vol, *Ey = F + EY * g.vol, *Ez = F + EZ * g.vol;
    for (uint32_t t = blockIdx.x * kRedThreads + threadIdx.x; t < tot; t += gridDim.x * kRedThreads) {
        const long long o = interior(g, t);
        double div = (widen(Ex[o]) - widen(Ex[o - 1])) * g.rdx_d[0];
        if (g.dim > 1) div += (widen(Ey[o]) - widen(Ey[o - g.sy])) * g.rdx_d[1];
        if (g.dim > 2) div += (widen(Ez[o]) - widen(Ez[o - g.sz])) * g.rdx_d[2];
        v[0] = fmax(v[0], fabs(div - rho[o] - rho_bg));
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        out[1] = *t1;
        out[2] = *t2;
    }
    grid_reduce<1, true>(v, partial, done, out);
}

// ---------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------
// partials, then the arrival counter of grid_reduce (zero between launches)
size_t diag_scratch_doubles() { return (size_t)kRedBlocks * 2 + 64; }
static unsigned *done_of(double *scratch) { return reinterpret_cast<unsigned *>(scratch + (size_t)kRedBlocks * 2); }
static int red_blocks(long long n) { return (int)std::max<long long>(1, std::min<long long>(kRedBlocks, div_up(n, kRedThreads))); }
static long long interior_cells(const Grid &g) { return (long long)g.n[0] * g.n[1] * g.n[2]; }

template <typename R>
void diag_field_energy(const R *F, const Grid &g, double *scratch, double *out2, cudaStream_t st)
{
    k_field_energy<R><<<red_blocks(interior_cells(g)), kRedThreads, 0, st>>>(F, g, scratch, done_of(scratch), out2);
}
template void diag_field_energy<float>(const float *, const Grid &, double *, double *, cudaStream_t);
template void diag_field_energy<double>(const double *, const Grid &, double *, double *, cudaStream_t);

void diag_kinetic_f32(const PartF32 &P, bool photon, double *scratch, double *out2, cudaStream_t st)
{
    k_kinetic<<<red_blocks(P.n), kRedThreads, 0, st>>>(P, photon ? 1 : 0, scratch, done_of(scratch), out2);
}
void diag_kinetic_f64(const PartF64 &P, bool photon, double *scratch, double *out2, cudaStream_t st)
{
    k_kinetic<<<red_blocks(P.n), kRedThreads, 0, st>>>(P, photon ? 1 : 0, scratch, done_of(scratch), out2);
}

void diag_rho_f32(const PartF32 &P, const Grid &g, double qw, double *rho, cudaStream_t st)
{
    if (P.n == 0 || qw == 0.0) return;  // (photons: no charge)
    int nb = div_up(P.n, 256);
    double h = 0.5 * g.dt;
    if (g.order == 4) {
        if (g.dim == 1) k_rho_f32<1, 4><<<nb, 256, 0, st>>>(P, g, h, 0.5 * qw, rho);
        else if (g.dim == 2) k_rho_f32<2, 4><<<nb, 256, 0, st>>>(P, g, h, 0.5 * qw, rho);
        else k_rho_f32<3, 4><<<nb, 256, 0, st>>>(P, g, h, 0.5 * qw, rho);
        return;
    }
    if (g.dim == 1) k_rho_f32<1, 2><<<nb, 256, 0, st>>>(P, g, h, 0.5 * qw, rho);
    else if (g.dim == 2) k_rho_f32<2, 2><<<nb, 256, 0, st>>>(P, g, h, 0.5 * qw, rho);
    else k_rho_f32<3, 2><<<nb, 256, 0, st>>>(P, g, h, 0.5 * qw, rho);
}
void diag_rho_f64(const PartF64 &P, const Grid &g, double qw, double *rho, cudaStream_t st)
{
    if (P.n == 0 || qw == 0.0) return;  // (photons: no charge)
    int nb = div_up(P.n, 256);
    double h = 0.5 * g.dt;
    if (g.order == 4) {
        if (g.dim == 1) k_rho_f64<1, 4><<<nb, 256, 0, st>>>(P, g, h, 0.5 * qw, rho);
        else if (g.dim == 2) k_rho_f64<2, 4><<<nb, 256, 0, st>>>(P, g, h, 0.5 * qw, rho);
        else k_rho_f64<3, 4><<<nb, 256, 0, st>>>(P, g, h, 0.5 * qw, rho);
        return;
    }
    if (g.dim == 1) k_rho_f64<1, 2><<<nb, 256, 0, st>>>(P, g, h, 0.5 * qw, rho);
    else if (g.dim == 2) k_rho_f64<2, 2><<<nb, 256, 0, st>>>(P, g, h, 0.5 * qw, rho);
    else k_rho_f64<3, 2><<<nb, 256, 0, st>>>(P, g, h, 0.5 * qw, rho);
}

template <typename R>
void diag_gauss(const R *F, const double *rho, const Grid &g, double rho_bg, const double *t1, const double *t2,
                double *scratch, double *out3, cudaStream_t st)
{
    k_gauss<R><<<red_blocks(interior_cells(g)), kRedThreads, 0, st>>>(F, rho, g, rho_bg, scratch, done_of(scratch), out3,
                                                                     t1, t2);
}
template void diag_gauss<float>(const float *, const double *, const Grid &, double, const double *, const double *,
                                double *, double *, cudaStream_t);
template void diag_gauss<double>(const double *, const double *, const Grid &, double, const double *, const double *,
                                 double *, double *, cudaStream_t);

// ---------------------------------------------------------------------
// exchange layout (FP64, x fastest, [0, N) or [0, N] per axis) <-> padded
// component: one thread per padded cell of a row, so that a component crosses
// to the host as one dense block and the host walks no arrays.  The blocks of
// a plane are numbered along x and planes are strided over (a launch's y and z
// hold 65535 blocks, and a grid may have more rows than four times that, or more
// planes)
// ---------------------------------------------------------------------
struct ExBox {
    int m[3];
};

// this thread's row and column of a plane of e0 x e1 cells
__device__ __forceinline__ bool ex_cell(int e0, int e1, int &i, int &j)
{
    const unsigned ny = (e1 + blockDim.y - 1) / blockDim.y, bx = blockIdx.x / ny;
    i = bx * blockDim.x + threadIdx.x;
    j = (blockIdx.x - bx * ny) * blockDim.y + threadIdx.y;
    return i < e0 && j < e1;
}

template <typename R>
__global__ void __launch_bounds__(256) k_pack(const R *__restrict__ comp, Grid g, ExBox b, double *__restrict__ out)
{
    int i, j;
    if (!ex_cell(b.m[0], b.m[1], i, j)) return;
    for (int k = blockIdx.y; k < b.m[2]; k += gridDim.y)
        out[((long long)k * b.m[1] + j) * b.m[0] + i] = (double)comp[goff(g, i, j, k)];
}

// every padded cell whose (periodic image of the) index lies in the box
template <typename R>
__global__ void __launch_bounds__(256) k_unpack(const double *__restrict__ src, Grid g, ExBox b, R *__restrict__ comp)
{
    int i, j;
    if (!ex_cell(g.ext[0], g.ext[1], i, j)) return;
    for (int k = blockIdx.y; k < g.ext[2]; k += gridDim.y) {
        int p[3] = {i - g.G[0], j - g.G[1], k - g.G[2]};
        const long long o = goff(g, p[0], p[1], p[2]);
        bool in = true;
#pragma unroll
        for (int d = 0; d < 3; d++) {
            if (d >= g.dim) continue;
            if (g.bc[d] == PERIODIC) p[d] = (p[d] % g.n[d] + g.n[d]) % g.n[d];
            else in &= p[d] >= 0 && p[d] < b.m[d];
        }
        if (in) comp[o] = (R)src[((long long)p[2] * b.m[1] + p[1]) * b.m[0] + p[0]];
    }
}

static dim3 ex_block(const Grid &g) { return g.dim == 1 ? dim3(256, 1, 1) : dim3(64, 4, 1); }
static dim3 ex_grid(const dim3 &blk, long long e0, long long e1, long long e2)
{
    return dim3((unsigned)div_up(e0, blk.x) * (unsigned)div_up(e1, blk.y), (unsigned)std::min(e2, 65535ll));
}

template <typename R>
void field_pack(const R *comp, const Grid &g, const long long *m, double *out, cudaStream_t st)
{
    const ExBox b{{(int)m[0], (int)m[1], (int)m[2]}};
    const dim3 blk = ex_block(g);
    k_pack<R><<<ex_grid(blk, m[0], m[1], m[2]), blk, 0, st>>>(comp, g, b, out);
}
template void field_pack<float>(const float *, const Grid &, const long long *, double *, cudaStream_t);
template void field_pack<double>(const double *, const Grid &, const long long *, double *, cudaStream_t);

template <typename R>
void field_unpack(const double *in, const Grid &g, const long long *m, R *comp, cudaStream_t st)
{
    const ExBox b{{(int)m[0], (int)m[1], (int)m[2]}};
    const dim3 blk = ex_block(g);
    k_unpack<R><<<ex_grid(blk, g.ext[0], g.ext[1], g.ext[2]), blk, 0, st>>>(in, g, b, comp);
}
template void field_unpack<float>(const double *, const Grid &, const long long *, float *, cudaStream_t);
template void field_unpack<double>(const double *, const Grid &, const long long *, double *, cudaStream_t);

}  // namespace pic
