// fdtd.cu -- Yee FDTD half steps (Eqs. (9), (10) over dt/2), the Mur
// absorbing faces with the laser entering through x-min, and the current
// fold of the ghost layers.
//
// One thread per padded cell, x fastest within a block: rows are read and
// written with unit stride (coalesced) and no thread does integer division.
// Blocks run through y before x: the ones at the x-min face, where the
// laser's sines are a long chain in one lane of a warp, start first and hide
// behind the others (2048 x 1024 cells, absorbing x faces and a laser: the
// field launches of a step took 55.6 us with the rows' blocks in their order,
// now 49.4; in FP64 242 and 209 us).  What bounds an update otherwise is
// memory: 277 MB a step in 42 us on periodic axes.
// Each thread updates the three components of its cell.  Along
// periodic axes the ghost layers are computed directly (a neighbour that
// falls off the padded box is taken one period away), so they stay
// bit-identical copies of their images without a separate exchange.
//
// E update modes: a half step (dt/2), or the second half step of step n
// fused with the first half step of step n+1 -- both use the same curl B and
// the same J^{n+1}, applied twice in registers, which gives the same bits as
// two separate launches while reading and writing E once.
#include "fdtd.cuh"

namespace pic {

// offset of the neighbour one cell along axis d (dir = +1/-1) of the cell
// at padded coordinate p, taken one period away at the padded edge
__device__ __forceinline__ int nb_off(const Grid &g, int d, int p, int dir)
{
    int s = d == 0 ? 1 : (d == 1 ? (int)g.sy : (int)g.sz);
    int q = p + dir;
    if (q < -g.G[d]) q += g.n[d];
    else if (q >= g.n[d] + g.G[d]) q -= g.n[d];
    return (q - p) * s;
}

// per-thread masks: bit d of `half_ok` / `node_ok` = the coordinate along
// axis d lies in the physical half-node / node range (always on periodic or
// inactive axes); component c is updated when every axis agrees
struct Phys {
    int half_ok, node_ok;
    __device__ __forceinline__ bool comp(int c) const
    {
        int ok = 1;
#pragma unroll
        for (int d = 0; d < 3; d++) ok &= stag(c, d) ? (half_ok >> d) : (node_ok >> d);
        return ok & 1;
    }
};

__device__ __forceinline__ Phys phys_of(const Grid &g, int i, int j, int k)
{
    int p[3] = {i, j, k};
    Phys r{7, 7};
#pragma unroll
    for (int d = 0; d < 3; d++) {
        if (d >= g.dim || g.bc[d] == PERIODIC) continue;
        if (p[d] < 0 || p[d] > g.n[d] - 1) r.half_ok &= ~(1 << d);
        if (p[d] < 0 || p[d] > g.n[d]) r.node_ok &= ~(1 << d);
    }
    return r;
}

// thread blocks: 256 along x in 1D, else kBlockX by kBlockY
constexpr unsigned kBlockX = 64, kBlockY = 4;

// (nf: leading blocks of the launch that fold instead)
__device__ __forceinline__ bool thread_cell(const Grid &g, int &i, int &j, int &k, unsigned nf = 0)
{
    const unsigned ny = ((unsigned)g.ext[1] + kBlockY - 1) / kBlockY;
    const unsigned b = blockIdx.x - nf, bx = b / ny;  // (1D: ny = 1)
    i = bx * blockDim.x + threadIdx.x;
    j = (b - bx * ny) * blockDim.y + threadIdx.y;
    k = blockIdx.y;
    if (i >= g.ext[0] || j >= g.ext[1]) return false;
    i -= g.G[0];
    j -= g.G[1];
    k -= g.G[2];
    return true;
}

__device__ __forceinline__ int loff(const Grid &g, int i, int j, int k)
{
    return (int)g.origin + k * (int)g.sz + j * (int)g.sy + i;
}

// A set of ncomp arrays (base + q*stride) with per-component staggering
// masks (bit d set = half node along axis d), e.g. Jx,Jy,Jz or rho.
struct FoldSet {
    int ncomp;
    long long stride;
    int mask[3];
};

// The fold of every axis at once.  Along a
// periodic axis what was deposited into a ghost belongs to its image, and both
// end up holding the sum (image + ghost, fixed order: x first); along an
// absorbing axis what was deposited outside the physical range leaves the
// domain and is discarded.  One thread per root cell: its coordinate along a
// periodic axis lies in [0, N), along another anywhere in the padded range,
// and along at least one axis it is in the shell that has work (the first such
// axis owns it).
struct FoldGrid {
    int shell[3], rest[3];   // roots per axis in and outside the shell
    unsigned first[4];       // first thread of each axis' share
};

__device__ __forceinline__ int shell_at(const Grid &g, int d, int u)
{
    if (g.bc[d] == PERIODIC) return u < g.G[d] ? u : g.n[d] - 2 * g.G[d] + u;
    return u < g.G[d] ? u - g.G[d] : g.n[d] + (u - g.G[d]);
}
__device__ __forceinline__ int rest_at(const Grid &g, int d, int u) { return g.bc[d] == PERIODIC ? u + g.G[d] : u; }

template <typename R, int DIM>
__device__ __forceinline__ void fold_root(R *base, const FoldSet &fs, const Grid &g, const FoldGrid &fg, unsigned t)
{
    int d = 0;
    unsigned u = t;
#pragma unroll
    for (int a = 1; a < DIM; a++)
        if (t >= fg.first[a]) {
            d = a;
            u = t - fg.first[a];
        }
    int p[3] = {0, 0, 0}, step[3] = {0, 0, 0};  // step: to the partner along a periodic axis
#pragma unroll
    for (int a = 0; a < DIM; a++) {
        const int in = fg.shell[a], out = fg.rest[a];
        const unsigned m = a == d ? in : (a < d ? out : in + out);
        const int v = (int)(u % m);
        u /= m;
        // (past the owning axis: the shell's roots, then the others)
        p[a] = a == d || (a > d && v < in) ? shell_at(g, a, v) : rest_at(g, a, a > d ? v - in : v);
        if (g.bc[a] == PERIODIC) step[a] = p[a] < g.G[a] ? g.n[a] : (p[a] >= g.n[a] - g.G[a] ? -g.n[a] : 0);
    }
    const int s[3] = {1, (int)g.sy, (int)g.sz};
#pragma unroll
    for (int q = 0; q < 3; q++) {
        if (q >= fs.ncomp) break;
        bool gone = false;
#pragma unroll
        for (int a = 0; a < DIM; a++)
            if (g.bc[a] != PERIODIC) gone |= p[a] < 0 || p[a] > (((fs.mask[q] >> a) & 1) ? g.n[a] - 1 : g.n[a]);
        R *J = base + q * fs.stride + loff(g, p[0], p[1], p[2]);
        // the root and its partners, x pairs first
        R v[1 << DIM];
#pragma unroll
        for (int m = 0; m < 1 << DIM; m++) {
            int o = 0;
            bool is = true;
#pragma unroll
            for (int a = 0; a < DIM; a++)
                if ((m >> a) & 1) {
                    is &= step[a] != 0;
                    o += step[a] * s[a];
                }
            v[m] = is ? J[o] : R(0);
        }
#pragma unroll
        for (int a = 0; a < DIM; a++)
#pragma unroll
            for (int m = 0; m < 1 << DIM; m++)
                if (!((m >> a) & 1) && (m & ((1 << a) - 1)) == 0 && step[a]) v[m] = v[m] + v[m | 1 << a];
        const R sum = gone ? R(0) : v[0];
#pragma unroll
        for (int m = 0; m < 1 << DIM; m++) {
            int o = 0;
            bool is = true;
#pragma unroll
            for (int a = 0; a < DIM; a++)
                if ((m >> a) & 1) {
                    is &= step[a] != 0;
                    o += step[a] * s[a];
                }
            if (is) J[o] = sum;
        }
    }
}

// The fold of J needs neither E nor B: its blocks lead the launch of the B half
// step after a push (nb of them in each of the gridDim.y z layers; none: no
// fold).  As a launch for each axis the fold cost a 2D step of 2048 x 1024
// cells 5.3 us (periodic: 47.4 before, 42.0 now) and a small one 4 us.
struct FoldBlocks {
    unsigned nb;
    FoldSet fs;
    FoldGrid fg;
};

template <typename R, int DIM>
__device__ __forceinline__ void fold_block(R *F, const Grid &g, const FoldBlocks &fb)
{
    const unsigned t = (blockIdx.y * fb.nb + blockIdx.x) * (blockDim.x * blockDim.y) + threadIdx.y * blockDim.x + threadIdx.x;
    if (t < fb.fg.first[DIM]) fold_root<R, DIM>(F + JX * g.vol, fb.fs, g, fb.fg, t);
}

// E += h (curl B - J), once (mode 0) or twice (mode 1); then J = 0 when
// zeroJ (J^n is no longer needed once the first half step of step n used it)
template <typename R, int DIM>
__device__ __forceinline__ void cell_E(R *F, const Grid &g, R h, int twice, int zeroJ, int i, int j, int k)
{
    const int o = loff(g, i, j, k);
    const long long V = g.vol;
    const R *__restrict__ Bx = F + BX * V;
    const R *__restrict__ By = F + BY * V;
    const R *__restrict__ Bz = F + BZ * V;
    R *Ex = F + EX * V, *Ey = F + EY * V, *Ez = F + EZ * V;
    R *Jx = F + JX * V, *Jy = F + JY * V, *Jz = F + JZ * V;
    const R rdx = pic::rdx<R>(g, 0), rdy = pic::rdx<R>(g, 1), rdz = pic::rdx<R>(g, 2);
    R cx = 0, cy = 0, cz = 0;
    const int mx = nb_off(g, 0, i, -1);
    cy -= (Bz[o] - Bz[o + mx]) * rdx;
    cz += (By[o] - By[o + mx]) * rdx;
    if (DIM >= 2) {
        const int my = nb_off(g, 1, j, -1);
        cx += (Bz[o] - Bz[o + my]) * rdy;
        cz -= (Bx[o] - Bx[o + my]) * rdy;
    }
    if (DIM >= 3) {
        const int mz = nb_off(g, 2, k, -1);
        cx -= (By[o] - By[o + mz]) * rdz;
        cy += (Bx[o] - Bx[o + mz]) * rdz;
    }
    const R jx = Jx[o], jy = Jy[o], jz = Jz[o];
    const Phys ph = phys_of(g, i, j, k);
    const R ax = h * (cx - jx), ay = h * (cy - jy), az = h * (cz - jz);
    if (ph.comp(EX)) { R e = Ex[o] + ax; if (twice) e += ax; Ex[o] = e; }
    if (ph.comp(EY)) { R e = Ey[o] + ay; if (twice) e += ay; Ey[o] = e; }
    if (ph.comp(EZ)) { R e = Ez[o] + az; if (twice) e += az; Ez[o] = e; }
    if (zeroJ) { Jx[o] = 0; Jy[o] = 0; Jz[o] = 0; }
}

template <typename R, int DIM>
__global__ void __launch_bounds__(256) k_update_E(R *__restrict__ F, Grid g, R h, int twice, int zeroJ)
{
    int i, j, k;
    if (thread_cell(g, i, j, k)) cell_E<R, DIM>(F, g, h, twice, zeroJ, i, j, k);
}

// incident B of the laser (a +x wave: Bz = Ey, By = -Ez) at time point q
// (see Laser); (j, k) are wrapped to the interior so that periodic ghost rows
// see the same laser as their images.  Rows outside the profile get none.
__device__ __forceinline__ float sin_r(float x) { return sinf(x); }
__device__ __forceinline__ double sin_r(double x) { return sin(x); }
__device__ __forceinline__ float cos_r(float x) { return cosf(x); }
__device__ __forceinline__ double cos_r(double x) { return cos(x); }

template <typename R>
__device__ inline R incident_B(const Grid &g, const Laser &L, int c, int q, int j, int k)
{
    if (g.dim >= 2 && g.bc[1] == PERIODIC) { j %= g.n[1]; if (j < 0) j += g.n[1]; }
    if (g.dim >= 3 && g.bc[2] == PERIODIC) { k %= g.n[2]; if (k < 0) k += g.n[2]; }
    if (g.dim < 2) j = 0;
    if (g.dim < 3) k = 0;
    if (j < 0 || j >= L.nty || k < 0 || k >= L.ntz) return R(0);
    const int t = k * L.nty + j;
    const R ph = (R)L.ph0[q];
    const R env = (R)L.env[q];
    if (c == BZ) {
        const R *A = (const R *)L.A[0], *P = (const R *)L.PHI[0];
        return A[t] * env * sin_r(ph + P[t]);
    }
    if (c == BY && L.pol == 1) {
        const R *A = (const R *)L.A[1], *P = (const R *)L.PHI[1];
        return -A[t] * env * cos_r(ph + P[t]);
    }
    return R(0);
}

template <typename R, int DIM>
__device__ __forceinline__ void mur_faces(R *const *B, const Grid &g, R h, const Laser &L, int i, int j, int k, int o,
                                          const R *oldv);

// B -= h curl E, then the Mur ghosts of the tangential B on absorbing
// faces: for the scattered part s = B - B_inc of an outgoing wave,
// s_ghost(new) = s_inner(old) + (a-1)/(a+1) (s_inner(new) - s_ghost(old)),
// a = h/dx.  The thread owning the first inner value writes the ghost.
template <typename R, int DIM>
__device__ __forceinline__ void cell_B(R *F, const Grid &g, R h, const Laser &L, int i, int j, int k)
{
    const int o = loff(g, i, j, k);
    const long long V = g.vol;
    const R *__restrict__ Ex = F + EX * V;
    const R *__restrict__ Ey = F + EY * V;
    const R *__restrict__ Ez = F + EZ * V;
    R *B[3] = {F + BX * V, F + BY * V, F + BZ * V};
    const R rdx = pic::rdx<R>(g, 0), rdy = pic::rdx<R>(g, 1), rdz = pic::rdx<R>(g, 2);
    R cx = 0, cy = 0, cz = 0;
    const int px = nb_off(g, 0, i, +1);
    cy -= (Ez[o + px] - Ez[o]) * rdx;
    cz += (Ey[o + px] - Ey[o]) * rdx;
    if (DIM >= 2) {
        const int py = nb_off(g, 1, j, +1);
        cx += (Ez[o + py] - Ez[o]) * rdy;
        cz -= (Ex[o + py] - Ex[o]) * rdy;
    }
    if (DIM >= 3) {
        const int pz = nb_off(g, 2, k, +1);
        cx -= (Ey[o + pz] - Ey[o]) * rdz;
        cy += (Ex[o + pz] - Ex[o]) * rdz;
    }
    const R cur[3] = {cx, cy, cz};
    const Phys ph = phys_of(g, i, j, k);
    R oldv[3];
#pragma unroll
    for (int c = 0; c < 3; c++) {
        oldv[c] = B[c][o];
        if (ph.comp(BX + c)) B[c][o] = oldv[c] - h * cur[c];
    }
    mur_faces<R, DIM>(B, g, h, L, i, j, k, o, oldv);
}

template <typename R, int DIM>
__global__ void __launch_bounds__(256) k_update_B(R *__restrict__ F, Grid g, R h, Laser L, FoldBlocks fb)
{
    int i, j, k;
    if (blockIdx.x < fb.nb) {
        fold_block<R, DIM>(F, g, fb);
        return;
    }
    if (thread_cell(g, i, j, k, fb.nb)) cell_B<R, DIM>(F, g, h, L, i, j, k);
}

// the Mur ghosts of cell (i, j, k) at offset o, after its B update (oldv:
// its B before the update).  Component c is staggered along the two axes
// other than c; a ghost beyond two faces at once belongs to the cell inside
// both, which takes the passes along the axes in their order, so the result
// does not depend on the order of the blocks.
template <typename R, int DIM>
__device__ __forceinline__ void mur_faces(R *const *B, const Grid &g, R h, const Laser &L, int i, int j, int k, int o,
                                          const R *oldv)
{
    const int p[3] = {i, j, k};
#pragma unroll
    for (int c = 0; c < 3; c++) {
        const int d1 = c == 0 ? 1 : 0, d2 = c == 2 ? 1 : 2;
        if (d1 >= DIM) continue;
        // a swept (updated) position along the axis c, and inside the faces along the other two
        if (c < DIM && g.bc[c] == ABSORB && (p[c] < 0 || p[c] > g.n[c])) continue;
        const bool ab1 = g.bc[d1] == ABSORB, ab2 = d2 < DIM && g.bc[d2] == ABSORB;
        if ((ab1 && (p[d1] < 0 || p[d1] >= g.n[d1])) || (ab2 && (p[d2] < 0 || p[d2] >= g.n[d2]))) continue;
        const bool at1 = ab1 && (p[d1] == 0 || p[d1] == g.n[d1] - 1), at2 = ab2 && (p[d2] == 0 || p[d2] == g.n[d2] - 1);
        if (!at1 && !at2) continue;
        const int s1 = d1 == 0 ? 1 : (int)g.sy, s2 = d2 == 1 ? (int)g.sy : (int)g.sz;
        const R a1 = h * pic::rdx<R>(g, d1), a2 = d2 < DIM ? h * pic::rdx<R>(g, d2) : R(0);
        const R m1 = at1 ? (a1 - R(1)) / (a1 + R(1)) : R(0), m2 = at2 ? (a2 - R(1)) / (a2 + R(1)) : R(0);
        R *Bc = B[c] + o;
        for (int f1 = 0; f1 < 3; f1++) {  // faces of axis d1: low, high, none
            if (f1 == 0 && !(ab1 && p[d1] == 0)) continue;
            if (f1 == 1 && !(ab1 && p[d1] == g.n[d1] - 1)) continue;
            if (f1 == 2 && !at2) continue;
            const int o1 = f1 == 0 ? -s1 : (f1 == 1 ? s1 : 0);
            R ig_new = 0, ig_old = 0, ii_new = 0, ii_old = 0;
            if (f1 == 0 && d1 == 0 && L.on) {
                ig_new = incident_B<R>(g, L, BX + c, 0, j, k);
                ig_old = incident_B<R>(g, L, BX + c, 1, j, k);
                ii_new = incident_B<R>(g, L, BX + c, 2, j, k);
                ii_old = incident_B<R>(g, L, BX + c, 3, j, k);
            }
            R g1_old = 0, g1_new = 0;
            if (f1 < 2) {
                g1_old = Bc[o1];
                const R sg_old = g1_old - ig_old;
                const R si_old = oldv[c] - ii_old;
                const R si_new = Bc[0] - ii_new;
                g1_new = ig_new + si_old + m1 * (si_new - sg_old);
            }
            for (int f2 = 0; f2 < 2; f2++) {
                if (!(ab2 && p[d2] == (f2 == 0 ? 0 : g.n[d2] - 1))) continue;
                const int o2 = f2 == 0 ? -s2 : s2;
                const R g2_old = Bc[o2];
                if (f1 == 2) {
                    Bc[o2] = oldv[c] + m2 * (Bc[0] - g2_old);
                    continue;
                }
                // beyond both faces: along d1 at the swept row (the high one), then along d2 likewise
                R v = Bc[o1 + o2];
                if (f2 == 1) v = g2_old + m1 * (g2_old - v);
                if (f1 == 1) v = g1_old + m2 * (g1_new - v);
                Bc[o1 + o2] = v;
            }
            if (f1 < 2) Bc[o1] = g1_new;
        }
    }
}

// ---------------------------------------------------------------------
// FP32, four cells per thread along x (float4 loads and stores; the padded
// rows start 16-byte aligned and hold a multiple of 4 cells when n_x is a
// multiple of 4).  Same arithmetic, in the same order, as the one-cell
// kernels above.  A component is stored as a vector when all four cells are
// physical for it, else cell by cell (ghost cells on absorbing axes belong
// to the Mur update).
// ---------------------------------------------------------------------
__device__ __forceinline__ float4 ld4(const float *p) { return *reinterpret_cast<const float4 *>(p); }
__device__ __forceinline__ void st4(float *p, const float (&v)[4])
{
    *reinterpret_cast<float4 *>(p) = make_float4(v[0], v[1], v[2], v[3]);
}
__device__ __forceinline__ void unpack4(const float4 &a, float (&v)[4])
{
    v[0] = a.x;
    v[1] = a.y;
    v[2] = a.z;
    v[3] = a.w;
}

__device__ __forceinline__ bool thread_cell4(const Grid &g, int &i, int &j, int &k, unsigned nf = 0)
{
    const unsigned ny = ((unsigned)g.ext[1] + kBlockY - 1) / kBlockY;
    const unsigned b = blockIdx.x - nf, bx = b / ny;
    i = 4 * (bx * blockDim.x + threadIdx.x);
    j = (b - bx * ny) * blockDim.y + threadIdx.y;
    k = blockIdx.y;
    if (i >= g.ext[0] || j >= g.ext[1]) return false;
    i -= g.G[0];
    j -= g.G[1];
    k -= g.G[2];
    return true;
}

__device__ __forceinline__ void store_phys(float *A, int o, const float (&v)[4], const Phys (&ph)[4], int c)
{
    const bool all = ph[0].comp(c) && ph[1].comp(c) && ph[2].comp(c) && ph[3].comp(c);
    if (all) {
        st4(A + o, v);
    } else {
#pragma unroll
        for (int e = 0; e < 4; e++)
            if (ph[e].comp(c)) A[o + e] = v[e];
    }
}

template <int DIM>
__global__ void __launch_bounds__(256) k_update_E4(float *__restrict__ F, Grid g, float h, int twice, int zeroJ)
{
    int i, j, k;
    if (!thread_cell4(g, i, j, k)) return;
    const int o = loff(g, i, j, k);
    const long long V = g.vol;
    const float *__restrict__ Bx = F + BX * V;
    const float *__restrict__ By = F + BY * V;
    const float *__restrict__ Bz = F + BZ * V;
    float *E[3] = {F + EX * V, F + EY * V, F + EZ * V};
    float *J[3] = {F + JX * V, F + JY * V, F + JZ * V};
    const float rdx = g.rdx_f[0], rdy = g.rdx_f[1], rdz = g.rdx_f[2];
    float bz[4], by[4];
    unpack4(ld4(Bz + o), bz);
    unpack4(ld4(By + o), by);
    const int mx = nb_off(g, 0, i, -1);
    const float bzl = Bz[o + mx], byl = By[o + mx];
    float cx[4] = {0.f, 0.f, 0.f, 0.f}, cy[4] = {0.f, 0.f, 0.f, 0.f}, cz[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int e = 0; e < 4; e++) {
        cy[e] -= (bz[e] - (e ? bz[e - 1] : bzl)) * rdx;
        cz[e] += (by[e] - (e ? by[e - 1] : byl)) * rdx;
    }
    float bx[4];
    if (DIM >= 2) {
        const int my = nb_off(g, 1, j, -1);
        float bzm[4], bxm[4];
        unpack4(ld4(Bx + o), bx);
        unpack4(ld4(Bz + o + my), bzm);
        unpack4(ld4(Bx + o + my), bxm);
#pragma unroll
        for (int e = 0; e < 4; e++) {
            cx[e] += (bz[e] - bzm[e]) * rdy;
            cz[e] -= (bx[e] - bxm[e]) * rdy;
        }
    }
    if (DIM >= 3) {
        const int mz = nb_off(g, 2, k, -1);
        float bym[4], bxm[4];
        unpack4(ld4(By + o + mz), bym);
        unpack4(ld4(Bx + o + mz), bxm);
#pragma unroll
        for (int e = 0; e < 4; e++) {
            cx[e] -= (by[e] - bym[e]) * rdz;
            cy[e] += (bx[e] - bxm[e]) * rdz;
        }
    }
    Phys ph[4];
#pragma unroll
    for (int e = 0; e < 4; e++) ph[e] = phys_of(g, i + e, j, k);
    const float *cur[3] = {cx, cy, cz};
#pragma unroll
    for (int c = 0; c < 3; c++) {
        float jv[4], ev[4];
        unpack4(ld4(J[c] + o), jv);
        unpack4(ld4(E[c] + o), ev);
#pragma unroll
        for (int e = 0; e < 4; e++) {
            const float a = h * (cur[c][e] - jv[e]);
            ev[e] += a;
            if (twice) ev[e] += a;
        }
        store_phys(E[c], o, ev, ph, EX + c);
    }
    if (zeroJ) {
        const float z[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int c = 0; c < 3; c++) st4(J[c] + o, z);
    }
}

template <int DIM>
__global__ void __launch_bounds__(256) k_update_B4(float *__restrict__ F, Grid g, float h, Laser L, FoldBlocks fb)
{
    int i, j, k;
    if (blockIdx.x < fb.nb) {
        fold_block<float, DIM>(F, g, fb);
        return;
    }
    if (!thread_cell4(g, i, j, k, fb.nb)) return;
    const int o = loff(g, i, j, k);
    const long long V = g.vol;
    const float *__restrict__ Ex = F + EX * V;
    const float *__restrict__ Ey = F + EY * V;
    const float *__restrict__ Ez = F + EZ * V;
    float *B[3] = {F + BX * V, F + BY * V, F + BZ * V};
    const float rdx = g.rdx_f[0], rdy = g.rdx_f[1], rdz = g.rdx_f[2];
    float ez[4], ey[4];
    unpack4(ld4(Ez + o), ez);
    unpack4(ld4(Ey + o), ey);
    const int px = nb_off(g, 0, i + 3, +1);
    const float ezr = Ez[o + 3 + px], eyr = Ey[o + 3 + px];
    float cx[4] = {0.f, 0.f, 0.f, 0.f}, cy[4] = {0.f, 0.f, 0.f, 0.f}, cz[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int e = 0; e < 4; e++) {
        cy[e] -= ((e < 3 ? ez[e + 1] : ezr) - ez[e]) * rdx;
        cz[e] += ((e < 3 ? ey[e + 1] : eyr) - ey[e]) * rdx;
    }
    float ex[4];
    if (DIM >= 2) {
        const int py = nb_off(g, 1, j, +1);
        float ezp[4], exp_[4];
        unpack4(ld4(Ex + o), ex);
        unpack4(ld4(Ez + o + py), ezp);
        unpack4(ld4(Ex + o + py), exp_);
#pragma unroll
        for (int e = 0; e < 4; e++) {
            cx[e] += (ezp[e] - ez[e]) * rdy;
            cz[e] -= (exp_[e] - ex[e]) * rdy;
        }
    }
    if (DIM >= 3) {
        const int pz = nb_off(g, 2, k, +1);
        float eyp[4], exp_[4];
        unpack4(ld4(Ey + o + pz), eyp);
        unpack4(ld4(Ex + o + pz), exp_);
#pragma unroll
        for (int e = 0; e < 4; e++) {
            cx[e] -= (eyp[e] - ey[e]) * rdz;
            cy[e] += (exp_[e] - ex[e]) * rdz;
        }
    }
    Phys ph[4];
#pragma unroll
    for (int e = 0; e < 4; e++) ph[e] = phys_of(g, i + e, j, k);
    const float *cur[3] = {cx, cy, cz};
    float oldv[3][4];
#pragma unroll
    for (int c = 0; c < 3; c++) {
        float nv[4];
        unpack4(ld4(B[c] + o), oldv[c]);
#pragma unroll
        for (int e = 0; e < 4; e++) nv[e] = oldv[c][e] - h * cur[c][e];
        store_phys(B[c], o, nv, ph, BX + c);
    }
    // Mur ghosts: only groups that touch an absorbing face
    bool face = false;
#pragma unroll
    for (int d = 0; d < DIM; d++) {
        if (g.bc[d] != ABSORB) continue;
        const int lo = d == 0 ? i : (d == 1 ? j : k), hi = d == 0 ? i + 3 : lo;
        face |= (lo <= 0 && hi >= 0) || (lo <= g.n[d] - 1 && hi >= g.n[d] - 1);
    }
    if (face) {
#pragma unroll
        for (int e = 0; e < 4; e++) {
            const float ov[3] = {oldv[0][e], oldv[1][e], oldv[2][e]};
            mur_faces<float, DIM>(B, g, h, L, i + e, j, k, o + e, ov);
        }
    }
}

// (the charge density's, on its own)
template <int DIM>
__global__ void __launch_bounds__(256) k_fold(double *__restrict__ base, FoldSet fs, Grid g, FoldGrid fg)
{
    const unsigned t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t < fg.first[DIM]) fold_root<double, DIM>(base, fs, g, fg, t);
}

// A 1D grid's share of a step between two pushes in one CTA: the fold, B half,
// E (once, or twice between steps), B half, with a barrier where the launches
// of larger grids end (256 cells: 16.6 us a step as four launches, 6.3 as one).
struct Fields1d {
    int fold, b1, twice, zeroJ, b2;
};

template <typename R>
__global__ void __launch_bounds__(1024) k_fields_1d(R *__restrict__ F, Grid g, R h, Fields1d what, FoldSet fs, FoldGrid fg,
                                                    Laser L1, Laser L2)
{
    if (what.fold) {
        for (unsigned t = threadIdx.x; t < fg.first[1]; t += blockDim.x) fold_root<R, 1>(F + JX * g.vol, fs, g, fg, t);
        // (the update of E reads J after the next barrier)
    }
    if (what.b1) {
        for (int i = threadIdx.x - g.G[0]; i < g.n[0] + g.G[0]; i += blockDim.x) cell_B<R, 1>(F, g, h, L1, i, 0, 0);
    }
    __syncthreads();
    for (int i = threadIdx.x - g.G[0]; i < g.n[0] + g.G[0]; i += blockDim.x)
        cell_E<R, 1>(F, g, h, what.twice, what.zeroJ, i, 0, 0);
    if (!what.b2) return;
    __syncthreads();
    for (int i = threadIdx.x - g.G[0]; i < g.n[0] + g.G[0]; i += blockDim.x) cell_B<R, 1>(F, g, h, L2, i, 0, 0);
}

// ---------------------------------------------------------------------
// host launchers
// ---------------------------------------------------------------------

static void grid_dims(const Grid &g, int e0, int e1, int e2, dim3 &blk, dim3 &grd)
{
    if (g.dim == 1) blk = dim3(256, 1, 1);
    else blk = dim3(kBlockX, kBlockY, 1);
    grd = dim3((unsigned)div_up(e1, blk.y) * (unsigned)div_up(e0, blk.x), (unsigned)e2);
}

static bool vec4_ok(const Grid &g) { return g.n[0] % 4 == 0 && g.G[0] % 4 == 0; }

template <typename R>
void launch_update_E(R *F, const Grid &g, double h, bool twice, bool zeroJ, cudaStream_t st)
{
    dim3 b, n;
    note_launch();
    if constexpr (sizeof(R) == 4) {
        if (vec4_ok(g)) {
            grid_dims(g, g.ext[0] / 4, g.ext[1], g.ext[2], b, n);
            if (g.dim == 1) k_update_E4<1><<<n, b, 0, st>>>(F, g, (float)h, twice, zeroJ);
            else if (g.dim == 2) k_update_E4<2><<<n, b, 0, st>>>(F, g, (float)h, twice, zeroJ);
            else k_update_E4<3><<<n, b, 0, st>>>(F, g, (float)h, twice, zeroJ);
            return;
        }
    }
    grid_dims(g, g.ext[0], g.ext[1], g.ext[2], b, n);
    if (g.dim == 1) k_update_E<R, 1><<<n, b, 0, st>>>(F, g, (R)h, twice, zeroJ);
    else if (g.dim == 2) k_update_E<R, 2><<<n, b, 0, st>>>(F, g, (R)h, twice, zeroJ);
    else k_update_E<R, 3><<<n, b, 0, st>>>(F, g, (R)h, twice, zeroJ);
}

static FoldGrid fold_grid(const Grid &g)
{
    FoldGrid fg{};
    long long e[3] = {1, 1, 1};
    for (int d = 0; d < g.dim; d++) {
        const bool per = g.bc[d] == PERIODIC;
        fg.shell[d] = 2 * g.G[d];
        e[d] = per ? g.n[d] : g.n[d] + 2 * g.G[d];
        fg.rest[d] = (int)(e[d] - fg.shell[d]);
    }
    for (int d = 0; d < g.dim; d++) {
        long long m = fg.shell[d];
        for (int a = 0; a < g.dim; a++) m *= a < d ? fg.rest[a] : (a > d ? e[a] : 1);
        fg.first[d + 1] = fg.first[d] + (unsigned)m;  // (a grid has less than 2^31 cells)
    }
    return fg;
}

static FoldSet fold_j(const Grid &g) { return FoldSet{3, g.vol, {1, 2, 4}}; }

template <typename R>
void launch_update_B(R *F, const Grid &g, double h, const Laser &L, bool fold, cudaStream_t st)
{
    FoldBlocks fb{};
    if (fold) {
        fb.fs = fold_j(g);
        fb.fg = fold_grid(g);
        fb.nb = (unsigned)div_up(fb.fg.first[g.dim], 256ll * g.ext[2]);
    }
    dim3 b, n;
    note_launch();
    if constexpr (sizeof(R) == 4) {
        if (vec4_ok(g)) {
            grid_dims(g, g.ext[0] / 4, g.ext[1], g.ext[2], b, n);
            n.x += fb.nb;
            if (g.dim == 1) k_update_B4<1><<<n, b, 0, st>>>(F, g, (float)h, L, fb);
            else if (g.dim == 2) k_update_B4<2><<<n, b, 0, st>>>(F, g, (float)h, L, fb);
            else k_update_B4<3><<<n, b, 0, st>>>(F, g, (float)h, L, fb);
            return;
        }
    }
    grid_dims(g, g.ext[0], g.ext[1], g.ext[2], b, n);
    n.x += fb.nb;
    if (g.dim == 1) k_update_B<R, 1><<<n, b, 0, st>>>(F, g, (R)h, L, fb);
    else if (g.dim == 2) k_update_B<R, 2><<<n, b, 0, st>>>(F, g, (R)h, L, fb);
    else k_update_B<R, 3><<<n, b, 0, st>>>(F, g, (R)h, L, fb);
}

// FP32 up to 2048 cells, FP64 up to 512: a step's field launches take (in one
// block / in three launches, us) 6.3 / 12.5 on 256 cells, 10.5 / 12.5 on 2048,
// 14.5 / 12.5 on 4096; in FP64 one SM's rate binds sooner, 8.4 / 12.5 on 256
// cells, 12.1 / 12.5 on 512 (24.1 / 28.9 with a laser), 18.7 / 12.5 on 1024
template <typename R>
bool fields_in_one_block(const Grid &g) { return g.dim == 1 && g.n[0] <= (sizeof(R) == 4 ? 2048 : 512); }
template bool fields_in_one_block<float>(const Grid &);
template bool fields_in_one_block<double>(const Grid &);

template <typename R>
void launch_fields_1d(R *F, const Grid &g, double h, bool begin, bool last, const Laser &L1, const Laser &L2,
                      cudaStream_t st)
{
    Fields1d w{};
    w.fold = w.b1 = begin ? 0 : 1;
    w.twice = begin || last ? 0 : 1;
    w.zeroJ = w.b2 = begin || !last ? 1 : 0;
    note_launch();
    k_fields_1d<R><<<1, g.ext[0] <= 256 ? 256 : 1024, 0, st>>>(F, g, (R)h, w, fold_j(g), fold_grid(g), L1, L2);
}
template void launch_fields_1d<float>(float *, const Grid &, double, bool, bool, const Laser &, const Laser &, cudaStream_t);
template void launch_fields_1d<double>(double *, const Grid &, double, bool, bool, const Laser &, const Laser &, cudaStream_t);

void launch_fold_rho(double *rho, const Grid &g, cudaStream_t st)
{
    const FoldSet fs{1, g.vol, {0}};
    const FoldGrid fg = fold_grid(g);
    const int nb = div_up(fg.first[g.dim], 256);
    note_launch();
    if (g.dim == 1) k_fold<1><<<nb, 256, 0, st>>>(rho, fs, g, fg);
    else if (g.dim == 2) k_fold<2><<<nb, 256, 0, st>>>(rho, fs, g, fg);
    else k_fold<3><<<nb, 256, 0, st>>>(rho, fs, g, fg);
}

template void launch_update_E<float>(float *, const Grid &, double, bool, bool, cudaStream_t);
template void launch_update_E<double>(double *, const Grid &, double, bool, bool, cudaStream_t);
template void launch_update_B<float>(float *, const Grid &, double, const Laser &, bool, cudaStream_t);
template void launch_update_B<double>(double *, const Grid &, double, const Laser &, bool, cudaStream_t);

}  // namespace pic
