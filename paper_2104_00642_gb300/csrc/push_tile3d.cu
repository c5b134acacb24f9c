// push_tile3d.cu -- tiled particle push for 3D grids (FP32 cell+offset form,
// shape order 2, without QED): the two phases of push_tile2d.cu with a 3D box.
#include <algorithm>
#include <cstring>

#include "push_tile_dev.cuh"
#include "tma.cuh"

namespace pic {

// this file's own boxes, gathers and deposits (those of the other tiled pushes
// have the same names)
namespace {

// Tiles of T^3 cells.  The box holds x in [t0-4, t0+T+4) (float4-aligned
// rows) and y, z in [t0-3, t0+T+4): a particle within two cells below or one
// above its tile's faces after the half drift finds all its nodes there.  In
// x the box of an edge tile stays inside the padded rows; rows and planes of
// a ragged grid's last tiles may lie past them (staged as zero, never
// deposited on: a cell below n reaches node n+2, the padding node n+3).
template <int T>
struct Box3p {
    static constexpr int WX = T + 8, WY = T + 7, WZ = T + 7;
    static constexpr int RS = WX, PS = WX * WY, N = WX * WY * WZ;
    // fields (6), current (3), deposit records (7 words per particle)
    static constexpr int SMEM = (9 * N + 7 * kChunk3Max) * (int)sizeof(float);
};

// element k of a small register array without dynamic indexing (selects)
template <int W>
__device__ __forceinline__ float sel(const float *v, int k)
{
    float r = v[0];
#pragma unroll
    for (int i = 1; i < W; i++) r = k == i ? v[i] : r;
    return r;
}

// Eq. (19) in 3D on the shared box
template <int T>
__device__ __forceinline__ void gather3d_box(const float *__restrict__ P, const int *o0, const int *icn,
                                             const float (*wn)[3], const int *ich, const float (*wh)[3], float *eb)
{
    using B = Box3p<T>;
#pragma unroll
    for (int c = 0; c < 6; c++) {
        const int sx = stag(c, 0), sy = stag(c, 1), sz = stag(c, 2);
        const int ix = (sx ? ich[0] : icn[0]) - 1 - o0[0];
        const int iy = (sy ? ich[1] : icn[1]) - 1 - o0[1];
        const int iz = (sz ? ich[2] : icn[2]) - 1 - o0[2];
        const float *wx = sx ? wh[0] : wn[0];
        const float *wy = sy ? wh[1] : wn[1];
        const float *wz = sz ? wh[2] : wn[2];
        const float *q = P + c * B::N + iz * B::PS + iy * B::RS + ix;
        float acc = 0.f;
#pragma unroll
        for (int cz = 0; cz < 3; cz++) {
            float sb = 0.f;
#pragma unroll
            for (int b = 0; b < 3; b++) {
                const float *r = q + cz * B::PS + b * B::RS;
                float s = wx[0] * r[0];
                s += wx[1] * r[1];
                s += wx[2] * r[2];
                sb += wy[b] * s;
            }
            acc += wz[cz] * sb;
        }
        eb[c] = acc;
    }
}

// Esirkepov in 3D on a window of W nodes a side (Eqs. (20)-(22)): W_x = dSx
// (ty tz + dSy dSz / 12) with t = S0 + dS/2 (= S0y S0z + (dSy S0z + S0y
// dSz)/2 + dSy dSz/3), cyclic for y and z; J_d is cJ_d times the prefix sum of
// W_d along d (W - 1 nonzero nodes).  Shared int32 fixed point; the
// coefficients carry the units.
template <int T, int W>
__device__ __forceinline__ void esirkepov3d_box(int *base, const float (*S0)[W], const float (*dS)[W], const float *cj)
{
    using B = Box3p<T>;
    float t[3][W], p[3][W - 1];
#pragma unroll
    for (int d = 0; d < 3; d++) {
#pragma unroll
        for (int k = 0; k < W; k++) t[d][k] = S0[d][k] + 0.5f * dS[d][k];
        p[d][0] = dS[d][0];
#pragma unroll
        for (int k = 1; k < W - 1; k++) p[d][k] = p[d][k - 1] + dS[d][k];
    }
    const float r12 = 1.0f / 12.0f;
    // the outermost loop of each component stays rolled (code size: an
    // unrolled body stalls on instruction fetch); its index picks the z (or
    // y) shape by selects
#pragma unroll 1
    for (int c = 0; c < W; c++) {
        const float tzc = sel<W>(t[2], c), dzc = sel<W>(dS[2], c) * r12;
        int *bc = base + c * B::PS;
#pragma unroll
        for (int b = 0; b < W; b++) {
            const float wx = fmaf(t[1][b], tzc, dS[1][b] * dzc) * cj[0];
#pragma unroll
            for (int a = 0; a < W - 1; a++) atomicAdd(bc + b * B::RS + a, __float2int_rn(p[0][a] * wx));
        }
#pragma unroll
        for (int a = 0; a < W; a++) {
            const float wy = fmaf(t[0][a], tzc, dS[0][a] * dzc) * cj[1];
#pragma unroll
            for (int b = 0; b < W - 1; b++) atomicAdd(bc + B::N + b * B::RS + a, __float2int_rn(p[1][b] * wy));
        }
    }
#pragma unroll 1
    for (int b = 0; b < W; b++) {
        const float tyb = sel<W>(t[1], b), dyb = sel<W>(dS[1], b) * r12;
        int *bb = base + 2 * B::N + b * B::RS;
#pragma unroll
        for (int a = 0; a < W; a++) {
            const float wz = fmaf(t[0][a], tyb, dS[0][a] * dyb) * cj[2];
#pragma unroll
            for (int c = 0; c < W - 1; c++) atomicAdd(bb + c * B::PS + a, __float2int_rn(p[2][c] * wz));
        }
    }
}

// one row of the deposits (as deposit_row2d of push_tile2d.cu)
template <int T, bool EXACT, bool CROSS>
__device__ __forceinline__ void deposit_row3d(const float *sR, int *sJ, int j, int S, int n, const float *cj)
{
    constexpr int W = CROSS ? 4 : 3;
    const int r = (int)(threadIdx.x & 31u) * S + j;
    if (r >= n) return;
    const int slot = CROSS ? kChunk3Max - 1 - r : r;
    const uint32_t pk = __float_as_uint(sR[6 * kChunk3Max + slot]);
    float S0[3][W], dS[3][W];
#pragma unroll
    for (int d = 0; d < 3; d++) {
        float w0[3], w1[3];
        int i;
        axis_wn_f32(0, sR[d * kChunk3Max + slot], i, w0);
        axis_wn_f32(0, sR[(3 + d) * kChunk3Max + slot], i, w1);
        const bool o0 = CROSS && ((pk >> (16 + 2 * d)) & 1u), o1 = CROSS && ((pk >> (17 + 2 * d)) & 1u);
#pragma unroll
        for (int k = 0; k < W; k++) {
            const float s0 = o0 ? (k >= 1 ? w0[k - 1] : 0.f) : (k < 3 ? w0[k < 3 ? k : 0] : 0.f);
            const float s1 = o1 ? (k >= 1 ? w1[k - 1] : 0.f) : (k < 3 ? w1[k < 3 ? k : 0] : 0.f);
            S0[d][k] = s0;
            dS[d][k] = weight_step<EXACT>(s1, s0);
        }
    }
    esirkepov3d_box<T, W>(sJ + (pk & 0xffffu), S0, dS, cj);
}

}  // namespace

// One item in the two phases of k_push_tile2d (push_tile2d.cu): push with
// consecutive lanes on consecutive particles, then the lane-strided deposit of
// the records, those whose nearest node did not move on 3^3 windows (54
// atomics), the others on 4^3 (144); units of the current box from the item's
// particles.
//
// Bound: the shared-memory pipe (76 %; 162 field loads and 54 to 144 atomics a
// particle, about two wavefronts each) and issue (60 %).  256^3-style thermal
// plasma, 16,777,216 particles at 200 keV: 2.63 ms a push in one pass over
// consecutive lanes (eight lanes on one cell) and its deferred list, now 1.72
// ms; 856,440 particles on a 61 x 45 x 39 grid: 757 us one thread per
// particle, now 130 us.  The box's row above the tile is two cells deep: 7 %
// fewer cells (six rows and planes around the tile) deferred enough particles
// to cost 1.96 ms.
//
// A particle whose stencil leaves its tile's box (it drifted since the sort)
// is not pushed here: its index goes to a list, and the list is pushed
// afterwards on the global path (launch_push_list_f32).  Nothing of the
// particle is written before that decision, and a warp never waits on one
// lane's slow path.
template <int T, bool EXACT>
__global__ void __launch_bounds__(kPushThreads, 3)
    k_push_tile3d(PartF32 P, const TileItem *__restrict__ items, const uint32_t *__restrict__ nitems,
                  float *__restrict__ F, Grid g, PushConst pc, int *err, double *e_abs, uint32_t *defer,
                  uint32_t *ndefer, const __grid_constant__ CUtensorMap tmap, int use_tma)
{
    using B = Box3p<T>;
    extern __shared__ __align__(16) float smem_raw[];
    __shared__ uint64_t mbar;
    __shared__ int sCnt[3];                    // records filed from the front (node unmoved) and the back; rows taken
    __shared__ int2 sSum[3][kPushThreads / 32];  // sums of v_d per warp
    // the TMA destination starts on a 128-byte boundary
    // (offset from the shared array itself, so that the compiler keeps every
    // access below in the shared address space)
    float *smem = smem_raw + ((128u - ((uint32_t)__cvta_generic_to_shared(smem_raw) & 127u)) & 127u) / 4u;
    float *sF = smem;                                    // 6 components
    int *sJ = reinterpret_cast<int *>(smem + 6 * B::N);  // 3 components, fixed point
    float *sR = smem + 9 * B::N;                         // records: oh (3), oe (3), window
    const int nit = (int)*nitems;
    if ((int)blockIdx.x >= nit) return;
    const long long V = g.vol;
    const float hdx[3] = {pc.hdx_f[0], pc.hdx_f[1], pc.hdx_f[2]};
    const float k = pc.qmdt2_f;
    float *Fg = F + g.origin;
    const int rs = (int)g.sy, ps = (int)g.sz;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    auto corner = [&](int tile, int *o) {
        o[0] = tile % g.ntile[0] * T - 4;
        o[1] = tile / g.ntile[0] % g.ntile[1] * T - 3;
        o[2] = tile / (g.ntile[0] * g.ntile[1]) * T - 3;
    };
    auto stage_box = [&](int tile) {  // one thread; padded x coordinate a multiple of 4 floats, as TMA requires
        int o[3];
        corner(tile, o);
        fence_proxy_async_smem();
        mbar_arrive_expect_tx(&mbar, 6 * B::N * (int)sizeof(float));
        tma_load_4d(sF, &tmap, o[0] + g.G[0], o[1] + g.G[1], o[2] + g.G[2], 0, &mbar);
    };
    if (threadIdx.x == 0) {
        sCnt[0] = sCnt[1] = sCnt[2] = 0;
        if (use_tma) {
            mbar_init(&mbar, 1);
            stage_box(items[blockIdx.x].tile);
        }
    }
    for (int e4 = threadIdx.x; e4 < 3 * B::N / 4; e4 += kPushThreads)
        reinterpret_cast<int4 *>(sJ)[e4] = make_int4(0, 0, 0, 0);
    __syncthreads();
    uint32_t phase = 0;
    for (int it = blockIdx.x; it < nit; it += gridDim.x) {
        const TileItem m = items[it];
        int o0[3];
        corner(m.tile, o0);
        // the first pass's particle state, ahead of the wait for the field box
        uint32_t p = (uint32_t)m.start + threadIdx.x;  // capacities are below 2^31
        const uint32_t pend = (uint32_t)(m.start + m.count);
        uint32_t ncell = kDead;
        float nst[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        auto fetch = [&](uint32_t pn) {
            ncell = kDead;
            if (pn < pend) {
                ncell = P.cell[pn];
#pragma unroll
                for (int d = 0; d < 3; d++) {
                    nst[d] = P.off[d][pn];
                    nst[3 + d] = P.u[d][pn];
                }
            }
        };
        fetch(p);
        bool landed = true;
        if (use_tma) {
            landed = mbar_wait(&mbar, phase, 1 << 22);  // bounded: a copy that never lands is reported
            phase ^= 1u;
        } else {
            for (int e = threadIdx.x; e < 6 * B::N; e += kPushThreads) {
                const int c = e / B::N, r = e - c * B::N;
                const int z = r / B::PS, y = (r - z * B::PS) / B::RS, x = r - z * B::PS - y * B::RS;
                const int gx = o0[0] + x, gy = o0[1] + y, gz = o0[2] + z;
                float v = 0.f;
                if (gx < g.n[0] + g.G[0] && gy < g.n[1] + g.G[1] && gz < g.n[2] + g.G[2])
                    v = __ldg(Fg + c * V + (long long)gz * ps + (long long)gy * rs + gx);
                sF[e] = v;
            }
        }
        if (__syncthreads_or(!landed)) {
            if (threadIdx.x == 0) atomicOr(err, ERR_TIMEOUT);
            return;
        }
        // push phase (a warp without particles skips its passes)
        float vsum[3] = {0.f, 0.f, 0.f}, vabs[3] = {0.f, 0.f, 0.f};
        for (uint32_t pbase = m.start + 32 * warp; pbase < pend; pbase += kPushThreads, p += kPushThreads) {
            const uint32_t cp = ncell;
            float o[3] = {nst[0], nst[1], nst[2]};
            float ux = nst[3], uy = nst[4], uz = nst[5];
            fetch(p + kPushThreads);
            bool act = cp != kDead;
            int c[3] = {0, 0, 0}, c1[3] = {0, 0, 0}, u0[3] = {0, 0, 0};
            float oh[3] = {0.f, 0.f, 0.f}, o1[3] = {0.f, 0.f, 0.f};
            int icn[3] = {0, 0, 0}, i1[3] = {0, 0, 0};
            float ig1 = 0.f;
            bool din = false, cross = false;
            if (act) {
                unpack_cell(g, cp, c[0], c[1], c[2]);
                const float ig = inv_gamma_tile<EXACT>(ux, uy, uz);
                const float u[3] = {ux, uy, uz};
                int ich[3];
                float wn[3][3], wh[3][3];
                bool gin = true;
#pragma unroll
                for (int d = 0; d < 3; d++) {
                    drift_sel_f32(c[d], o[d], hdx[d], u[d], ig);
                    oh[d] = o[d];
                    axis_w_f32(c[d], o[d], icn[d], wn[d], ich[d], wh[d]);
                    gin &= c[d] - 1 >= o0[d] && c[d] + 2 < o0[d] + (d == 0 ? B::WX : B::WY);
                }
                if (gin) {
                    float eb[6];
                    gather3d_box<T>(sF, o0, icn, wn, ich, wh, eb);
                    if (pc.pusher) vay<float>(ux, uy, uz, k * eb[0], k * eb[1], k * eb[2], k * eb[3], k * eb[4], k * eb[5]);
                    else boris_tile<EXACT>(ux, uy, uz, k * eb[0], k * eb[1], k * eb[2], k * eb[3], k * eb[4], k * eb[5]);
                    ig1 = inv_gamma_tile<EXACT>(ux, uy, uz);
                    const float un[3] = {ux, uy, uz};
                    // Esirkepov on x^{n+1/2} -> x^{n+3/2}: the window of both end points
                    bool ok = true;
                    din = true;
#pragma unroll
                    for (int d = 0; d < 3; d++) {
                        drift_sel_f32(c[d], o[d], hdx[d], un[d], ig1);
                        c1[d] = c[d];
                        o1[d] = o[d];
                        drift_sel_f32(c[d], o[d], hdx[d], un[d], ig1);
                        i1[d] = c[d] + (o[d] >= 0.5f ? 1 : 0);
                        ok &= (i1[d] - icn[d] >= -1 && i1[d] - icn[d] <= 1);
                        cross |= i1[d] != icn[d];
                        u0[d] = min(icn[d], i1[d]) - 1;
                        din &= u0[d] >= o0[d] && u0[d] + 3 < o0[d] + (d == 0 ? B::WX : B::WY);
                    }
                    // a non-finite momentum (a NaN or infinite field) is reported and the particle
                    // removed before anything uses its position: NaN positions would give no valid
                    // cell or node index to the gather, the deposit or the diagnostics (and would
                    // otherwise be reported as a Courant violation)
                    if (!isfinite(ux + uy + uz)) {
                        atomicOr(err, ERR_NONFINITE);
                        P.cell[p] = kDead;
                        act = din = false;
                    } else if (!ok) {
                        atomicOr(err, ERR_CFL);
                        act = din = false;  // keeps its stored state
                    }
                }
                if (act && !din) defer[atomicAdd(ndefer, 1u)] = p;  // pushed by the list from its unchanged state
            }
            // file the deposit record: from the front, or (node moved) from the back
            const unsigned mk = __ballot_sync(0xffffffffu, din && !cross), mc = __ballot_sync(0xffffffffu, din && cross);
            int at = 0;
            if (lane == 0 && mk) at = atomicAdd(&sCnt[0], __popc(mk));
            if (lane == 1 && mc) at = atomicAdd(&sCnt[1], __popc(mc));
            const int a0 = __shfl_sync(0xffffffffu, at, 0), a1 = __shfl_sync(0xffffffffu, at, 1);
            if (!din) continue;
            const unsigned lt = (1u << lane) - 1u;
            const int slot = cross ? kChunk3Max - 1 - a1 - __popc(mc & lt) : a0 + __popc(mk & lt);
            uint32_t pk = (uint32_t)((u0[2] - o0[2]) * B::PS + (u0[1] - o0[1]) * B::RS + (u0[0] - o0[0]));
#pragma unroll
            for (int d = 0; d < 3; d++) {
                sR[d * kChunk3Max + slot] = oh[d];
                sR[(3 + d) * kChunk3Max + slot] = o[d];
                pk |= (uint32_t)(icn[d] - 1 - u0[d]) << (16 + 2 * d) | (uint32_t)(i1[d] - 1 - u0[d]) << (17 + 2 * d);
            }
            sR[6 * kChunk3Max + slot] = __uint_as_float(pk);
            const float v[3] = {ux * ig1, uy * ig1, uz * ig1};
#pragma unroll
            for (int d = 0; d < 3; d++) {
                if (EXACT) vsum[d] += v[d];
                vabs[d] += fabsf(v[d]);
            }
            // boundaries
            int cc[3] = {c1[0], c1[1], c1[2]};
            bool dead = false;
#pragma unroll
            for (int d = 0; d < 3; d++) {
                const bool lo = cc[d] < 0, hi = cc[d] >= g.n[d], per = g.bc[d] == PERIODIC;
                dead |= !per && (lo || hi);
                cc[d] += per ? (lo ? g.n[d] : (hi ? -g.n[d] : 0)) : 0;
            }
            if (dead) {
                P.cell[p] = kDead;
                double uu = (double)ux * ux + (double)uy * uy + (double)uz * uz;
                atomicAdd(e_abs, pc.wmdV * uu / (sqrt(1.0 + uu) + 1.0));
            } else {
                P.cell[p] = pack_cell(g, cc[0], cc[1], cc[2]);
            }
#pragma unroll
            for (int d = 0; d < 3; d++) P.off[d][p] = o1[d];
            P.u[0][p] = ux;
            P.u[1][p] = uy;
            P.u[2][p] = uz;
        }
        warp_sums<EXACT, kPushThreads / 32>(vabs, vsum, sSum);
        __syncthreads();
        // the next item's field box, while this one's records are deposited
        if (use_tma && threadIdx.x == 0 && it + (int)gridDim.x < nit) stage_box(items[it + gridDim.x].tile);
        // deposit phase
        // (a node's share of a particle's |q w v_d|: at most the square of the
        // largest weight, 3/4)
        const int nk = sCnt[0], nc = sCnt[1];
        float sc[3], cj[3];
#pragma unroll
        for (int d = 0; d < 3; d++) {
            sc[d] = box_units(sSum[d], pc.qw_f, nk + nc, pc.cJ_f[d], 0.5625f);
            cj[d] = pc.cJ_f[d] * sc[d];
        }
        const int Sk = deposit_rows(nk), Sc = deposit_rows(nc);
        for (int j = next_row(&sCnt[2]); j < Sc + Sk; j = next_row(&sCnt[2])) {
            if (j < Sc) deposit_row3d<T, EXACT, true>(sR, sJ, j, Sc, nc, cj);
            else deposit_row3d<T, EXACT, false>(sR, sJ, j - Sc, Sk, nk, cj);
        }
        __syncthreads();
        if (threadIdx.x == 0) sCnt[0] = sCnt[1] = sCnt[2] = 0;
        // flush the current box, four values at a time, and leave it zero (rows
        // past a ragged grid's padding hold zeros only)
        const float unit[3] = {1.0f / sc[0], 1.0f / sc[1], 1.0f / sc[2]};
        for (int e4 = threadIdx.x; e4 < 3 * B::N / 4; e4 += kPushThreads) {
            const int4 iv = reinterpret_cast<const int4 *>(sJ)[e4];
            if ((iv.x | iv.y | iv.z | iv.w) == 0) continue;
            reinterpret_cast<int4 *>(sJ)[e4] = make_int4(0, 0, 0, 0);
            const int e = 4 * e4;
            const int c = e / B::N, r = e - c * B::N;
            const int z = r / B::PS, y = (r - z * B::PS) / B::RS, x = r - z * B::PS - y * B::RS;
            const float junit = c == 0 ? unit[0] : (c == 1 ? unit[1] : unit[2]);
            float *dst = Fg + (JX + c) * V + (long long)(o0[2] + z) * ps + (long long)(o0[1] + y) * rs + o0[0] + x;
            atomicAdd(reinterpret_cast<float4 *>(dst), make_float4(iv.x * junit, iv.y * junit, iv.z * junit, iv.w * junit));
        }
        // (the next item's first barrier orders the flush before its records)
    }
}

template <bool EXACT>
static void launch_exact(const PartF32 &P, const TileItem *items, const uint32_t *nitems, long long max_items, float *F,
                         const Grid &g, const PushConst &pc, int *err, double *e_abs, uint32_t *defer, uint32_t *ndefer,
                         bool maybe_sparse, cudaStream_t st)
{
    constexpr int T = 4;
    constexpr int smem = Box3p<T>::SMEM + 128;  // + alignment of the TMA destination
    static int nsm = 0, per_sm = 0;
    if (!per_sm) {
        cudaFuncSetAttribute(k_push_tile3d<T, EXACT>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_push_tile3d<T, EXACT>, kPushThreads, smem);
        if (per_sm < 1) per_sm = 1;
    }
    // the six field components as one 4D tensor (x, y, z, component)
    CUtensorMap tmap;
    const int box[4] = {Box3p<T>::WX, Box3p<T>::WY, Box3p<T>::WZ, 6};
    const bool tma = tma_encode_field_map3(&tmap, F, g.ext, g.sy, g.sz, g.vol, 6, box);
    if (!tma) memset(&tmap, 0, sizeof tmap);
    long long grid = std::min<long long>(max_items, (long long)nsm * per_sm);  // one resident wave
    if (grid < 1) grid = 1;
    cudaMemsetAsync(ndefer, 0, sizeof(uint32_t), st);
    note_launch();
    k_push_tile3d<T, EXACT><<<(int)grid, kPushThreads, smem, st>>>(P, items, nitems, F, g, pc, err, e_abs, defer, ndefer,
                                                                   tmap, tma ? 1 : 0);
    launch_push_list_f32(P, defer, ndefer, P.n, F, g, pc, err, e_abs, maybe_sparse ? nitems : nullptr, st);
}

void launch_push_tile3d(const PartF32 &P, const TileItem *items, const uint32_t *nitems, long long max_items,
                        float *F, const Grid &g, const PushConst &pc, int *err, double *e_abs, uint32_t *defer,
                        uint32_t *ndefer, bool maybe_sparse, cudaStream_t st)
{
    if (P.n == 0) return;
    // Sizes that are not multiples of 4 were the one-thread push's: these take its
    // root and quotients and the finer units, so that nothing of them is less
    // precise than there (61 x 45 x 39 cells, 8 steps: E 4.1e-7 off 64 bits with
    // the fast ones, 3.3e-7 now, 3.8e-7 one thread per particle; the case takes
    // 1.56 ms instead of 1.54).
    const bool whole = g.n[0] % 4 == 0 && g.n[1] % 4 == 0 && g.n[2] % 4 == 0;
    if (whole) launch_exact<false>(P, items, nitems, max_items, F, g, pc, err, e_abs, defer, ndefer, maybe_sparse, st);
    else launch_exact<true>(P, items, nitems, max_items, F, g, pc, err, e_abs, defer, ndefer, maybe_sparse, st);
}

bool tile3d_push_supported(const Grid &g)
{
    for (int d = 0; d < 3; d++)
        if (g.tile_log2[d] != 2 || g.G[d] != 4) return false;
    return g.dim == 3;
}

}  // namespace pic
