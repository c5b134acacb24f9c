// push_tile2d.cu -- tiled particle push for 2D grids (FP32 cell+offset form),
// shape orders 2 and 4, without the QED Monte Carlo (push_tile.cu has the QED
// species' pushes).
//
// Particles are counting-sorted by tile (T x T cells) every K steps.  Each
// work item is a chunk of at most kChunkMax particles that sat in one tile at
// the last sort.  A persistent CTA takes items in turn and, per item:
//   1. stages the six field components of the tile box [t0-4, t0+T+8) x
//      [t0-4, t0+T+5) into shared memory (rows are contiguous in HBM);
//   2. pushes every particle of the chunk (half drift, gather from shared
//      memory, Boris, two half drifts) and leaves a deposit record each;
//   3. deposits the records (Esirkepov) into a shared current box of the same
//      shape with shared-memory atomics;
//   4. flushes the current box to HBM with vector atomics (float4), once.
// A particle that drifted so far since the sort that its stencil leaves the
// box is handled on the global path (gather from HBM, global atomics), so the
// result does not depend on the sort interval.
#include <algorithm>
#include <cstring>

#include "push_tile_dev.cuh"
#include "tma.cuh"

namespace pic {

// this file's own boxes, gathers and deposits (those of the other tiled pushes
// have the same names)
namespace {

template <int T>
struct Box2p {
    static constexpr int WX = T + 12;  // x: [t0-4, t0+T+8), a multiple of 4 floats
    static constexpr int WY = T + 9;   // y: [t0-4, t0+T+5)
    static constexpr int N = WX * WY;  // one field component
    // the current box has rows of its own pitch: neighbouring rows of cells
    // then start T banks apart, so lanes on 32 cells of a tile add to 32 banks
    static constexpr int RJ = T == 16 ? 48 : 24;
    static constexpr int NJ = RJ * WY;
    // fields (6), current (3), deposit records (6 words per particle)
    static constexpr int SMEM = (6 * N + 3 * NJ + 6 * kChunkMax) * (int)sizeof(float);
};

// Eq. (19) in 2D on a strided view: F_c(x, y) = P[c*cs + (y-oy)*rs + (x-ox)]
template <int ORDER = 2>
__device__ __forceinline__ void gather2d(const float *__restrict__ P, long long cs, int rs, int ox, int oy,
                                         const int *icn, const float (*wn)[ORDER + 1], const int *ich,
                                         const float (*wh)[ORDER + 1], float *eb)
{
    constexpr int PN = ORDER + 1, H = ORDER / 2;
#pragma unroll
    for (int c = 0; c < 6; c++) {
        const int sx = stag(c, 0), sy = stag(c, 1);
        const int ix = (sx ? ich[0] : icn[0]) - H - ox;
        const int iy = (sy ? ich[1] : icn[1]) - H - oy;
        const float *wx = sx ? wh[0] : wn[0];
        const float *wy = sy ? wh[1] : wn[1];
        const float *row = P + c * cs + (long long)iy * rs + ix;
        float acc = 0.f;
#pragma unroll
        for (int b = 0; b < PN; b++) {
            const float *r = row + (long long)b * rs;
            float s = wx[0] * r[0];
#pragma unroll
            for (int a = 1; a < PN; a++) s += wx[a] * r[a];
            acc += wy[b] * s;
        }
        eb[c] = acc;
    }
}

// Esirkepov in 2D on a window of W nodes a side (Eqs. (20)-(22)): W_x = dSx
// (S0y + dSy/2), W_y = dSy (S0x + dSx/2), and J_z = q w v_z times the time
// average of the node-shape product, S0xS0y + (dSx S0y + S0x dSy)/2 +
// dSx dSy/3, written as tx ty + dSx dSy/12 with tx = S0x + dSx/2, ty = S0y +
// dSy/2.  `Acc` adds one value at window offset (a, b) of component c.
template <int W, class Acc>
__device__ __forceinline__ void esirkepov2d(const float (*S0)[W], const float (*dS)[W], float cjx, float cjy,
                                            float jvz, Acc &acc)
{
    float tx[W], ty[W], dx12[W];
#pragma unroll
    for (int k = 0; k < W; k++) {
        tx[k] = S0[0][k] + 0.5f * dS[0][k];
        ty[k] = S0[1][k] + 0.5f * dS[1][k];
        dx12[k] = dS[0][k] * (1.0f / 12.0f);
    }
    float px[W - 1], py[W - 1];  // prefix sums of dS along x and y
    px[0] = dS[0][0];
    py[0] = dS[1][0];
#pragma unroll
    for (int k = 1; k < W - 1; k++) {
        px[k] = px[k - 1] + dS[0][k];
        py[k] = py[k - 1] + dS[1][k];
    }
#pragma unroll
    for (int b = 0; b < W; b++)
#pragma unroll
        for (int a = 0; a < W - 1; a++) acc.add(0, a, b, cjx * px[a] * ty[b]);
#pragma unroll
    for (int b = 0; b < W - 1; b++)
#pragma unroll
        for (int a = 0; a < W; a++) acc.add(1, a, b, cjy * py[b] * tx[a]);
#pragma unroll
    for (int b = 0; b < W; b++)
#pragma unroll
        for (int a = 0; a < W; a++) acc.add(2, a, b, jvz * (tx[a] * ty[b] + dx12[a] * dS[1][b]));
}

// current straight into HBM (particles whose window left the box)
struct AccGlobal {
    float *base;
    long long cs;
    int rs;
    __device__ __forceinline__ void add(int c, int a, int b, float v)
    {
        if (v != 0.f) atomicAdd(base + c * cs + (long long)b * rs + a, v);
    }
};

// warp-aggregated current into the shared box: the lanes of grp share the
// window origin; each value is summed over the group with one warp
// reduction and added by the group's first lane with one shared atomic
struct AccWarp {
    int *base;
    int cs, rs;
    unsigned grp;
    bool lead;
    __device__ __forceinline__ void add(int c, int a, int b, float v)
    {
        const int s = __reduce_add_sync(grp, __float2int_rn(v));
        if (lead && s) atomicAdd(base + c * cs + b * rs + a, s);
    }
};

// One row of the deposits: records lane S + j, S rows of 32.  CROSS: the
// nearest node moved along an axis (filed from the back; union window of
// ORDER + 2 nodes); else start and end share the window of ORDER + 1 nodes.
//
// Lane striding: the n records are cut into 32 contiguous segments of S and
// lane l of every row is on segment l.  Records of one cell lie together (the
// particles are cell-sorted), so the 32 lanes of one shared atomic are on 32
// different cells, whatever the order in the tile; S is odd, so the record
// reads are conflict-free too.
template <int T, int ORDER, bool AGG, bool CROSS>
__device__ __forceinline__ void deposit_row2d(const float *sR, int *sJ, int j, int S, int n, float sjx, float sjy,
                                              float sqw)
{
    using B = Box2p<T>;
    constexpr int W = ORDER + (CROSS ? 2 : 1), PN = ORDER + 1;
    const int lane = threadIdx.x & 31;
    const int r = AGG ? j * 32 + lane : lane * S + j;
    const bool valid = r < n;
    const int slot = CROSS ? kChunkMax - 1 - r : r;
    int key = -1;
    float jvz = 0.f;
    float S0[2][W], dS[2][W];
    if (valid) {
        const uint32_t pk = __float_as_uint(sR[5 * kChunkMax + slot]);
        key = (int)(pk & 0xffffu);
        jvz = sqw * sR[4 * kChunkMax + slot];
#pragma unroll
        for (int d = 0; d < 2; d++) {
            const float oh = sR[d * kChunkMax + slot], oe = sR[(2 + d) * kChunkMax + slot];
            float w0[PN], w1[PN];
            int i;
            axis_wn_f32<ORDER>(0, oh, i, w0);
            axis_wn_f32<ORDER>(0, oe, i, w1);
            if constexpr (CROSS) {
                const bool o0 = (pk >> (16 + 2 * d)) & 1u, o1 = (pk >> (17 + 2 * d)) & 1u;
#pragma unroll
                for (int k = 0; k < W; k++) {
                    const float s0 = o0 ? (k >= 1 ? w0[k - 1] : 0.f) : (k < PN ? w0[k] : 0.f);
                    const float s1 = o1 ? (k >= 1 ? w1[k - 1] : 0.f) : (k < PN ? w1[k] : 0.f);
                    S0[d][k] = s0;
                    dS[d][k] = weight_step<ORDER == 4>(s1, s0);
                }
            } else {
#pragma unroll
                for (int k = 0; k < W; k++) {
                    S0[d][k] = w0[k];
                    dS[d][k] = weight_step<ORDER == 4>(w1[k], w0[k]);
                }
            }
        }
    }
    if constexpr (AGG) {
        const unsigned smask = __ballot_sync(0xffffffffu, valid);
        if (valid) {
            const unsigned grp = __match_any_sync(smask, key);
            AccWarp acc{sJ + key, B::NJ, B::RJ, grp, lane == __ffs(grp) - 1};
            esirkepov2d<W>(S0, dS, sjx, sjy, jvz, acc);
        }
    } else if (valid) {
        AccSharedUnits acc{sJ + key, B::NJ, B::RJ};
        esirkepov2d<W>(S0, dS, sjx, sjy, jvz, acc);
    }
}

}  // namespace

// One item in two phases.
//   push:    consecutive lanes on consecutive particles -- state read and
//            written in place, coalesced; particles of one cell read the same
//            field nodes, a shared-memory broadcast -- leaving a 24-byte
//            record per particle: its offsets at the deposit's two end
//            points, v_z and its window;
//   deposit: the records, lane-strided, those whose nearest node did not move
//            (3 x 3 windows, 21 atomics at order 2) apart from those whose
//            node moved (4 x 4, 40 atomics).
// A single pass (gather, push and atomics per particle, lane-strided) was
// bound by the shared-memory pipe (85 %; 250 bank-conflict wavefronts per 32
// particles, lanes sharing cells); now issue is its first bound (60 % of the
// slots, 1170 instructions and 122 conflict wavefronts per 32 of the foil's heated
// electrons): its 2,097,152 electrons 101 -> 89 us, its protons 97 -> 82 us a push
// while the pulse comes up.  At order 4 (262,144 particles of 1 keV on a 128 x
// 128 grid) 201 us on the one-thread-per-particle kernel -> 39 us (2070
// instructions per 32 particles, 55 % of the issue slots).
//
// Order 4 was the one-thread push's: it keeps that kernel's root and quotients
// and takes the finer units (EXACT and SIGNED in push_tile_dev.cuh), so that
// nothing is less precise than there (1 keV, 128 x 128 cells, 16 steps: E
// 9.3e-7 off 64 bits with the fast ones, 5.4e-7 now, 6.1e-7 one thread per
// particle), for 4 % of that case's time.
//
// Fixed point: the units of the item's current box come from its particles,
// about 2^31 for the sum over them of the most that each can add to one node
// (|q w| times the largest values of the shapes times |v_d| and what the FP32
// offsets round a move by, see box_units), so no node can overflow, and
// wrapped intermediate sums are exact.
//
// The field box of an item is one TMA tile copy (tmap: the six field
// components as a 3D tensor, x fastest) issued by one thread: of the CTA's
// first item at entry, of each next item as soon as the push phase has read
// the present one's.
//
// AGG: the deposit phase walks consecutive records and sums the lanes that
// share a window before one atomic per value.
template <int T, int ORDER, bool AGG, int NT>
__global__ void __launch_bounds__(NT, 768 / NT)
    k_push_tile2d(PartF32 P, const TileItem *__restrict__ items, const uint32_t *__restrict__ nitems,
                  float *__restrict__ F, Grid g, PushConst pc, int *err, double *e_abs,
                  const __grid_constant__ CUtensorMap tmap, int use_tma)
{
    using B = Box2p<T>;
    constexpr int H = ORDER / 2, PN = ORDER + 1;
    extern __shared__ __align__(16) float smem_raw[];
    __shared__ uint64_t mbar;
    __shared__ int sCnt[3];                      // records filed from the front (node unmoved) and the back; rows taken
    __shared__ int2 sSum[3][NT / 32];  // sums of v_d per warp
    // the TMA destination starts on a 128-byte boundary
    // (offset from the shared array itself, so that the compiler keeps every
    // access below in the shared address space)
    float *smem = smem_raw + ((128u - ((uint32_t)__cvta_generic_to_shared(smem_raw) & 127u)) & 127u) / 4u;
    float *sF = smem;                                    // 6 components
    int *sJ = reinterpret_cast<int *>(smem + 6 * B::N);  // 3 components, fixed point
    float *sR = smem + 6 * B::N + 3 * B::NJ;             // records: oh_x, oh_y, oe_x, oe_y, v_z, window
    const int nit = (int)*nitems;
    if ((int)blockIdx.x >= nit) return;
    const long long V = g.vol;
    const float hdx0 = pc.hdx_f[0], hdx1 = pc.hdx_f[1];
    const float k = pc.qmdt2_f;
    const float cjx = pc.cJ_f[0], cjy = pc.cJ_f[1], qw = pc.qw_f;
    float *Fg = F + g.origin;  // interior origin
    const int rs = (int)g.sy;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    auto stage_box = [&](int tile) {  // one thread: the field box of a tile
        // padded coordinates of the box corner; x = tx*T is a multiple of 4
        // floats (16 bytes) as the copy engine requires
        fence_proxy_async_smem();
        mbar_arrive_expect_tx(&mbar, 6 * B::N * (int)sizeof(float));
        tma_load_3d(sF, &tmap, tile % g.ntile[0] * T - 4 + g.G[0], tile / g.ntile[0] * T - 4 + g.G[1], 0, &mbar);
    };
    if (threadIdx.x == 0) {
        sCnt[0] = sCnt[1] = sCnt[2] = 0;
        if (use_tma) {
            mbar_init(&mbar, 1);
            stage_box(items[blockIdx.x].tile);
        }
    }
    for (int e = threadIdx.x; e < 3 * B::NJ / 4; e += NT) reinterpret_cast<int4 *>(sJ)[e] = make_int4(0, 0, 0, 0);
    __syncthreads();
    uint32_t phase = 0;
    for (int it = blockIdx.x; it < nit; it += gridDim.x) {
        const TileItem m = items[it];
        const int tx = m.tile % g.ntile[0], ty = m.tile / g.ntile[0];
        const int bx0 = tx * T - 4, by0 = ty * T - 4;
        // the first pass's particle state, ahead of the wait for the field box
        uint32_t p = (uint32_t)m.start + threadIdx.x;  // capacities are below 2^31
        const uint32_t pend = (uint32_t)(m.start + m.count);
        uint32_t ncell = kDead;
        float nst[5] = {0.f, 0.f, 0.f, 0.f, 0.f};
        auto fetch = [&](uint32_t pn) {
            ncell = kDead;
            if (pn < pend) {
                ncell = P.cell[pn];
                nst[0] = P.off[0][pn];
                nst[1] = P.off[1][pn];
                nst[2] = P.u[0][pn];
                nst[3] = P.u[1][pn];
                nst[4] = P.u[2][pn];
            }
        };
        fetch(p);
        bool landed = true;
        if (use_tma) {
            // bounded wait: a copy that never lands sets an error flag and the
            // CTA stops, all its threads together (the host reports the flag)
            landed = mbar_wait(&mbar, phase, 1 << 22);
            phase ^= 1u;
        } else {
            for (int e = threadIdx.x; e < 6 * B::N; e += NT) {
                const int c = e / B::N, r = e - c * B::N;
                const int y = r / B::WX, x = r - y * B::WX;
                const int gx = bx0 + x, gy = by0 + y;
                float v = 0.f;
                if (gx < g.n[0] + g.G[0] && gy < g.n[1] + g.G[1]) v = __ldg(Fg + c * V + (long long)gy * rs + gx);
                sF[e] = v;
            }
        }
        if (__syncthreads_or(!landed)) {
            if (threadIdx.x == 0) atomicOr(err, ERR_TIMEOUT);
            return;
        }
        // push phase (the records are filed by the warp; a warp without
        // particles skips its passes)
        float vsum[3] = {0.f, 0.f, 0.f}, vabs[3] = {0.f, 0.f, 0.f};
        for (uint32_t pbase = m.start + 32 * warp; pbase < pend; pbase += NT, p += NT) {
            const uint32_t cp = ncell;
            float ux = nst[2], uy = nst[3], uz = nst[4];
            float o[2] = {nst[0], nst[1]};
            fetch(p + NT);
            bool act = cp != kDead;  // a live particle of this item
            int c[2] = {0, 0}, c1[2] = {0, 0}, u0[2] = {0, 0};
            float o1[2] = {0.f, 0.f}, oh[2] = {0.f, 0.f};
            float ig1 = 0.f;
            float eb[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
            int icn[2] = {0, 0}, i1[2] = {0, 0};  // nearest nodes at the deposit's end points
            bool ok = true;
            if (act) {
                int dummy;
                unpack_cell(g, cp, c[0], c[1], dummy);
                float ig = inv_gamma_tile<ORDER == 4>(ux, uy, uz);
                drift_sel_f32(c[0], o[0], hdx0, ux, ig);
                drift_sel_f32(c[1], o[1], hdx1, uy, ig);
                oh[0] = o[0];
                oh[1] = o[1];
                int ich[2];
                float wn[2][PN], wh[2][PN];
                axis_w_f32<ORDER>(c[0], o[0], icn[0], wn[0], ich[0], wh[0]);
                axis_w_f32<ORDER>(c[1], o[1], icn[1], wn[1], ich[1], wh[1]);
                const bool gin =
                    c[0] - H >= bx0 && c[0] + H + 1 < bx0 + B::WX && c[1] - H >= by0 && c[1] + H + 1 < by0 + B::WY;
                if (gin) gather2d<ORDER>(sF, B::N, B::WX, bx0, by0, icn, wn, ich, wh, eb);
                else gather2d<ORDER>(Fg, V, rs, 0, 0, icn, wn, ich, wh, eb);
                if (pc.pusher) vay<float>(ux, uy, uz, k * eb[0], k * eb[1], k * eb[2], k * eb[3], k * eb[4], k * eb[5]);
                else boris_tile<ORDER == 4>(ux, uy, uz, k * eb[0], k * eb[1], k * eb[2], k * eb[3], k * eb[4], k * eb[5]);
                ig1 = inv_gamma_tile<ORDER == 4>(ux, uy, uz);
                drift_sel_f32(c[0], o[0], hdx0, ux, ig1);
                drift_sel_f32(c[1], o[1], hdx1, uy, ig1);
                c1[0] = c[0];
                c1[1] = c[1];
                o1[0] = o[0];
                o1[1] = o[1];
                drift_sel_f32(c[0], o[0], hdx0, ux, ig1);
                drift_sel_f32(c[1], o[1], hdx1, uy, ig1);
                // Esirkepov on x^{n+1/2} -> x^{n+3/2}: the window of both end points
#pragma unroll
                for (int d = 0; d < 2; d++) {
                    i1[d] = c[d] + (o[d] >= 0.5f ? 1 : 0);
                    ok &= (i1[d] - icn[d] >= -1 && i1[d] - icn[d] <= 1);
                    u0[d] = min(icn[d], i1[d]) - H;
                }
                // a non-finite momentum (a NaN or infinite field) is reported and the particle
                // removed before anything uses its position: NaN positions would give no valid
                // cell or node index to the gather, the deposit or the diagnostics (and would
                // otherwise be reported as a Courant violation)
                if (!isfinite(ux + uy + uz)) {
                    atomicOr(err, ERR_NONFINITE);
                    P.cell[p] = kDead;
                    act = false;
                } else if (!ok) {
                    atomicOr(err, ERR_CFL);
                    act = false;  // keeps its stored state
                }
            }
            const float vz = uz * ig1;
            const bool cross = i1[0] != icn[0] || i1[1] != icn[1];
            const bool din =
                act && u0[0] >= bx0 && u0[0] + PN < bx0 + B::WX && u0[1] >= by0 && u0[1] + PN < by0 + B::WY;
            if (act && !din) {
                float S0[2][PN + 1], dS[2][PN + 1];
#pragma unroll
                for (int d = 0; d < 2; d++) {
                    float w0[PN], w1[PN];
                    int i;
                    axis_wn_f32<ORDER>(0, oh[d], i, w0);
                    axis_wn_f32<ORDER>(0, o[d], i, w1);
                    const bool s0u = icn[d] - H > u0[d], s1u = i1[d] - H > u0[d];
#pragma unroll
                    for (int a = 0; a <= PN; a++) {
                        const float s0 = s0u ? (a >= 1 ? w0[a - 1] : 0.f) : (a < PN ? w0[a] : 0.f);
                        const float s1 = s1u ? (a >= 1 ? w1[a - 1] : 0.f) : (a < PN ? w1[a] : 0.f);
                        S0[d][a] = s0;
                        dS[d][a] = weight_step<ORDER == 4>(s1, s0);
                    }
                }
                AccGlobal acc{Fg + JX * V + (long long)u0[1] * rs + u0[0], V, rs};
                esirkepov2d<PN + 1>(S0, dS, cjx, cjy, qw * vz, acc);
            }
            // file the deposit record: from the front, or (node moved) from the back
            const unsigned mk = __ballot_sync(0xffffffffu, din && !cross), mc = __ballot_sync(0xffffffffu, din && cross);
            int at = 0;
            if (lane == 0 && mk) at = atomicAdd(&sCnt[0], __popc(mk));
            if (lane == 1 && mc) at = atomicAdd(&sCnt[1], __popc(mc));
            const int a0 = __shfl_sync(0xffffffffu, at, 0), a1 = __shfl_sync(0xffffffffu, at, 1);
            if (din) {
                const unsigned lt = (1u << lane) - 1u;
                const int slot = cross ? kChunkMax - 1 - a1 - __popc(mc & lt) : a0 + __popc(mk & lt);
                sR[slot] = oh[0];
                sR[kChunkMax + slot] = oh[1];
                sR[2 * kChunkMax + slot] = o[0];
                sR[3 * kChunkMax + slot] = o[1];
                sR[4 * kChunkMax + slot] = vz;
                uint32_t pk = (uint32_t)((u0[1] - by0) * B::RJ + (u0[0] - bx0));
#pragma unroll
                for (int d = 0; d < 2; d++)
                    pk |= (uint32_t)(icn[d] - H - u0[d]) << (16 + 2 * d) | (uint32_t)(i1[d] - H - u0[d]) << (17 + 2 * d);
                sR[5 * kChunkMax + slot] = __uint_as_float(pk);
                const float v[3] = {ux * ig1, uy * ig1, vz};
#pragma unroll
                for (int d = 0; d < 3; d++) {
                    if (ORDER == 4) vsum[d] += v[d];
                    vabs[d] += fabsf(v[d]);
                }
            }
            if (!act) continue;
            // boundaries
            int cc[2] = {c1[0], c1[1]};
            bool dead = false;
#pragma unroll
            for (int d = 0; d < 2; d++) {
                const bool lo = cc[d] < 0, hi = cc[d] >= g.n[d], per = g.bc[d] == PERIODIC;
                dead |= !per && (lo || hi);
                cc[d] += per ? (lo ? g.n[d] : (hi ? -g.n[d] : 0)) : 0;
            }
            if (dead) {
                P.cell[p] = kDead;
                double uu = (double)ux * ux + (double)uy * uy + (double)uz * uz;
                atomicAdd(e_abs, pc.wmdV * uu / (sqrt(1.0 + uu) + 1.0));
            } else {
                P.cell[p] = pack_cell(g, cc[0], cc[1], 0);
            }
            P.off[0][p] = o1[0];
            P.off[1][p] = o1[1];
            P.u[0][p] = ux;
            P.u[1][p] = uy;
            P.u[2][p] = uz;
        }
        warp_sums<ORDER == 4, NT / 32>(vabs, vsum, sSum);
        __syncthreads();
        // the next item's field box, while this one's records are deposited
        if (use_tma && threadIdx.x == 0 && it + (int)gridDim.x < nit) stage_box(items[it + gridDim.x].tile);
        // deposit phase
        // (the largest share of a particle's current on one node, per unit of
        // |q w v_d|: along x and y the prefix of the shape difference times the
        // other axis' shape, along z both shapes; then 1/2^31 of the sum)
        constexpr float kW = ORDER == 2 ? 0.75f : 115.0f / 192.0f, kP = ORDER == 2 ? 1.0f : 2.0f / 3.0f;
        const int nk = sCnt[0], nc = sCnt[1];
        const float scx = box_units(sSum[0], qw, nk + nc, cjx, kP * kW), scy = box_units(sSum[1], qw, nk + nc, cjy, kP * kW),
                    scz = box_units(sSum[2], qw, 0, 0.f, kW * kW);  // (v_z itself is in the record)
        const float sjx = cjx * scx, sjy = cjy * scy, sqw = qw * scz;
        const int Sk = deposit_rows(nk), Sc = deposit_rows(nc);
        for (int j = next_row(&sCnt[2]); j < Sc + Sk; j = next_row(&sCnt[2])) {
            if (j < Sc) deposit_row2d<T, ORDER, AGG, true>(sR, sJ, j, Sc, nc, sjx, sjy, sqw);
            else deposit_row2d<T, ORDER, AGG, false>(sR, sJ, j - Sc, Sk, nk, sjx, sjy, sqw);
        }
        __syncthreads();
        if (threadIdx.x == 0) sCnt[0] = sCnt[1] = sCnt[2] = 0;
        // flush the current box, four values at a time, and leave it zero
        const float unit[3] = {1.0f / scx, 1.0f / scy, 1.0f / scz};
        for (int v4 = threadIdx.x; v4 < 3 * B::WY * (B::WX / 4); v4 += NT) {
            const int row = v4 / (B::WX / 4), x = 4 * (v4 - row * (B::WX / 4));
            const int c = row / B::WY, y = row - c * B::WY;
            int4 *cellv = reinterpret_cast<int4 *>(sJ + c * B::NJ + y * B::RJ + x);
            const int4 iv = *cellv;
            if ((iv.x | iv.y | iv.z | iv.w) == 0) continue;
            *cellv = make_int4(0, 0, 0, 0);
            const float junit = c == 0 ? unit[0] : (c == 1 ? unit[1] : unit[2]);
            const float4 v = make_float4(iv.x * junit, iv.y * junit, iv.z * junit, iv.w * junit);
            const int gx = bx0 + x, gy = by0 + y;
            if (gx < -g.G[0] || gx + 3 >= g.n[0] + g.G[0] || gy < -g.G[1] || gy >= g.n[1] + g.G[1]) {
                // partial vector at the edge of the padded box (holds zeros only
                // for accepted particles; kept exact for safety)
                float vv[4] = {v.x, v.y, v.z, v.w};
                for (int l = 0; l < 4; l++)
                    if (vv[l] != 0.f && gx + l >= -g.G[0] && gx + l < g.n[0] + g.G[0] && gy >= -g.G[1] &&
                        gy < g.n[1] + g.G[1])
                        atomicAdd(Fg + (JX + c) * V + (long long)gy * rs + gx + l, vv[l]);
                continue;
            }
            atomicAdd(reinterpret_cast<float4 *>(Fg + (JX + c) * V + (long long)gy * rs + gx), v);
        }
        // (the next item's first barrier orders the flush before its records)
    }
}

template <int T, int ORDER, bool AGG, int NT = kPushThreads>
static void launch_T(const PartF32 &P, const TileItem *items, const uint32_t *nitems, long long max_items, float *F,
                     const Grid &g, const PushConst &pc, int *err, double *e_abs, cudaStream_t st)
{
    constexpr int smem = Box2p<T>::SMEM + 128;  // + alignment of the TMA destination
    static int nsm = 0, per_sm = 0;  // resident CTAs per SM
    if (!per_sm) {
        cudaFuncSetAttribute(k_push_tile2d<T, ORDER, AGG, NT>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_push_tile2d<T, ORDER, AGG, NT>, NT, smem);
        if (per_sm < 1) per_sm = 1;
    }
    // the six field components as one 3D tensor (x, y, component); tiles of
    // the box shape.  Without a tensor map the kernel stages with loads.
    CUtensorMap tmap;
    const int box[3] = {Box2p<T>::WX, Box2p<T>::WY, 6};
    const bool tma = tma_encode_field_map(&tmap, F, g.ext[0], g.ext[1], g.sy, g.vol, 6, box);
    if (!tma) memset(&tmap, 0, sizeof tmap);
    long long grid = std::min<long long>(max_items, (long long)nsm * per_sm);  // one resident wave
    if (grid < 1) grid = 1;
    note_launch();
    k_push_tile2d<T, ORDER, AGG, NT><<<(int)grid, NT, smem, st>>>(P, items, nitems, F, g, pc, err, e_abs, tmap,
                                                                       tma ? 1 : 0);
}

template <int T>
static void launch_variant(const PartF32 &P, const TileItem *items, const uint32_t *nitems, long long max_items,
                           float *F, const Grid &g, const PushConst &pc, int *err, double *e_abs, cudaStream_t st,
                           bool agg)
{
    if constexpr (T == 8)
        // tiles of 8 x 8 cells hold few particles: CTAs of 128 threads, six an SM,
        // where there are tiles for all of them (768 x 768 cells, 1.5 a cell: 127 us
        // a step with 256 threads, 107 with 128, 2 a cell 137 and 122; order 4 275
        // and 211; 96 x 96 cells, 144 tiles, 8 a cell: 35 and 38)
        if (!agg && g.ntiles >= 6ll * sm_count()) {
            if (g.order == 4) launch_T<T, 4, false, 128>(P, items, nitems, max_items, F, g, pc, err, e_abs, st);
            else launch_T<T, 2, false, 128>(P, items, nitems, max_items, F, g, pc, err, e_abs, st);
            return;
        }
    if (g.order == 4) launch_T<T, 4, false>(P, items, nitems, max_items, F, g, pc, err, e_abs, st);
    else if (agg) launch_T<T, 2, true>(P, items, nitems, max_items, F, g, pc, err, e_abs, st);
    else launch_T<T, 2, false>(P, items, nitems, max_items, F, g, pc, err, e_abs, st);
}

void launch_push_tile2d(const PartF32 &P, const TileItem *items, const uint32_t *nitems, long long max_items,
                        float *F, const Grid &g, const PushConst &pc, int *err, double *e_abs, cudaStream_t st,
                        bool agg)
{
    if (P.n == 0) return;
    if ((1 << g.tile_log2[0]) == 16) launch_variant<16>(P, items, nitems, max_items, F, g, pc, err, e_abs, st, agg);
    else launch_variant<8>(P, items, nitems, max_items, F, g, pc, err, e_abs, st, agg);
}

}  // namespace pic
