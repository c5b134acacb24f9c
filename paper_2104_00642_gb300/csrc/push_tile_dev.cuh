// push_tile_dev.cuh -- device helpers shared by the tiled pushes (push_tile2d.cu
// and push_tile3d.cu; of the QED species push_tile.cu and push_qed_tile3d.cu).
#pragma once
#include "push_dev.cuh"
#include "push_tile.cuh"

namespace pic {

// shapes of the start (i0, w0) and end (i1, w1) points on the 4-node union
// window [u0, u0+3], u0 = min(i0, i1) - 1 (|i1 - i0| <= 1)
__device__ __forceinline__ int union4(int i0, const float *w0, int i1, const float *w1, float *S0, float *dS)
{
    const int u0 = min(i0, i1) - 1;
    const int o0 = i0 - 1 - u0, o1 = i1 - 1 - u0;  // each 0 or 1
#pragma unroll
    for (int k = 0; k < 4; k++) {
        float s0 = o0 ? (k >= 1 ? w0[k - 1] : 0.f) : (k <= 2 ? w0[k] : 0.f);
        float s1 = o1 ? (k >= 1 ? w1[k - 1] : 0.f) : (k <= 2 ? w1[k] : 0.f);
        S0[k] = s0;
        dS[k] = s1 - s0;
    }
    return u0;
}

// current into the shared box as 32-bit fixed point (integer shared-memory
// atomics are native; float ones are not), the values already in the units of
// the box (the caller folds the scale into the deposit's coefficients).  Where
// the units are fixed per launch they are 2^20 per C, C = |q w| max(dx_d/dt):
// an item's particles (at most 1024, each adding at most C in magnitude to a
// node) keep a node below 2^30, and rounding a value costs at most 2^-21 C.
struct AccSharedUnits {
    int *base;
    int cs, rs;
    __device__ __forceinline__ void add(int c, int a, int b, float v)
    {
        atomicAdd(base + c * cs + b * rs + a, __float2int_rn(v));
    }
};

// the whole warp on one window: each value summed over the 32 lanes (one
// warp reduction; 32 values of at most 2^20 units stay inside int32) and
// added once by the lead lane
struct AccWarpAll {
    int *base;
    int cs, rs;
    bool lead;
    __device__ __forceinline__ void add(int c, int a, int b, float v)
    {
        const int s = __reduce_add_sync(0xffffffffu, __float2int_rn(v));
        if (lead) atomicAdd(base + c * cs + b * rs + a, s);
    }
};

// drift_f32 with selects instead of branches (a warp of a hot plasma always
// has lanes on both sides of a branch, three drifts per axis and particle):
// the offset o + h u ginv, h = dt/(2 dx), with face crossing
__device__ __forceinline__ void drift_sel_f32(int &c, float &o, float h, float u, float ginv)
{
    const float on = fmaf(h * u, ginv, o);
    const bool up = on >= 1.0f, dn = on < 0.0f;
    const float w = dn ? on + 1.0f : on;  // in (0, 1], or on itself
    const bool face = dn && w >= 1.0f;    // a tiny negative offset rounded up to 1: the particle sits on the face
    o = up ? on - 1.0f : (face ? 0.0f : w);
    c += (up ? 1 : 0) - (dn && !face ? 1 : 0);
}

// Per-warp sums of v_d over the records a thread filed, from its sums of |v_d|
// and (SIGNED) of v_d: of the positive ones (x) and of the negative ones (y), or
// of all |v_d| (x).  In units of 2^-20, rounded up per thread (an item's 1024
// records stay below 2^30), so that one integer reduction a value does it.
template <bool SIGNED, int NW>
__device__ __forceinline__ void warp_sums(const float *vabs, const float *v, int2 (*sum)[NW])
{
#pragma unroll
    for (int d = 0; d < 3; d++) {
        int2 t = make_int2(0, 0);
        if constexpr (SIGNED) {
            t.x = __reduce_add_sync(0xffffffffu, __float2int_ru((vabs[d] + v[d]) * 524288.0f));
            t.y = __reduce_add_sync(0xffffffffu, __float2int_ru((vabs[d] - v[d]) * 524288.0f));
        } else {
            t.x = __reduce_add_sync(0xffffffffu, __float2int_ru(vabs[d] * 1048576.0f));
        }
        if ((threadIdx.x & 31u) == 0) sum[d][threadIdx.x >> 5] = t;
    }
}

// Fixed-point units per unit of current for an item of n records whose
// particles' sums of v_d are in sum (per warp), each adding values of the sign
// of q w v_d, at most shape |q w v_d| to a node: a node's value lies between the
// sums of the particles of either sign, so the larger of the two takes 2^31
// less a margin for the roundings (at most half a unit per particle, and FP32's
// in the sums).  In a plasma that is half the sum of all |v_d|, which does for
// the others, and half the rounding of a node.
//
// What a record adds along an active axis is not q w v_d but q w dx_d / dt
// (cj) times the difference of two weights at FP32 offsets: two drifts, each
// rounded by up to 2^-24 cells, and weights good to about 2^-22 (order 4).  For
// slow particles that is most of the move, so every record counts with 2^-20
// cells more; of a thermal particle's move it is 1e-5.
template <int NW>
__device__ __forceinline__ float box_units(const int2 (&sum)[NW], float qw, int n, float cj, float shape)
{
    int p = 0, m = 0;
#pragma unroll
    for (int w = 0; w < NW; w++) {
        p += sum[w].x;
        m += sum[w].y;
    }
    constexpr float u = 9.5367432e-7f;  // 2^-20
    return 2.14e9f / fmaxf(shape * fmaf(fabsf(qw), (float)max(p, m) * u, (float)n * fabsf(cj * u)), 1e-28f);
}

// the deposit phase's rows of 32 records (an odd number: see deposit_row2d),
// taken by the CTA's warps as they come free, the costlier ones first: a
// fixed share of the rows left warps waiting at the barrier (2.5 of 11 warps
// stalled there in the 3D push, 9 rows on 8 warps)
__device__ __forceinline__ int deposit_rows(int n) { return n ? ((n + 31) >> 5) | 1 : 0; }
__device__ __forceinline__ int next_row(int *taken)
{
    int j = 0;
    if ((threadIdx.x & 31u) == 0) j = atomicAdd(taken, 1);
    return __shfl_sync(0xffffffffu, j, 0);
}

// Boris (Eqs. (13)-(16)) with the FP32 reciprocal square root and divide
// of the special-function unit (a few ulp, far inside the FP32 tolerance)
__device__ __forceinline__ void boris_fast(float &ux, float &uy, float &uz, float ex, float ey, float ez, float bx,
                                           float by, float bz)
{
    float umx = ux + ex, umy = uy + ey, umz = uz + ez;
    float ginv = rsqrtf(1.0f + umx * umx + umy * umy + umz * umz);
    float tx = bx * ginv, ty = by * ginv, tz = bz * ginv;
    float t2 = tx * tx + ty * ty + tz * tz;
    float upx = umx + (umy * tz - umz * ty);
    float upy = umy + (umz * tx - umx * tz);
    float upz = umz + (umx * ty - umy * tx);
    float f = __fdividef(2.0f, 1.0f + t2);
    float sx = tx * f, sy = ty * f, sz = tz * f;
    ux = umx + (upy * sz - upz * sy) + ex;
    uy = umy + (upz * sx - upx * sz) + ey;
    uz = umz + (upx * sy - upy * sx) + ez;
}

// the FP64 island above gamma ~ 1e4, out of line: a lane below it never
// issues its FP64 instructions (this GPU runs FP64 at 1/73 of FP32)
static __device__ __noinline__ float inv_gamma_island(float ux, float uy, float uz)
{
    const double d2 = (double)ux * ux + (double)uy * uy + (double)uz * uz;
    return (float)(1.0 / sqrt(1.0 + d2));
}

__device__ __forceinline__ float inv_gamma_fast(float ux, float uy, float uz)
{
    float u2 = ux * ux + uy * uy + uz * uz;
    if (u2 < 1e8f) return rsqrtf(1.0f + u2);
    return inv_gamma_island(ux, uy, uz);
}

// The difference of an end point's weight and a start point's.  A step's end
// point is the next step's start point, so that what its weights round off
// cancels over the steps -- if it rounds alike in both places.  EXACT says so;
// left to the compiler the end point's last product is contracted into the
// difference and the roundings add up (E of a 1 keV plasma at order 4, 16
// steps: 9.3e-7 off 64 bits instead of 5.4e-7).
template <bool EXACT>
__device__ __forceinline__ float weight_step(float w1, float w0)
{
    return EXACT ? __fsub_rn(w1, w0) : w1 - w0;
}

// 1/gamma and Boris' update of a tiled push.  EXACT: with the correctly rounded
// root and quotients, as the one-thread pushes have them.
template <bool EXACT>
__device__ __forceinline__ float inv_gamma_tile(float ux, float uy, float uz)
{
    if constexpr (!EXACT) return inv_gamma_fast(ux, uy, uz);
    const float u2 = ux * ux + uy * uy + uz * uz;
    if (u2 < 1e8f) return 1.0f / sqrtf(1.0f + u2);
    return inv_gamma_island(ux, uy, uz);
}
template <bool EXACT>
__device__ __forceinline__ void boris_tile(float &ux, float &uy, float &uz, float ex, float ey, float ez, float bx,
                                           float by, float bz)
{
    if constexpr (EXACT) boris<float>(ux, uy, uz, ex, ey, ez, bx, by, bz);
    else boris_fast(ux, uy, uz, ex, ey, ez, bx, by, bz);
}

}  // namespace pic
