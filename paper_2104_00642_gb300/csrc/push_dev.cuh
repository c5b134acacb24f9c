// push_dev.cuh -- device helpers of the particle kernels: per-axis nearest
// node and W_2 weights (Sec. II.D), the gather of Eq. (19), Esirkepov's
// window and deposit (Eqs. (20)-(22)), and the FP32 offset drift.
#pragma once
#include "fp64_dev.cuh"
#include "push.cuh"

namespace pic {

// ---------------------------------------------------------------------
// per-axis nearest node and W_2 weights
// ---------------------------------------------------------------------

// W_4 (the cell integral of the order-4 shape S_4 of Eq. (18), the quartic
// B-spline): nodes ic-2 .. ic+2 for a particle at delta in [-1/2, 1/2)
template <typename R>
__device__ __forceinline__ void w4(R delta, R *w)
{
    const R d2 = delta * delta, d4 = d2 * d2;
    const R a = R(1) - R(2) * delta, b = R(1) + R(2) * delta;
    w[0] = (a * a) * (a * a) * R(1.0 / 384.0);
    w[1] = (R(19) - R(44) * delta + R(24) * d2 + R(16) * d2 * delta - R(16) * d4) * R(1.0 / 96.0);
    w[2] = R(115.0 / 192.0) - R(0.625) * d2 + R(0.25) * d4;
    w[3] = (R(19) + R(44) * delta + R(24) * d2 - R(16) * d2 * delta - R(16) * d4) * R(1.0 / 96.0);
    w[4] = (b * b) * (b * b) * R(1.0 / 384.0);
}

// the weights of shape order ORDER (2: W_2 on 3 nodes, 4: W_4 on 5 nodes)
template <typename R, int ORDER>
__device__ __forceinline__ void shape_w(R delta, R *w)
{
    if constexpr (ORDER == 4) w4<R>(delta, w);
    else w2<R>(delta, w);
}

// FP32 form: X = c + o
template <int ORDER = 2>
__device__ __forceinline__ void axis_w_f32(int c, float o, int &icn, float *wn, int &ich, float *wh)
{
    bool up = o >= 0.5f;
    icn = c + (up ? 1 : 0);
    shape_w<float, ORDER>(up ? o - 1.0f : o, wn);
    ich = c;
    shape_w<float, ORDER>(o - 0.5f, wh);
}

template <int ORDER = 2>
__device__ __forceinline__ void axis_wn_f32(int c, float o, int &icn, float *wn)
{
    bool up = o >= 0.5f;
    icn = c + (up ? 1 : 0);
    shape_w<float, ORDER>(up ? o - 1.0f : o, wn);
}

// FP64 form: X = x / dx
template <int ORDER = 2>
__device__ __forceinline__ void axis_w_f64(double X, int &icn, double *wn, int &ich, double *wh)
{
    icn = (int)floor(X + 0.5);
    shape_w<double, ORDER>(X - (double)icn, wn);
    ich = (int)floor(X);
    shape_w<double, ORDER>(X - ((double)ich + 0.5), wh);
}

template <int ORDER = 2>
__device__ __forceinline__ void axis_wn_f64(double X, int &icn, double *wn)
{
    icn = (int)floor(X + 0.5);
    shape_w<double, ORDER>(X - (double)icn, wn);
}

// Eq. (19): each component with its own staggered nearest node per axis,
// ORDER + 1 nodes per axis from ic - ORDER/2
template <typename R, int DIM, int ORDER = 2>
__device__ __forceinline__ void gather(const R *__restrict__ F, const Grid &g, const int *icn,
                                       const R (*wn)[ORDER + 1], const int *ich, const R (*wh)[ORDER + 1], R *eb)
{
    constexpr int P = ORDER + 1, H = ORDER / 2;
#pragma unroll
    for (int c = 0; c < 6; c++) {
        int ic[3];
        const R *w[3];
        ic[0] = stag(c, 0) ? ich[0] : icn[0];
        w[0] = stag(c, 0) ? wh[0] : wn[0];
        ic[1] = DIM >= 2 ? (stag(c, 1) ? ich[1] : icn[1]) : 0;
        w[1] = DIM >= 2 ? (stag(c, 1) ? wh[1] : wn[1]) : nullptr;
        ic[2] = DIM >= 3 ? (stag(c, 2) ? ich[2] : icn[2]) : 0;
        w[2] = DIM >= 3 ? (stag(c, 2) ? wh[2] : wn[2]) : nullptr;
        const R *Fc = F + (long long)c * g.vol;
        R acc = 0;
        if (DIM == 1) {
            long long o = goff(g, ic[0] - H, 0, 0);
#pragma unroll
            for (int a = 0; a < P; a++) acc += w[0][a] * __ldg(Fc + o + a);
        } else if (DIM == 2) {
#pragma unroll
            for (int b = 0; b < P; b++) {
                long long o = goff(g, ic[0] - H, ic[1] - H + b, 0);
                R r = 0;
#pragma unroll
                for (int a = 0; a < P; a++) r += w[0][a] * __ldg(Fc + o + a);
                acc += w[1][b] * r;
            }
        } else {
#pragma unroll
            for (int cc = 0; cc < P; cc++) {
                R r2 = 0;
#pragma unroll
                for (int b = 0; b < P; b++) {
                    long long o = goff(g, ic[0] - H, ic[1] - H + b, ic[2] - H + cc);
                    R r = 0;
#pragma unroll
                    for (int a = 0; a < P; a++) r += w[0][a] * __ldg(Fc + o + a);
                    r2 += w[1][b] * r;
                }
                acc += w[2][cc] * r2;
            }
        }
        eb[c] = acc;
    }
}

// the start and end shapes on the window of W nodes from min(i0, i1) - ORDER/2:
// W = ORDER + 1 (nearest node unmoved) or ORDER + 2 (moved by one at most)
template <typename R, int ORDER, int W>
__device__ __forceinline__ void window_w(int i0, const R *w0, int i1, const R *w1, R *S0, R *dS)
{
    constexpr int P = ORDER + 1;
    const bool o0 = W > P && i0 > i1, o1 = W > P && i1 > i0;
#pragma unroll
    for (int k = 0; k < W; k++) {
        const R s0 = o0 ? (k >= 1 ? w0[k - 1] : R(0)) : (k < P ? w0[k < P ? k : 0] : R(0));
        const R s1 = o1 ? (k >= 1 ? w1[k - 1] : R(0)) : (k < P ? w1[k < P ? k : 0] : R(0));
        S0[k] = s0;
        dS[k] = s1 - s0;
    }
}

// nonzero, by the bits (a compare of doubles takes the FP64 pipe)
__device__ __forceinline__ bool nonzero(double v) { return (__double2hiint(v) << 1 | __double2loint(v)) != 0; }
__device__ __forceinline__ bool nonzero(float v) { return v != 0.f; }

// Esirkepov's deposit into the global current on a window of W nodes
// (Eqs. (20)-(22)), with t = S0 + dS/2: along an active axis d the prefix sum
// of dS_d times the time average of the other axes' shapes (t_a t_b + dS_a
// dS_b / 12); along an inactive axis q w v_d times that average of all.
// base: the window's first node.
template <typename R, int DIM, int W>
__device__ __forceinline__ void deposit_window(R *__restrict__ F, const Grid &g, const int *base, const R (*S0)[W],
                                               const R (*dS)[W], const R *cJ, R jvy, R jvz)
{
    const long long o = goff(g, base[0], DIM > 1 ? base[1] : 0, DIM > 2 ? base[2] : 0);
    R *Jx = F + JX * g.vol + o, *Jy = F + JY * g.vol + o, *Jz = F + JZ * g.vol + o;
    const int sy = (int)g.sy, sz = (int)g.sz;
    R t[DIM][W], p[DIM][W - 1], d12[DIM][W];
#pragma unroll
    for (int d = 0; d < DIM; d++) {
        p[d][0] = cJ[d] * dS[d][0];
#pragma unroll
        for (int k = 0; k < W; k++) {
            t[d][k] = S0[d][k] + R(0.5) * dS[d][k];
            d12[d][k] = dS[d][k] * R(1.0 / 12.0);
            if (k > 0 && k < W - 1) p[d][k] = p[d][k - 1] + cJ[d] * dS[d][k];
        }
    }
    auto add = [](R *at, R v) {
        if (nonzero(v)) atomicAdd(at, v);
    };
    if constexpr (DIM == 1) {
#pragma unroll
        for (int a = 0; a < W; a++) {
            if (a < W - 1) add(Jx + a, p[0][a]);
            add(Jy + a, jvy * t[0][a]);
            add(Jz + a, jvz * t[0][a]);
        }
    } else if constexpr (DIM == 2) {
#pragma unroll
        for (int a = 0; a < W; a++) {
            const R ja = jvz * t[0][a], jd = jvz * d12[0][a];
#pragma unroll
            for (int b = 0; b < W; b++) {
                if (a < W - 1) add(Jx + b * sy + a, p[0][a] * t[1][b]);
                if (b < W - 1) add(Jy + b * sy + a, p[1][b] * t[0][a]);
                add(Jz + b * sy + a, ja * t[1][b] + jd * dS[1][b]);
            }
        }
    } else {
#pragma unroll 1
        for (int c = 0; c < W; c++) {
            R tc = t[2][0], dc = d12[2][0];
#pragma unroll
            for (int k = 1; k < W; k++) {
                tc = c == k ? t[2][k] : tc;
                dc = c == k ? d12[2][k] : dc;
            }
#pragma unroll
            for (int b = 0; b < W; b++) {
                const R w = t[1][b] * tc + dS[1][b] * dc;
#pragma unroll
                for (int a = 0; a < W - 1; a++) add(Jx + c * sz + b * sy + a, p[0][a] * w);
            }
#pragma unroll
            for (int a = 0; a < W; a++) {
                const R w = t[0][a] * tc + dS[0][a] * dc;
#pragma unroll
                for (int b = 0; b < W - 1; b++) add(Jy + c * sz + b * sy + a, p[1][b] * w);
            }
        }
#pragma unroll 1
        for (int b = 0; b < W; b++) {
            R tb = t[1][0], db = d12[1][0];
#pragma unroll
            for (int k = 1; k < W; k++) {
                tb = b == k ? t[1][k] : tb;
                db = b == k ? d12[1][k] : db;
            }
#pragma unroll
            for (int a = 0; a < W; a++) {
                const R w = t[0][a] * tb + dS[0][a] * db;
#pragma unroll
                for (int c = 0; c < W - 1; c++) add(Jz + c * sz + b * sy + a, p[2][c] * w);
            }
        }
    }
}

// the deposit of one particle from the nearest nodes and weights of its end
// points, on the smaller window when no lane of the warp's active ones moved
// its nearest node
template <typename R, int DIM, int ORDER>
__device__ __forceinline__ void deposit_moved(R *__restrict__ F, const Grid &g, const int *i0, const R (*w0)[ORDER + 1],
                                              const int *i1, const R (*w1)[ORDER + 1], const R *cJ, R jvy, R jvz)
{
    int base[3] = {0, 0, 0};
    bool moved = false;
#pragma unroll
    for (int d = 0; d < DIM; d++) {
        base[d] = min(i0[d], i1[d]) - ORDER / 2;
        moved |= i0[d] != i1[d];
    }
    if (__any_sync(__activemask(), moved)) {
        R S0[DIM][ORDER + 2], dS[DIM][ORDER + 2];
#pragma unroll
        for (int d = 0; d < DIM; d++) window_w<R, ORDER, ORDER + 2>(i0[d], w0[d], i1[d], w1[d], S0[d], dS[d]);
        deposit_window<R, DIM, ORDER + 2>(F, g, base, S0, dS, cJ, jvy, jvz);
    } else {
        R S0[DIM][ORDER + 1], dS[DIM][ORDER + 1];
#pragma unroll
        for (int d = 0; d < DIM; d++) window_w<R, ORDER, ORDER + 1>(i0[d], w0[d], i1[d], w1[d], S0[d], dS[d]);
        deposit_window<R, DIM, ORDER + 1>(F, g, base, S0, dS, cJ, jvy, jvz);
    }
}

// FP32 offset drift with face crossing: offset on (after a drift of less than a
// cell) back into [0, 1) and its cell
__device__ __forceinline__ void drift_to(int &c, float &o, float on)
{
    if (on >= 1.0f) {
        on -= 1.0f;
        c += 1;
    } else if (on < 0.0f) {
        on += 1.0f;
        c -= 1;
        if (on >= 1.0f) {  // a tiny negative offset rounded up to 1: the particle sits on the face
            on = 0.0f;
            c += 1;
        }
    }
    o = on;
}
__device__ __forceinline__ void drift_f32(int &c, float &o, float d) { drift_to(c, o, o + d); }
}  // namespace pic
