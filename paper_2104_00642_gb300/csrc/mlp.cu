// mlp.cu -- training and evaluation kernels of the surrogate network that
// stands in for the QED tables (Sec. IV, Eqs. (23)/(24)).
//
// Training (one Adam step per iteration, all on the device, captured once
// as a CUDA graph and replayed):
//   data   : Philox (x0, r) samples, targets from the FP64 tables
//   fwd    : per warp 32 rows, mma.sync BF16 hidden layers, stores Z1..Z3
//   bwd    : per warp: dY, head gradients, deltas D3 -> D2 -> D1 through
//            the transposed weights on the tensor cores
//   wgrad  : dW_l = sum_rows D_{l+1} (x) bf16(a_l) in FP32, db_l = sum D
//   update : the partial sums added up, FP32 master update (Adam), BF16 image
//            rewrite, loss latch
// The samples need the iteration's number only, not the parameters: those of
// the next iteration are drawn beside the weight gradients, into the other of
// two buffers (MlpSlot; one graph per parity).
// Loss L = (1/B) sum_rows [(y0 - s)^2 + w (y1 - l)^2].
#include <cmath>

#include "mlp_host.cuh"
#include "qed.cuh"

namespace pic {

namespace {

__device__ __forceinline__ float bf16_round(float v) { return __bfloat162float(__float2bfloat16_rn(v)); }

// write parameter i (packed order) into the image
__device__ __forceinline__ void image_put(MlpImage *img, int i, float v)
{
    if (i < kOffB0) {
        img->W0[i - kOffW0] = bf16_round(v);
    } else if (i < kOffW1) {
        img->b0[i - kOffB0] = v;
    } else if (i < kOffB1 || (i >= kOffW2 && i < kOffB2)) {
        const bool two = i >= kOffW2;
        const int q = i - (two ? kOffW2 : kOffW1), n = q / kMlpH, k = q % kMlpH;
        __nv_bfloat16 *W = reinterpret_cast<__nv_bfloat16 *>(two ? img->W2 : img->W1);
        __nv_bfloat16 *WT = reinterpret_cast<__nv_bfloat16 *>(two ? img->W2T : img->W1T);
        const __nv_bfloat16 b = __float2bfloat16_rn(v);
        W[n * 2 * kMlpPitch + k] = b;
        WT[k * 2 * kMlpPitch + n] = b;
    } else if (i < kOffW2) {
        img->b1[i - kOffB1] = v;
    } else if (i < kOffW3) {
        img->b2[i - kOffB2] = v;
    } else if (i < kOffB3) {
        img->W3[i - kOffW3] = bf16_round(v);
    } else {
        img->b3[i - kOffB3] = v;
    }
}

__global__ void k_mlp_image(const float *__restrict__ P, MlpImage *img)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < kMlpNParams) image_put(img, i, P[i]);
}

// the samples of iteration *from + add and what its update needs of the
// schedule, into slot `to`: x0 uniform in [-1, 1] (ln chi uniform over the
// range), r uniform as the Monte Carlo draws it; targets from the FP64 tables
struct MlpData {
    QedTables T;
    int p;
    MlpNorm nrm;
    uint32_t k0, k1;
    const int *from;
    int add;
    MlpAdam a;
    MlpSlot to;
    long long B;
    float *X, *Y;
};
__device__ __forceinline__ void draw_sample(const MlpData &m, long long i)
{
    const QedTables &T = m.T;
    const MlpNorm &nrm = m.nrm;
    const MlpAdam &a = m.a;
    const MlpSlot &to = m.to;
    const int p = m.p, k = *m.from + m.add;
    const long long B = m.B;
    const uint32_t k0 = m.k0, k1 = m.k1;
    float *X = m.X, *Y = m.Y;
    if (i == 0) {
        const double frac = a.iters > 1 ? fmin((double)k / (double)(a.iters - 1), 1.0) : 1.0;
        *to.it = k;
        to.sched[0] = a.lr_final + 0.5 * (a.lr0 - a.lr_final) * (1.0 + cos(3.14159265358979323846 * frac));
        to.sched[1] = 1.0 - pow((double)a.beta1, (double)(k + 1));
        to.sched[2] = 1.0 - pow((double)a.beta2, (double)(k + 1));
    }
    if (i >= B) return;
    uint32_t w[4];
    philox4x32_10((uint32_t)i, (uint32_t)(i >> 32), (uint32_t)k, QP_TRAIN + p, k0, k1, w);
    const float x0 = (float)(2.0 * uniform24(w[0]) - 1.0);
    // emission: half the rows take r uniform, half r = 1 - (1 - t)^2 with t
    // uniform (uniform in the network's r coordinate), so that the hard end of
    // the spectrum (r -> 1), which carries most of the emitted energy, is
    // sampled as densely as the soft end
    const double t = uniform24(w[1]);
    const double r = p == QED_RAD && (w[2] & 1u) ? 1.0 - (1.0 - t) * (1.0 - t) : t;
    const double lnchi = ((double)x0 - nrm.x0b) / nrm.x0a, chi = exp(lnchi);
    const double rr = p == QED_PAIR ? fmin(r, 1.0 - r) : r;
    const double s = cbrt(qed_sample<double>(T, p, chi, rr));
    const double lg = qed_lnG_table<double>(T, p, (lnchi - T.lnchi0) / T.dlnchi);
    X[2 * i] = x0;
    X[2 * i + 1] = (float)mlp_rcoord(p, r);
    Y[2 * i] = (float)s;
    Y[2 * i + 1] = (float)((lg - nrm.mu) / nrm.sd);
}
__global__ void __launch_bounds__(256) k_mlp_data(MlpData m) { draw_sample(m, (long long)blockIdx.x * 256 + threadIdx.x); }

// rows of this thread's quad group: rr = 16 (r >> 1) + 8 (r & 1) + g
__device__ __forceinline__ long long quad_row(long long row0, int r, int g) { return row0 + 16 * (r >> 1) + 8 * (r & 1) + g; }

// (one m-tile of 16 rows a warp, eight warps a CTA: see k_mlp_bwd)
__global__ void __launch_bounds__(256) k_mlp_fwd(const MlpImage *img, long long B, const float *__restrict__ X,
                                                 MlpZ Z, float *__restrict__ Y)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const long long row0 = ((long long)blockIdx.x * 8 + (threadIdx.x >> 5)) * 16;
    const int g = (threadIdx.x & 31) >> 2, t = threadIdx.x & 3;
    float x[4][2] = {}, y[4][2];
    if (row0 < B)  // B is a multiple of 32: whole warps
#pragma unroll
        for (int r = 0; r < 2; r++) {
            const long long row = quad_row(row0, r, g);
            x[r][0] = X[2 * row];
            x[r][1] = X[2 * row + 1];
        }
    mlp_stage(smem, img, kMlpStageBytes);
    __syncthreads();
    if (row0 >= B) return;
    mlp_forward_rows<true>(*reinterpret_cast<const MlpImage *>(smem), x, y, Z, row0, 1);
    if (t == 0)
#pragma unroll
        for (int r = 0; r < 2; r++) {
            const long long row = quad_row(row0, r, g);
            Y[2 * row] = y[r][0];
            Y[2 * row + 1] = y[r][1];
        }
}

// head: per-warp partials of dW3 (128), db3 (2) and the loss (1)
constexpr int kHeadPartial = 2 * kMlpH + 3;

// Two warps take a group of 32 rows, one m-tile (16 rows) each: a CTA per SM
// leaves every warp alone on its scheduler, waiting for one layer's values
// after the other, so a warp's share is halved and all its pre-activations are
// requested before the weights are staged (35.7 -> 13.2 us a batch of 16384).
// The head's sums run over the four rows of a lane in order, as in one warp:
// the second warp goes on from the first one's.
__global__ void __launch_bounds__(256) k_mlp_bwd(const MlpImage *img, long long B, const float *__restrict__ Tg,
                                                 const float *__restrict__ Y, MlpZ Z, MlpZ D, float *__restrict__ head,
                                                 float w_rate)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const int group = (threadIdx.x >> 5) & 3, m = threadIdx.x >> 7;
    // per group and lane: the first warp's 32 head sums, loss and row sums
    float(*pass)[36][32] = reinterpret_cast<float(*)[36][32]>(smem + kMlpTrainStageBytes);
    const long long row0 = ((long long)blockIdx.x * 4 + group) * 32;
    const bool live = row0 < B;  // B is a multiple of 32: whole groups
    float2 z[3][8][2];
#pragma unroll
    for (int l = 2; l >= 0; l--)
#pragma unroll
        for (int nt = 0; nt < 8; nt++)
#pragma unroll
            for (int h = 0; h < 2; h++)
                z[l][nt][h] = live ? *reinterpret_cast<const float2 *>(&Z.z[l][quad_row(row0, 2 * m + h, g) * kMlpH + 8 * nt + 2 * t])
                                   : make_float2(0.f, 0.f);
    mlp_stage(smem, img, kMlpTrainStageBytes);
    __syncthreads();
    const MlpImage &S = *reinterpret_cast<const MlpImage *>(smem);
    const float invB = 1.0f / (float)B;
    float dy[2][2], lv[2][2];
#pragma unroll
    for (int h = 0; h < 2; h++) {
        const long long row = quad_row(row0, 2 * m + h, g);
#pragma unroll
        for (int o = 0; o < 2; o++) {
            const float e = live ? Y[2 * row + o] - Tg[2 * row + o] : 0.f, w = o ? w_rate : 1.0f;
            dy[h][o] = 2.0f * w * e * invB;
            lv[h][o] = w * e;
            lv[h][o] = lv[h][o] * e;
        }
    }
    // head: D3 = (dy W3) * silu'(z3); dW3 = sum dy a3; db3 = sum dy
    float d[8][4], a[8][4];
#pragma unroll
    for (int nt = 0; nt < 8; nt++)
#pragma unroll
        for (int h = 0; h < 2; h++) {
            const int c = 8 * nt + 2 * t;
            const float zz[2] = {z[2][nt][h].x, z[2][nt][h].y};
#pragma unroll
            for (int e = 0; e < 2; e++) {
                a[nt][2 * h + e] = silu(zz[e]);
                const float da = dy[h][0] * S.W3[c + e] + dy[h][1] * S.W3[kMlpH + c + e];
                d[nt][2 * h + e] = da * dsilu(zz[e]);
            }
            if (live)
                *reinterpret_cast<float2 *>(&D.z[2][quad_row(row0, 2 * m + h, g) * kMlpH + c]) =
                    make_float2(d[nt][2 * h], d[nt][2 * h + 1]);
        }
    // this group's partial sums of the head gradient and the loss (summed over
    // groups in a fixed order by k_mlp_update: training is deterministic)
    auto head_sums = [&](float (*gw)[16], float &lsum) {
#pragma unroll
        for (int nt = 0; nt < 8; nt++)
#pragma unroll
            for (int h = 0; h < 2; h++)
#pragma unroll
                for (int e = 0; e < 2; e++) {
                    gw[0][2 * nt + e] = fmaf(dy[h][0], a[nt][2 * h + e], gw[0][2 * nt + e]);
                    gw[1][2 * nt + e] = fmaf(dy[h][1], a[nt][2 * h + e], gw[1][2 * nt + e]);
                }
#pragma unroll
        for (int h = 0; h < 2; h++)
#pragma unroll
            for (int o = 0; o < 2; o++) lsum = fmaf(lv[h][o], invB, lsum);
    };
    float gw[2][16], lsum = 0.f;
#pragma unroll
    for (int q = 0; q < 16; q++) gw[0][q] = gw[1][q] = 0.f;
    if (m == 0) {
        head_sums(gw, lsum);
#pragma unroll
        for (int q = 0; q < 16; q++) {
            pass[group][q][lane] = gw[0][q];
            pass[group][16 + q][lane] = gw[1][q];
        }
        pass[group][32][lane] = lsum;
        pass[group][33][lane] = dy[0][0] + dy[1][0];
        pass[group][34][lane] = dy[0][1] + dy[1][1];
    }
    __syncthreads();
    if (m == 1 && live) {
#pragma unroll
        for (int q = 0; q < 16; q++) {
            gw[0][q] = pass[group][q][lane];
            gw[1][q] = pass[group][16 + q][lane];
        }
        lsum = pass[group][32][lane];
        head_sums(gw, lsum);
        float *ph = head + (row0 / 32) * kHeadPartial;
#pragma unroll
        for (int o = 0; o < 2; o++)
#pragma unroll
            for (int q = 0; q < 16; q++) {
                float v = gw[o][q];
                v += __shfl_xor_sync(0xffffffffu, v, 4);
                v += __shfl_xor_sync(0xffffffffu, v, 8);
                v += __shfl_xor_sync(0xffffffffu, v, 16);
                if (g == 0) ph[o * kMlpH + 8 * (q >> 1) + 2 * t + (q & 1)] = v;
            }
        // db3 and the loss: the quad's lanes hold the same rows; count lane t == 0
#pragma unroll
        for (int o = 0; o < 2; o++) {
            float v = t == 0 ? pass[group][33 + o][lane] + dy[0][o] + dy[1][o] : 0.f;
#pragma unroll
            for (int sh = 16; sh > 0; sh >>= 1) v += __shfl_xor_sync(0xffffffffu, v, sh);
            if (lane == 0) ph[2 * kMlpH + o] = v;
        }
        lsum = t == 0 ? lsum : 0.f;
#pragma unroll
        for (int sh = 16; sh > 0; sh >>= 1) lsum += __shfl_xor_sync(0xffffffffu, lsum, sh);
        if (lane == 0) ph[2 * kMlpH + 2] = lsum;
    }
    if (!live) return;
    // D2 = (D3 W2) * silu'(z2), D1 = (D2 W1) * silu'(z1), on the tensor cores
    uint32_t A[4][4];
    float acc[8][4];
    auto ident = [](float x, float y) { return pack_bf16(x, y); };
#pragma unroll
    for (int l = 1; l >= 0; l--) {
        mlp_repack(d, A, ident);
        mlp_layer(l == 1 ? S.W2T : S.W1T, nullptr, A, acc);
#pragma unroll
        for (int nt = 0; nt < 8; nt++)
#pragma unroll
            for (int h = 0; h < 2; h++) {
                d[nt][2 * h] = acc[nt][2 * h] * dsilu(z[l][nt][h].x);
                d[nt][2 * h + 1] = acc[nt][2 * h + 1] * dsilu(z[l][nt][h].y);
                *reinterpret_cast<float2 *>(&D.z[l][quad_row(row0, 2 * m + h, g) * kMlpH + 8 * nt + 2 * t]) =
                    make_float2(d[nt][2 * h], d[nt][2 * h + 1]);
            }
    }
}
constexpr int kBwdSmem = kMlpTrainStageBytes + 4 * 36 * 32 * (int)sizeof(float);

// dW_l[j][k] = sum_rows D_{l+1}[row][j] in_l[row][k], db_l[j] = sum_rows D;
// in_0 = X (K = 2), in_l = bf16(silu(Z_l)) as the forward fed the tensor
// cores.  blockIdx.y = l; blocks stride over 64-row chunks staged in shared
// memory; a warp owns 8 j and all k, a thread 8 j x 2 k: the row's D are
// broadcasts, its A two banks a lane (4 x 4 tiles, 16 lanes apart in j, took
// twice the shared-memory wavefronts).
// Each block writes its partial sums (packed parameter order, layers 0-2)
// to its own row of `part`; k_mlp_update (k_mlp_reduce for a gradient alone)
// adds the rows in a fixed order.
//
// The blocks past the three layers (blockIdx.y = 3, training) draw the next
// iteration's samples: they need nothing of this one, and the FP64 units they
// keep busy are idle otherwise (19 us as a kernel of its own; 10 us on a
// second branch of the graph, for its fork and join).
constexpr int kWgRows = 64;
constexpr int kWgBlocks = 64;
__global__ void __launch_bounds__(256) k_mlp_wgrad(long long B, const float *__restrict__ X, MlpZ Z, MlpZ D,
                                                   float *__restrict__ part, MlpData next)
{
    if (blockIdx.y == 3) {
        for (long long i = (long long)blockIdx.x * 256 + threadIdx.x; i < B; i += (long long)gridDim.x * 256)
            draw_sample(next, i);
        return;
    }
    float *grad = part + (size_t)blockIdx.x * kOffW3;
    __shared__ __align__(16) float Ds[kWgRows][kMlpH];
    __shared__ __align__(16) float As[kWgRows][kMlpH];
    const int l = blockIdx.y;
    const float *Dl = D.z[l];
    const int j0 = 8 * (threadIdx.x >> 5), k0 = 2 * (threadIdx.x & 31), jb = threadIdx.x & 7;
    float acc[8][2], bacc = 0.f;
#pragma unroll
    for (int a = 0; a < 8; a++) acc[a][0] = acc[a][1] = 0.f;
    // a chunk's values in registers, requested while the chunk before it is
    // multiplied
    constexpr int kPer = kWgRows * kMlpH / 4 / 256;
    float4 dv[kPer], zv[kPer];
    auto fetch = [&](long long r0) {
#pragma unroll
        for (int q = 0; q < kPer; q++) {
            const int idx = threadIdx.x + 256 * q, r = idx / (kMlpH / 4), c = 4 * (idx % (kMlpH / 4));
            const long long row = r0 + r;
            dv[q] = zv[q] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (row < B) {
                dv[q] = *reinterpret_cast<const float4 *>(&Dl[row * kMlpH + c]);
                if (l > 0) zv[q] = *reinterpret_cast<const float4 *>(&Z.z[l - 1][row * kMlpH + c]);
                else if (c == 0) zv[q] = make_float4(X[2 * row], X[2 * row + 1], 0.f, 0.f);
            }
        }
    };
    const long long stride = (long long)gridDim.x * kWgRows;
    fetch((long long)blockIdx.x * kWgRows);
    for (long long r0 = (long long)blockIdx.x * kWgRows; r0 < B; r0 += stride) {
        __syncthreads();
#pragma unroll
        for (int q = 0; q < kPer; q++) {
            const int idx = threadIdx.x + 256 * q, r = idx / (kMlpH / 4), c = 4 * (idx % (kMlpH / 4));
            float4 av = zv[q];
            if (l > 0 && r0 + r < B) {
                const uint32_t a01 = silu2_bf16(av.x, av.y), a23 = silu2_bf16(av.z, av.w);
                av = make_float4(bf16_lo(a01), bf16_hi(a01), bf16_lo(a23), bf16_hi(a23));
            }
            *reinterpret_cast<float4 *>(&Ds[r][c]) = dv[q];
            *reinterpret_cast<float4 *>(&As[r][c]) = av;
        }
        __syncthreads();
        if (r0 + stride < B) fetch(r0 + stride);
        if (l == 0) {  // two inputs: one thread a row of dW_0 (the 64 x 64 product would be 62/64 zeros)
            if (threadIdx.x < kMlpH)
#pragma unroll 8
                for (int r = 0; r < kWgRows; r++) {
                    const float d = Ds[r][threadIdx.x];
                    bacc += d;
                    acc[0][0] = fmaf(d, As[r][0], acc[0][0]);
                    acc[0][1] = fmaf(d, As[r][1], acc[0][1]);
                }
            continue;
        }
#pragma unroll 4
        for (int r = 0; r < kWgRows; r++) {
            const float4 d0 = *reinterpret_cast<const float4 *>(&Ds[r][j0]);
            const float4 d1 = *reinterpret_cast<const float4 *>(&Ds[r][j0 + 4]);
            const float2 a = *reinterpret_cast<const float2 *>(&As[r][k0]);
            const float dd[8] = {d0.x, d0.y, d0.z, d0.w, d1.x, d1.y, d1.z, d1.w};
            bacc += Ds[r][j0 + jb];
#pragma unroll
            for (int p = 0; p < 8; p++) {
                acc[p][0] = fmaf(dd[p], a.x, acc[p][0]);
                acc[p][1] = fmaf(dd[p], a.y, acc[p][1]);
            }
        }
    }
    if (l == 0) {
        if (threadIdx.x < kMlpH) {
            grad[kOffW0 + 2 * threadIdx.x] = acc[0][0];
            grad[kOffW0 + 2 * threadIdx.x + 1] = acc[0][1];
            grad[kOffB0 + threadIdx.x] = bacc;
        }
        return;
    }
    const int offW = l == 1 ? kOffW1 : kOffW2, offB = l == 1 ? kOffB1 : kOffB2;
#pragma unroll
    for (int p = 0; p < 8; p++)
        *reinterpret_cast<float2 *>(&grad[offW + (j0 + p) * kMlpH + k0]) = make_float2(acc[p][0], acc[p][1]);
    if (k0 < 16) grad[offB + j0 + jb] = bacc;
}

// The gradient and the loss from the partial sums, in a fixed order: layers
// 0-2 over the wgrad blocks, the head and the loss over the warps.  The first
// kRedBlk0 blocks own a parameter of layers 0-2 per thread, 32 of its partials
// read at a time; the others own kRedCols columns of the head's partials,
// staged through shared memory, each summed by one thread (512 dependent
// reads a thread took 22 us).  Small blocks: Adam's FP64 quotients and root
// bind on the two FP64 lanes of an SM.  put(i, sum) takes the sums (i =
// kMlpNParams: the loss).
constexpr int kRedThreads = 64, kRedCols = 2, kRedRows = 512;
constexpr int kRedBlk0 = (kOffW3 + kRedThreads - 1) / kRedThreads;
constexpr int kRedBlk1 = (kHeadPartial + kRedCols - 1) / kRedCols;
template <class Put>
__device__ __forceinline__ void reduce_partials(const float *__restrict__ part, int nblk,
                                                const float *__restrict__ head, int nwarp, Put put)
{
    if (blockIdx.x < kRedBlk0) {
        const int i = blockIdx.x * kRedThreads + threadIdx.x;
        if (i >= kOffW3) return;
        float s = 0.f;
        for (int b0 = 0; b0 < nblk; b0 += 32) {
            float v[32];
#pragma unroll
            for (int b = 0; b < 32; b++) v[b] = b0 + b < nblk ? part[(size_t)(b0 + b) * kOffW3 + i] : 0.f;
#pragma unroll
            for (int b = 0; b < 32; b++)
                if (b0 + b < nblk) s += v[b];
        }
        put(i, s);
        return;
    }
    __shared__ float t[kRedRows][kRedCols + 1];
    const int c0 = (blockIdx.x - kRedBlk0) * kRedCols;
    float s = 0.f;
    for (int w0 = 0; w0 < nwarp; w0 += kRedRows) {
        const int rows = min(kRedRows, nwarp - w0);
        __syncthreads();
        for (int e = threadIdx.x; e < rows * kRedCols; e += kRedThreads) {
            const int r = e / kRedCols, c = e % kRedCols;
            if (c0 + c < kHeadPartial) t[r][c] = head[(size_t)(w0 + r) * kHeadPartial + c0 + c];
        }
        __syncthreads();
        if (threadIdx.x < kRedCols) {
#pragma unroll 16
            for (int r = 0; r < rows; r++) s += t[r][threadIdx.x];
        }
    }
    if (threadIdx.x < kRedCols && c0 + (int)threadIdx.x < kHeadPartial) put(kOffW3 + c0 + threadIdx.x, s);
}

__global__ void __launch_bounds__(kRedThreads) k_mlp_reduce(const float *__restrict__ part, int nblk,
                                                            const float *__restrict__ head, int nwarp,
                                                            float *__restrict__ grad, float *loss)
{
    reduce_partials(part, nblk, head, nwarp, [&](int i, float s) {
        if (i < kMlpNParams) grad[i] = s;
        else *loss = s;
    });
}

// the sums straight into Adam's update of the FP32 master and the BF16 image,
// and the loss of the iteration; sched: the learning rate and the bias
// corrections (k_mlp_data)
__global__ void __launch_bounds__(kRedThreads) k_mlp_update(const float *__restrict__ part, int nblk,
                                                            const float *__restrict__ head, int nwarp,
                                                            float *__restrict__ P, float *__restrict__ M,
                                                            float *__restrict__ V, MlpImage *img,
                                                            const double *__restrict__ sched, MlpAdam a, float *loss_last)
{
    const double lr = sched[0], c1 = sched[1], c2 = sched[2];
    reduce_partials(part, nblk, head, nwarp, [&](int i, float g) {
        if (i == kMlpNParams) {
            *loss_last = g;
            return;
        }
        const float m = a.beta1 * M[i] + (1.0f - a.beta1) * g;
        const float v = a.beta2 * V[i] + (1.0f - a.beta2) * g * g;
        M[i] = m;
        V[i] = v;
        const float p = P[i] - (float)(lr * ((double)m / c1) / (sqrt((double)v / c2) + a.eps));
        P[i] = p;
        image_put(img, i, p);
    });
}

// raw network on normalised inputs (testing): one warp per 32 rows
__global__ void __launch_bounds__(128) k_mlp_eval(const MlpImage *img, long long n, const float *__restrict__ X,
                                                  float *__restrict__ Y)
{
    extern __shared__ __align__(16) unsigned char smem[];
    mlp_stage(smem, img, kMlpStageBytes);
    __syncthreads();
    const MlpImage &S = *reinterpret_cast<const MlpImage *>(smem);
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (!__any_sync(0xffffffffu, i < n)) return;
    const bool ok = i < n;
    float y0, y1;
    mlp_eval_warp(S, ok ? X[2 * i] : 0.f, ok ? X[2 * i + 1] : 0.f, y0, y1);
    if (ok) {
        Y[2 * i] = y0;
        Y[2 * i + 1] = y1;
    }
}

// what the Monte Carlo uses for (chi, r): the network inside its range,
// the tables (of the simulation's precision) outside (r == nullptr: G;
// else the energy fraction)
template <typename R>
__global__ void __launch_bounds__(128) k_qed_eval_surr(const MlpImage *img, MlpNorm nrm, QedTables T, int p,
                                                       long long n, const double *__restrict__ chi,
                                                       const double *__restrict__ r, double *__restrict__ out)
{
    extern __shared__ __align__(16) unsigned char smem[];
    mlp_stage(smem, img, kMlpStageBytes);
    __syncthreads();
    const MlpImage &S = *reinterpret_cast<const MlpImage *>(smem);
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (!__any_sync(0xffffffffu, i < n)) return;
    const bool ok = i < n;
    const double c = ok ? chi[i] : 1.0, rv = ok && r ? r[i] : 0.5;
    double lnchi;
    const bool inr = ok && mlp_in_range(nrm, c, lnchi);
    float x0 = 0.f, x1 = 0.f, y0 = 0.f, y1 = 0.f;
    if (inr) mlp_inputs(nrm, p, lnchi, rv, x0, x1);
    if (__any_sync(0xffffffffu, inr)) mlp_eval_warp_sparse(S, inr, x0, x1, y0, y1);
    if (!ok) return;
    if constexpr (sizeof(R) == 4) {  // in FP32, as the FP32 pushes evaluate it
        const float cf = (float)c, rf = (float)rv;
        if (r) out[i] = inr ? mlp_fraction_f32(p, y0, rf) : qed_sample_f32(T, p, cf, rf);
        else out[i] = inr ? mlp_rate_f32(nrm, p, cf, y1) : qed_rate_f32(T, p, cf);
    } else {
        if (r) out[i] = inr ? mlp_fraction(p, y0, rv) : qed_sample<R>(T, p, c, rv);
        else out[i] = inr ? mlp_rate(nrm, p, c, y1) : qed_rate<R>(T, p, c);
    }
}

// errors of the network against the FP64 tables on a (ln chi, r) grid of
// cell midpoints: acc[0] = max |d ln G|, acc[1] = max |d s|, acc[2] = sum d s^2
__global__ void __launch_bounds__(128) k_mlp_validate(const MlpImage *img, MlpNorm nrm, QedTables T, int p, int nc,
                                                      int nr, double *acc)
{
    extern __shared__ __align__(16) unsigned char smem[];
    mlp_stage(smem, img, kMlpStageBytes);
    __syncthreads();
    const MlpImage &S = *reinterpret_cast<const MlpImage *>(smem);
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long n = (long long)nc * nr;
    if (!__any_sync(0xffffffffu, i < n)) return;
    const bool ok = i < n;
    const int ic = ok ? (int)(i / nr) : 0, jr = ok ? (int)(i % nr) : 0;
    const double lnchi = nrm.lnchi_lo + (ic + 0.5) / nc * (nrm.lnchi_hi - nrm.lnchi_lo);
    const double r = (jr + 0.5) / nr;
    float x0, x1, y0, y1;
    mlp_inputs(nrm, p, lnchi, r, x0, x1);
    mlp_eval_warp(S, x0, x1, y0, y1);
    if (!ok) return;
    const double chi = exp(lnchi);
    const double s_tab = cbrt(qed_sample<double>(T, p, chi, p == QED_PAIR ? fmin(r, 1.0 - r) : r));
    const double es = fabs((double)y0 - s_tab);
    const double eg = fabs((double)fmaf(nrm.sd, y1, nrm.mu) - qed_lnG_table<double>(T, p, (lnchi - T.lnchi0) / T.dlnchi));
    // non-negative doubles order as their bit patterns
    atomicMax(reinterpret_cast<unsigned long long *>(&acc[0]), (unsigned long long)__double_as_longlong(eg));
    atomicMax(reinterpret_cast<unsigned long long *>(&acc[1]), (unsigned long long)__double_as_longlong(es));
    atomicAdd(&acc[2], es * es);
    const double ft = s_tab * s_tab * s_tab;
    atomicAdd(&acc[4 + 2 * ic], mlp_fraction(p, y0, r));
    atomicAdd(&acc[5 + 2 * ic], p == QED_PAIR && r > 0.5 ? 1.0 - ft : ft);
}

int div_up_i(long long a, int b) { return (int)((a + b - 1) / b); }

void launch_bwd(const MlpImage *img, long long B, const float *Tg, const float *Y, const MlpZ &Z, const MlpZ &D,
                float *head, float w_rate, cudaStream_t st)
{
    static bool attr = false;
    if (!attr) {
        cudaFuncSetAttribute(k_mlp_bwd, cudaFuncAttributeMaxDynamicSharedMemorySize, kBwdSmem);
        attr = true;
    }
    k_mlp_bwd<<<div_up_i(B, 128), 256, kBwdSmem, st>>>(img, B, Tg, Y, Z, D, head, w_rate);
}

}  // namespace

void launch_mlp_image(const float *P, MlpImage *img, cudaStream_t st)
{
    note_launch();
    k_mlp_image<<<div_up_i(kMlpNParams, 256), 256, 0, st>>>(P, img);
}

void launch_mlp_forward(const MlpImage *img, long long B, const float *X, const MlpZ &Z, float *Y, cudaStream_t st)
{
    note_launch();
    k_mlp_fwd<<<div_up_i(B, 128), 256, kMlpStageBytes, st>>>(img, B, X, Z, Y);
}

size_t mlp_partial_floats(long long B) { return (size_t)kWgBlocks * kOffW3 + (size_t)(B / 32) * kHeadPartial; }

void launch_mlp_backward(const MlpImage *img, long long B, const float *X, const float *Tg, const float *Y,
                         const MlpZ &Z, const MlpZ &D, float *partials, float *grad, float w_rate, float *loss,
                         cudaStream_t st)
{
    float *part = partials, *head = partials + (size_t)kWgBlocks * kOffW3;
    note_launch(3);
    launch_bwd(img, B, Tg, Y, Z, D, head, w_rate, st);
    const int nb = std::min(div_up_i(B, kWgRows), kWgBlocks);
    k_mlp_wgrad<<<dim3(nb, 3), 256, 0, st>>>(B, X, Z, D, part, MlpData{});
    k_mlp_reduce<<<kRedBlk0 + kRedBlk1, kRedThreads, 0, st>>>(part, nb, head, (int)(B / 32), grad, loss);
}

static MlpData data_of(const MlpNet &net, MlpScratch &S, const MlpTraining &t, int from, int add, int to)
{
    return {t.T, t.p, net.nrm, t.key[0], t.key[1], S.slot[from].it, add, t.a, S.slot[to], t.B, S.XT[to], S.XT[to] + 2 * S.rows};
}

void launch_mlp_data(const MlpNet &net, MlpScratch &S, const MlpTraining &t, cudaStream_t st)
{
    note_launch();
    k_mlp_data<<<div_up_i(t.B, 256), 256, 0, st>>>(data_of(net, S, t, 0, 0, 0));
}

void mlp_train_iteration(MlpNet &net, MlpScratch &S, const MlpTraining &t, int slot, cudaStream_t st)
{
    float *X = S.XT[slot], *Tg = X + 2 * S.rows;
    float *part = S.partials, *head = S.partials + (size_t)kWgBlocks * kOffW3;
    launch_mlp_forward(net.img, t.B, X, S.Z, S.Y, st);
    note_launch(3);
    launch_bwd(net.img, t.B, Tg, S.Y, S.Z, S.D, head, t.w_rate, st);
    const int nb = std::min(div_up_i(t.B, kWgRows), kWgBlocks);
    k_mlp_wgrad<<<dim3(nb, 4), 256, 0, st>>>(t.B, X, S.Z, S.D, part, data_of(net, S, t, slot, 1, 1 - slot));
    k_mlp_update<<<kRedBlk0 + kRedBlk1, kRedThreads, 0, st>>>(part, nb, head, (int)(t.B / 32), net.P, net.M, net.V,
                                                             net.img, S.slot[slot].sched, t.a, S.loss + 1);
}

void launch_mlp_eval(const MlpImage *img, long long n, const float *X, float *Y, cudaStream_t st)
{
    note_launch();
    k_mlp_eval<<<div_up_i(n, 128), 128, kMlpStageBytes, st>>>(img, n, X, Y);
}

void launch_qed_eval_surr(const MlpImage *img, const MlpNorm &nrm, const QedTables &T, bool f64, int p, long long n,
                          const double *chi, const double *r, double *out, cudaStream_t st)
{
    note_launch();
    if (f64) k_qed_eval_surr<double><<<div_up_i(n, 128), 128, kMlpStageBytes, st>>>(img, nrm, T, p, n, chi, r, out);
    else k_qed_eval_surr<float><<<div_up_i(n, 128), 128, kMlpStageBytes, st>>>(img, nrm, T, p, n, chi, r, out);
}

void launch_mlp_validate(const MlpImage *img, const MlpNorm &nrm, const QedTables &T, int p, int nc, int nr,
                         double *acc, cudaStream_t st)
{
    note_launch();
    k_mlp_validate<<<div_up_i((long long)nc * nr, 128), 128, kMlpStageBytes, st>>>(img, nrm, T, p, nc, nr, acc);
}

}  // namespace pic
