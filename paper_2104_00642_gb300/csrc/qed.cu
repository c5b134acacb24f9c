// qed.cu -- QED tables (built on the host in FP64 from Eqs. (23), (24)),
// the table-evaluation entry points, and the kernels that append emitted
// photons and created pairs to their species.
//
// Tables.  The Bessel functions enter only through K_{2/3}(y) and
// Int_y^inf K_{1/3}; both are tabulated once on a fine logarithmic y grid
// from their integral representations
//   K_nu(y) = Int_0^inf exp(-y cosh t) cosh(nu t) dt,
//   Int_y^inf K_{1/3} = Int_0^inf exp(-y cosh t) cosh(t/3) / cosh t dt,
// and interpolated (cubic in ln y).  For every chi of the table grid the
// spectrum is integrated cumulatively on a fine grid of s = fraction^(1/3)
// (removing the u^{-2/3} behaviour of Eq. (23) at small u), giving the
// total G(chi) and, by inverse interpolation, the inverse CDF.
#include <cmath>
#include <mutex>
#include <vector>

#include "qed.cuh"
#include "qed_host.cuh"
#include <type_traits>

#include "scan_dev.cuh"
#include "sort.cuh"

namespace pic {

namespace {

constexpr int kNchi = 256;
constexpr double kChiMin = 1e-4, kChiMax = 1e3;
constexpr int kNr = 512;
constexpr int kNs = 4096;
constexpr int kNy = 8001;
constexpr double kYmin = 1e-10, kYmax = 700.0;

// ln K + y is tabulated (not ln K): K ~ exp(-y) at large y, and ln K + y is
// smooth in ln y over the whole range
struct BesselTable {
    double lny0, dlny;
    std::vector<double> lnk23, lnik13;  // ln K_{2/3}(y) + y, ln Int_y K_{1/3} + y
};

double trap_bessel(double nu, double y, bool over_cosh)
{
    // exp(-y cosh t) falls below e^-800 at t_max; the integrand is analytic
    // in a strip, so the trapezoid rule converges exponentially in 1/h
    const double tmax = std::acosh(std::max(800.0 / y, 1.0)) + 0.5;
    const int n = std::max(64, (int)std::ceil(tmax / 0.04));
    const double h = tmax / n;
    double s = 0.0;
    for (int i = 0; i <= n; i++) {
        const double t = i * h, ch = std::cosh(t);
        double f = std::exp(-y * ch) * std::cosh(nu * t);
        if (over_cosh) f /= ch;
        s += (i == 0 || i == n) ? 0.5 * f : f;
    }
    return s * h;
}

const BesselTable &bessel_table()
{
    static BesselTable B;
    static std::once_flag once;
    std::call_once(once, [] {
        B.lny0 = std::log(kYmin);
        B.dlny = (std::log(kYmax) - B.lny0) / (kNy - 1);
        B.lnk23.resize(kNy);
        B.lnik13.resize(kNy);
        for (int i = 0; i < kNy; i++) {
            const double y = std::exp(B.lny0 + i * B.dlny);
            B.lnk23[i] = std::log(trap_bessel(2.0 / 3.0, y, false)) + y;
            B.lnik13[i] = std::log(trap_bessel(1.0 / 3.0, y, true)) + y;
        }
    });
    return B;
}

// the host view of the Bessel table in the layout the device reads
QedTables bessel_view()
{
    const BesselTable &B = bessel_table();
    QedTables T{};
    T.bes_k23 = B.lnk23.data();
    T.bes_ik13 = B.lnik13.data();
    T.nbes = kNy;
    T.bes_lny0 = B.lny0;
    T.bes_dlny = B.dlny;
    T.bes_ymin = kYmin;
    T.bes_ymax = kYmax;
    return T;
}

// K_{2/3}(y) and Int_y^inf K_{1/3}: the same evaluation the device makes
// (qed_bessel: below the table the leading small-argument behaviour, exact
// to O(y^{4/3}); zero beyond kYmax)
void bessel(double y, double &k23, double &ik13)
{
    static const QedTables T = bessel_view();
    qed_bessel(T, y, k23, ik13);
}

// Eq. (23): ((1-u) + 1/(1-u)) K_{2/3}(y) - Int_y^inf K_{1/3}, y = 2u / (3 chi (1-u))
double spec_rad(double u, double chi)
{
    if (u <= 0.0 || u >= 1.0) return 0.0;
    double k, ik;
    bessel(2.0 * u / (3.0 * chi * (1.0 - u)), k, ik);
    return ((1.0 - u) + 1.0 / (1.0 - u)) * k - ik;
}

// Eq. (24): ((v^2 + (1-v)^2) / (v (1-v))) K_{2/3}(y) + Int_y^inf K_{1/3}, y = 2 / (3 chi v (1-v))
double spec_pair(double v, double chi)
{
    if (v <= 0.0 || v >= 1.0) return 0.0;
    double k, ik;
    bessel(2.0 / (3.0 * chi * v * (1.0 - v)), k, ik);
    return ((v * v + (1.0 - v) * (1.0 - v)) / (v * (1.0 - v))) * k + ik;
}

struct HostTables {
    std::vector<double> lnG[2], inv[2];
};

// Cumulative integral of a spectrum on a grid of fractions f_k, built from
// cells in a local variable where the integrand is smooth:
//   emission, f <= 1/2: f = s^3 (the u^{-2/3} behaviour at small u);
//   emission, f >= 1/2: 1 - f = t^3 (the (1-u)^{-1/3} peak of width ~1/(3 chi)
//     below u = 1 at large chi);
//   pairs, f <= 1/2: f = t^3 (v^{-1/3} above the cut-off at large chi).
// Two-point Gauss per cell.  f[k] increases; C[k] = Int_0^{f_k} F.
void cumulate(int p, double chi, std::vector<double> &f, std::vector<double> &C)
{
    const int n = p == QED_RAD ? 2 * kNs : kNs;
    f.assign(n + 1, 0.0);
    C.assign(n + 1, 0.0);
    const double g = 0.5 / std::sqrt(3.0), w_half = std::cbrt(0.5);
    const double h = w_half / kNs;
    for (int k = 0; k < n; k++) {
        double acc = 0.0;
        for (int q = 0; q < 2; q++) {
            const double z = (q ? g : -g);
            if (p == QED_PAIR || k < kNs) {  // f = w^3, w in [0, (1/2)^(1/3)]
                const double w = (k + 0.5 + z) * h, fr = w * w * w;
                acc += 3.0 * w * w * (p == QED_RAD ? spec_rad(fr, chi) : spec_pair(fr, chi));
            } else {  // 1 - f = t^3, t from (1/2)^(1/3) down to 0
                const double t = w_half - (k - kNs + 0.5 + z) * h, fr = 1.0 - t * t * t;
                acc += 3.0 * t * t * spec_rad(fr, chi);
            }
        }
        C[k + 1] = C[k] + 0.5 * h * acc;
        if (p == QED_PAIR || k < kNs) {
            const double w = (k + 1) * h;
            f[k + 1] = w * w * w;
        } else {
            const double t = w_half - (k + 1 - kNs) * h;
            f[k + 1] = 1.0 - t * t * t;
        }
    }
    if (p == QED_RAD) f[n] = 1.0;
    else f[n] = 0.5;
}

const HostTables &host_tables()
{
    static HostTables H;
    static std::once_flag once;
    std::call_once(once, [] {
        std::vector<double> f, C;
        for (int p = 0; p < 2; p++) {
            H.lnG[p].resize(kNchi);
            H.inv[p].resize((size_t)kNchi * kNr);
        }
        const double lc0 = std::log(kChiMin), dlc = (std::log(kChiMax) - lc0) / (kNchi - 1);
        for (int i = 0; i < kNchi; i++) {
            const double chi = std::exp(lc0 + i * dlc);
            for (int p = 0; p < 2; p++) {
                cumulate(p, chi, f, C);
                const int n = (int)C.size() - 1;
                const double tot = C[n];
                const double G = p == QED_RAD ? tot : 2.0 * tot;  // pairs: symmetric about v = 1/2
                // pairs: ln G + 8/(3 chi) (the exponential small-chi factor removed);
                // underflowed nodes are filled below by linear extrapolation
                H.lnG[p][i] = G > 1e-300 ? std::log(G) + (p == QED_PAIR ? 8.0 / (3.0 * chi) : 0.0) : NAN;
                int k = 0;
                for (int j = 0; j < kNr; j++) {
                    // r grids dense where the inverse is singular: near r = 1
                    // for emission (the high-energy tail), near r = 0 for pairs
                    const double tj = (double)j / (kNr - 1);
                    const double rj = p == QED_RAD ? 1.0 - (1.0 - tj) * (1.0 - tj) : 0.5 * tj * tj;
                    const double target = rj * G;
                    double fr;
                    if (!(tot > 0.0)) fr = f[n] * j / (kNr - 1);
                    else if (j == kNr - 1) fr = f[n];
                    else {
                        while (k < n - 1 && C[k + 1] < target) k++;
                        const double dC = C[k + 1] - C[k];
                        const double a = std::min(std::max(dC > 0.0 ? (target - C[k]) / dC : 0.0, 0.0), 1.0);
                        // interpolate in the cell's local variable, as integrated
                        if (p == QED_PAIR || k < kNs) {
                            const double w0 = std::cbrt(f[k]), w1 = std::cbrt(f[k + 1]), w = w0 + a * (w1 - w0);
                            fr = w * w * w;
                        } else {
                            const double t0 = std::cbrt(1.0 - f[k]), t1 = std::cbrt(1.0 - f[k + 1]);
                            const double t = t0 + a * (t1 - t0);
                            fr = 1.0 - t * t * t;
                        }
                    }
                    H.inv[p][(size_t)i * kNr + j] = std::cbrt(fr);
                }
            }
        }
        for (int p = 0; p < 2; p++) {
            int first = 0;
            while (first < kNchi - 1 && std::isnan(H.lnG[p][first])) first++;
            for (int i = first - 1; i >= 0; i--) H.lnG[p][i] = 2.0 * H.lnG[p][i + 1] - H.lnG[p][i + 2];
        }
    });
    return H;
}

}  // namespace

void qed_spectra(int p, double frac, double chi, double *F) { *F = p == QED_RAD ? spec_rad(frac, chi) : spec_pair(frac, chi); }

size_t qed_table_bytes()
{
    return 2 * ((size_t)kNchi + (size_t)kNchi * kNr) * (sizeof(float) + sizeof(double)) + 2 * (size_t)kNy * 8;
}

// fill a device buffer (qed_table_bytes) and the table view pointing into it
int qed_upload_tables(void *dev, QedTables *T, cudaStream_t st)
{
    const HostTables &H = host_tables();
    std::vector<float> hf;
    std::vector<double> hd;
    for (int p = 0; p < 2; p++) {
        hd.insert(hd.end(), H.lnG[p].begin(), H.lnG[p].end());
        hd.insert(hd.end(), H.inv[p].begin(), H.inv[p].end());
    }
    hf.assign(hd.begin(), hd.end());
    char *base = (char *)dev;
    if (cudaMemcpyAsync(base, hd.data(), hd.size() * 8, cudaMemcpyHostToDevice, st) != cudaSuccess) return -1;
    if (cudaMemcpyAsync(base + hd.size() * 8, hf.data(), hf.size() * 4, cudaMemcpyHostToDevice, st) != cudaSuccess)
        return -1;
    if (cudaStreamSynchronize(st) != cudaSuccess) return -1;
    // the Bessel table after the rate and inverse-CDF tables
    const BesselTable &B = bessel_table();
    char *bes = base + hd.size() * 8 + hf.size() * 4;
    if (cudaMemcpyAsync(bes, B.lnk23.data(), (size_t)kNy * 8, cudaMemcpyHostToDevice, st) != cudaSuccess) return -1;
    if (cudaMemcpyAsync(bes + (size_t)kNy * 8, B.lnik13.data(), (size_t)kNy * 8, cudaMemcpyHostToDevice, st) !=
        cudaSuccess)
        return -1;
    if (cudaStreamSynchronize(st) != cudaSuccess) return -1;
    const double *d = (const double *)base;
    const float *f = (const float *)(base + hd.size() * 8);
    size_t off = 0;
    for (int p = 0; p < 2; p++) {
        T->lnG_d[p] = d + off;
        T->lnG_f[p] = f + off;
        off += kNchi;
        T->inv_d[p] = d + off;
        T->inv_f[p] = f + off;
        off += (size_t)kNchi * kNr;
    }
    T->nchi = kNchi;
    T->nr = kNr;
    T->bes_k23 = (const double *)bes;
    T->bes_ik13 = (const double *)bes + kNy;
    T->nbes = kNy;
    T->bes_lny0 = B.lny0;
    T->bes_dlny = B.dlny;
    T->bes_ymin = kYmin;
    T->bes_ymax = kYmax;
    T->lnchi0 = std::log(kChiMin);
    T->dlnchi = (std::log(kChiMax) - T->lnchi0) / (kNchi - 1);
    T->lnchi0_f = (float)T->lnchi0;
    T->inv_dlnchi_f = (float)(1.0 / T->dlnchi);
    return 0;
}

// ---------------------------------------------------------------------
// table evaluation (inspection entry points)
// ---------------------------------------------------------------------
template <typename R>
__global__ void k_qed_eval(QedTables T, int p, long long n, const double *chi, const double *r, double *out)
{
    long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    if constexpr (sizeof(R) == 4)  // the FP32 form's own FP32 arithmetic, as its pushes evaluate it
        out[i] = r ? (double)qed_sample_f32(T, p, (float)chi[i], (float)r[i]) : (double)qed_rate_f32(T, p, (float)chi[i]);
    else
        out[i] = r ? qed_sample<R>(T, p, chi[i], r[i]) : qed_rate<R>(T, p, chi[i]);
}

void launch_qed_eval(const QedTables &T, bool f64, int p, long long n, const double *chi, const double *r, double *out,
                     cudaStream_t st)
{
    if (n <= 0) return;
    note_launch();
    if (f64) k_qed_eval<double><<<div_up(n, 256), 256, 0, st>>>(T, p, n, chi, r, out);
    else k_qed_eval<float><<<div_up(n, 256), 256, 0, st>>>(T, p, n, chi, r, out);
}

// ---------------------------------------------------------------------
// spawning: the events of a species are ranked in array order and the
// children appended at the end of their species (deterministic order: the
// pairs, then each emitting species' photons).  One kernel sums the flags of
// blocks of kScanItems of every source; its last block to arrive scans the
// sums, reserves the children's places and moves the counts.  The spawn kernel
// strides over the blocks of flags: a block whose scanned sums show no event
// is skipped without reading its flags; otherwise its events are listed in
// array order in shared memory and taken one per thread.  (Two launches a
// step: two an emitting species took 38 us of a 120 us step of the cascade of
// 2000 replicas, all of it latency, now 17.)
// ---------------------------------------------------------------------
constexpr int kSpawnThreads = 256, kSpawnPer = kScanItems / kSpawnThreads;

inline int spawn_grid(long long m)
{
    static int nsm = 0;
    if (!nsm) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    }
    return (int)std::min<long long>((m + kScanItems - 1) / kScanItems, 4ll * nsm);
}

// this thread's kSpawnPer flags (0 or 1) of block b from p0 as a bit mask;
// m: the flags' end (the parents' device count: what lies past it is no event)
__device__ __forceinline__ uint32_t flag_bits(const uint32_t *__restrict__ ev, long long m, long long p0)
{
    uint32_t bits = 0;
    if (p0 + kSpawnPer <= m && (reinterpret_cast<uintptr_t>(ev) & 15u) == 0) {
#pragma unroll
        for (int k = 0; k < kSpawnPer; k += 4) {
            const uint4 v = *reinterpret_cast<const uint4 *>(ev + p0 + k);
            bits |= (v.x ? 1u : 0u) << k | (v.y ? 2u : 0u) << k | (v.z ? 4u : 0u) << k | (v.w ? 8u : 0u) << k;
        }
    } else {
#pragma unroll
        for (int k = 0; k < kSpawnPer; k++)
            if (p0 + k < m && ev[p0 + k]) bits |= 1u << k;
    }
    return bits;
}

// Source blockIdx.y: bsum[b] = events before block b, bsum[nb] = all of them;
// then, source by source, the flags that were summed (ctl.m), the children's
// first places (ctl.base; two target species for pairs) and the new counts.  A
// pair is created only where both its electron and its positron find room, so
// both counts advance by the same number.
template <class P_t>
__global__ void __launch_bounds__(kSpawnThreads) k_flag_sums(const __grid_constant__ SpawnSet<P_t> S)
{
    __shared__ uint32_t sh[32];
    __shared__ bool last;
    {
        const SpawnSource<P_t> &src = S.src[blockIdx.y];
        uint32_t *bsum = src.bsum;
        const long long m = max(0ll, min(src.p.n, *src.p.dn));
        const long long nb = (m + kScanItems - 1) / kScanItems;
        for (long long b = blockIdx.x; b < nb; b += gridDim.x) {
            const uint32_t bits = flag_bits(src.ev, m, b * kScanItems + (long long)threadIdx.x * kSpawnPer);
            uint32_t tot;
            block_excl_scan<kSpawnThreads>((uint32_t)__popc(bits), sh, tot);
            if (threadIdx.x == 0) bsum[b] = tot;
        }
    }
    // (all of the block has read its source's count: the last block moves it)
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        last = atomicAdd(&S.ctl->done, 1u) == gridDim.x * gridDim.y - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    uint32_t total[kSpawnSources];
#pragma unroll
    for (int q = 0; q < kSpawnSources; q++) {
        if (q >= S.n) break;
        uint32_t *bsum = S.src[q].bsum;
        const long long m = max(0ll, min(S.src[q].p.n, *S.src[q].p.dn));
        const long long nb = (m + kScanItems - 1) / kScanItems;
        uint32_t carry = 0;
        for (long long b0 = 0; b0 < nb; b0 += kSpawnThreads * 8) {
            uint32_t v[8], s = 0, tot;
            const long long i0 = b0 + threadIdx.x * 8;
#pragma unroll
            for (int k = 0; k < 8; k++) {
                v[k] = i0 + k < nb ? __ldcg(bsum + i0 + k) : 0u;
                s += v[k];
            }
            uint32_t run = carry + block_excl_scan<kSpawnThreads>(s, sh, tot);
#pragma unroll
            for (int k = 0; k < 8; k++) {
                if (i0 + k < nb) bsum[i0 + k] = run;
                run += v[k];
            }
            carry += tot;
        }
        total[q] = carry;
        if (threadIdx.x == 0) {
            bsum[nb] = carry;
            S.ctl->m[q] = m;  // (before any count moves)
        }
    }
    // (a source without a particle has no barrier in its scan: a warp that read
    // its count after thread 0 moved it would scan alone)
    __syncthreads();
    if (threadIdx.x != 0) return;
#pragma unroll
    for (int q = 0; q < kSpawnSources; q++) {
        if (q >= S.n) break;
        const bool pair = q == 0 && S.pairs;
        const SpawnTarget<P_t> &a = pair ? S.el : S.ph;
        const long long n = total[q], n0 = *a.count;
        S.ctl->base[q][0] = n0;
        bool over = n0 + n > a.cap;
        long long take = min(n, a.cap - n0);
        if (pair) {
            const long long n1 = *S.po.count;
            S.ctl->base[q][1] = n1;
            over |= n1 + n > S.po.cap;
            take = min(take, S.po.cap - n1);
        }
        if (over) atomicOr(S.err, ERR_CAPACITY);
        take = max(take, 0ll);
        *a.count += take;
        if (pair) *S.po.count += take;
    }
    S.ctl->done = 0u;
}

// the events of block b listed in array order (their places in the block);
// returns their number (block-uniform)
__device__ __forceinline__ int list_events(const uint32_t *__restrict__ ev, long long m,
                                           const uint32_t *__restrict__ bsum, long long b, uint16_t *list)
{
    __shared__ uint32_t sh[32];
    if (bsum[b + 1] == bsum[b]) return 0;
    __syncthreads();  // (the list of the block before is done with)
    uint32_t bits = flag_bits(ev, m, b * kScanItems + (long long)threadIdx.x * kSpawnPer), tot;
    uint32_t run = block_excl_scan<kSpawnThreads>((uint32_t)__popc(bits), sh, tot);
    for (; bits; bits &= bits - 1) list[run++] = (uint16_t)(threadIdx.x * kSpawnPer + __ffs(bits) - 1);
    __syncthreads();
    return (int)tot;
}

// The photon emitted by particle p of src: its event data, at the parent's
// x^{n+1}; FP32 event data are 4 floats per particle, FP64 4 doubles.
template <class P_t>
__device__ __forceinline__ void spawn_photon(const SpawnSet<P_t> &S, const SpawnSource<P_t> &src, long long p,
                                             long long dst)
{
    const P_t &parent = src.p, &ph = S.ph.p;
    uint32_t w[4];
    const uint64_t pid = src.p.id[p];
    philox4x32_10((uint32_t)pid, (uint32_t)(pid >> 32), S.step, QP_EMIT, S.key[0], S.key[1], w);
    const uint64_t cid = ((uint64_t)w[3] << 32) | w[2];
    ph.cell[dst] = parent.cell[p];
    if constexpr (std::is_same_v<P_t, PartF32>) {
        const float *evk = reinterpret_cast<const float *>(src.evk);
#pragma unroll
        for (int d = 0; d < 3; d++)
            if (d < S.dim) ph.off[d][dst] = parent.off[d][p];
        ph.u[0][dst] = evk[4 * p];
        ph.u[1][dst] = evk[4 * p + 1];
        ph.u[2][dst] = evk[4 * p + 2];
        ph.tau[dst] = initial_tau_f32(cid, S.key);
    } else {
        const double4 ed = reinterpret_cast<const double4 *>(src.evk)[p];
#pragma unroll
        for (int d = 0; d < 3; d++)
            if (d < S.dim) ph.x[d][dst] = parent.x[d][p];
        ph.u[0][dst] = ed.x;
        ph.u[1][dst] = ed.y;
        ph.u[2][dst] = ed.z;
        ph.tau[dst] = initial_tau(cid, S.key);
    }
    ph.id[dst] = cid;
    S.ph.ev[dst] = 0;
}

// The pair of photon p of src (event data: its momentum k and the positron
// fraction v), born where the photon converted (its x^{n+1}); the photon dies.
template <class P_t>
__device__ __forceinline__ void spawn_pair(const SpawnSet<P_t> &S, const SpawnSource<P_t> &src, long long p, long long de,
                                           long long dp)
{
    const P_t &phot = src.p, &el = S.el.p, &po = S.po.p;
    uint32_t w[4];
    const uint64_t pid = src.p.id[p];
    philox4x32_10((uint32_t)pid, (uint32_t)(pid >> 32), S.step, QP_PAIR, S.key[0], S.key[1], w);
    const uint64_t eid = ((uint64_t)w[3] << 32) | w[2], pid2 = eid + 1;
    double kx, ky, kz, v;
    if constexpr (std::is_same_v<P_t, PartF32>) {
        const float *evk = reinterpret_cast<const float *>(src.evk);
        kx = evk[4 * p], ky = evk[4 * p + 1], kz = evk[4 * p + 2], v = evk[4 * p + 3];
#pragma unroll
        for (int d = 0; d < 3; d++) {
            if (d >= S.dim) break;
            el.off[d][de] = phot.off[d][p];
            po.off[d][dp] = phot.off[d][p];
        }
    } else {
        const double4 ed = reinterpret_cast<const double4 *>(src.evk)[p];
        kx = ed.x, ky = ed.y, kz = ed.z, v = ed.w;
#pragma unroll
        for (int d = 0; d < 3; d++) {
            if (d >= S.dim) break;
            el.x[d][de] = phot.x[d][p];
            po.x[d][dp] = phot.x[d][p];
        }
    }
    const double k = sqrt(kx * kx + ky * ky + kz * kz);
    const uint32_t cell = phot.cell[p];
    el.cell[de] = cell;
    po.cell[dp] = cell;
    phot.cell[p] = kDead;
    const double ep = v * k, em = (1.0 - v) * k;  // eps_+ and eps_- (m c^2)
    const double pm = sqrt(fmax(em * em - 1.0, 0.0)), pp = sqrt(fmax(ep * ep - 1.0, 0.0));
    const double inv = k > 0.0 ? 1.0 / k : 0.0;
    using R = std::remove_reference_t<decltype(*el.u[0])>;
    el.u[0][de] = (R)(pm * kx * inv);
    el.u[1][de] = (R)(pm * ky * inv);
    el.u[2][de] = (R)(pm * kz * inv);
    po.u[0][dp] = (R)(pp * kx * inv);
    po.u[1][dp] = (R)(pp * ky * inv);
    po.u[2][dp] = (R)(pp * kz * inv);
    el.id[de] = eid;
    po.id[dp] = pid2;
    if constexpr (std::is_same_v<P_t, PartF32>) {
        el.tau[de] = initial_tau_f32(eid, S.key);
        po.tau[dp] = initial_tau_f32(pid2, S.key);
    } else {
        el.tau[de] = initial_tau(eid, S.key);
        po.tau[dp] = initial_tau(pid2, S.key);
    }
    S.el.ev[de] = 0;
    S.po.ev[dp] = 0;
}

// source blockIdx.y; the children land past every source's summed flags, so
// the sources do not meet
template <class P_t>
__global__ void __launch_bounds__(kSpawnThreads) k_spawn(const __grid_constant__ SpawnSet<P_t> S)
{
    __shared__ uint16_t list[kScanItems];
    const int k = blockIdx.y;
    const SpawnSource<P_t> &src = S.src[k];
    const bool pair = k == 0 && S.pairs;
    const long long m = S.ctl->m[k], base = S.ctl->base[k][0], base1 = pair ? S.ctl->base[k][1] : 0;
    const long long nb = (m + kScanItems - 1) / kScanItems;
    for (long long b = blockIdx.x; b < nb; b += gridDim.x) {
        const int n = list_events(src.ev, m, src.bsum, b, list);
        for (int e = threadIdx.x; e < n; e += kSpawnThreads) {
            const long long p = b * kScanItems + list[e];
            const uint32_t rank = src.bsum[b] + e;
            if (pair) {
                if (base + rank < S.el.cap && base1 + rank < S.po.cap) spawn_pair(S, src, p, base + rank, base1 + rank);
            } else if (base + rank < S.ph.cap) {
                spawn_photon(S, src, p, base + rank);
            }
        }
    }
}

__global__ void k_init_qed(long long first, long long n, uint64_t id0, uint64_t *id, double *tau, uint32_t k0,
                           uint32_t k1)
{
    const long long a = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (a >= n) return;
    const uint64_t v = id0 + (uint64_t)(first + a);
    id[first + a] = v;
    const uint32_t key[2] = {k0, k1};
    tau[first + a] = initial_tau(v, key);
}

void launch_init_qed(long long first, long long n, uint64_t id0, uint64_t *id, double *tau, const uint32_t *key,
                     cudaStream_t st)
{
    if (n <= 0) return;
    note_launch();
    k_init_qed<<<div_up(n, 256), 256, 0, st>>>(first, n, id0, id, tau, key[0], key[1]);
}

template <class P_t>
void launch_spawn(SpawnSet<P_t> &S, uint32_t *scratch, cudaStream_t st)
{
    if (S.n == 0) return;
    long long most = 0;
    for (int k = 0; k < S.n; k++) {
        S.src[k].bsum = scratch;
        scratch += (S.src[k].p.n + kScanItems - 1) / kScanItems + 1;
        most = std::max(most, S.src[k].p.n);
    }
    const dim3 grid(spawn_grid(most), S.n);
    note_launch(2);
    k_flag_sums<P_t><<<grid, kSpawnThreads, 0, st>>>(S);
    k_spawn<P_t><<<grid, kSpawnThreads, 0, st>>>(S);
}
template void launch_spawn<PartF32>(SpawnSet<PartF32> &, uint32_t *, cudaStream_t);
template void launch_spawn<PartF64>(SpawnSet<PartF64> &, uint32_t *, cudaStream_t);

}  // namespace pic
