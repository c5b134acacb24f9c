// sort.cu -- stable counting sort of particles by tile (the tile holding a
// particle's cell) and, inside a tile, by cell (row-major within the tile),
// dead particles last, and the per-tile start offsets.  Cell order inside a
// tile puts the particles of one cell next to each other, so the lanes of a
// warp in the tiled push read the same field nodes and deposit into the
// same window.
//
// The sort is a least-significant-digit radix sort of (tile key, index)
// pairs with 8-bit digits.  Each pass is reduce-then-scan: per-block digit
// histograms (4096 keys per block; the first digit's come with the keys), one
// device-wide exclusive scan of the (digit, block) counts, then a scatter in
// which every warp ranks its 512 consecutive keys by itself (match masks and a
// per-warp digit counter), the warps' counters are prefixed once, and the keys
// are written.  Every pass is stable, so the final permutation is the one a
// stable sort by key gives, independent of scheduling.
//
// Every kernel stops at the device's particle count: the host's bound on it
// grows with every step that can create particles, and the slots between the
// two hold nothing.
#include <utility>

#include "scan_dev.cuh"
#include "sort.cuh"

namespace pic {

constexpr int kSortThreads = 256;
constexpr int kSortRounds = 16;
constexpr int kSortItems = kSortThreads * kSortRounds;  // keys per block
constexpr int kSortWarps = kSortThreads / 32;

// the keys, and the histograms of their first digit; *neff: the entries the
// later kernels sort (the device count may change under them)
__global__ void __launch_bounds__(kSortThreads) k_make_keys(const uint32_t *__restrict__ cell,
                                                            const long long *__restrict__ dn, long long n, Grid g,
                                                            uint32_t *key, uint32_t *counts, int nb, long long *neff)
{
    __shared__ uint32_t h[256];
    h[threadIdx.x] = 0;
    const long long live = min(n, *dn);
    if (blockIdx.x == 0 && threadIdx.x == 0) *neff = live;
    __syncthreads();
    const int lb = g.tile_log2[0] + g.tile_log2[1] + g.tile_log2[2];  // bits of the cell within a tile
    const long long start = (long long)blockIdx.x * kSortItems + threadIdx.x;
#pragma unroll 4
    for (int r = 0; r < kSortRounds; r++) {
        const long long i = start + r * kSortThreads;
        if (i >= live) break;
        const uint32_t c = cell[i];
        uint32_t k;
        if (c == kDead) k = (uint32_t)g.ntiles << lb;
        else {
            int a, b, d;
            unpack_cell(g, c, a, b, d);
            const uint32_t local = (uint32_t)(a & ((1 << g.tile_log2[0]) - 1)) |
                                   ((uint32_t)(b & ((1 << g.tile_log2[1]) - 1)) << g.tile_log2[0]) |
                                   ((uint32_t)(d & ((1 << g.tile_log2[2]) - 1)) << (g.tile_log2[0] + g.tile_log2[1]));
            k = (tile_of(g, a, b, d) << lb) | local;
        }
        key[i] = k;
        atomicAdd(&h[k & 255u], 1u);
    }
    __syncthreads();
    counts[(long long)threadIdx.x * nb + blockIdx.x] = h[threadIdx.x];
}

__global__ void __launch_bounds__(kSortThreads) k_radix_hist(const uint32_t *__restrict__ kin,
                                                            const long long *__restrict__ neff, int shift,
                                                            uint32_t *counts, int nb)
{
    __shared__ uint32_t h[256];
    const int tid = threadIdx.x;
    h[tid] = 0;
    const long long n = *neff;
    __syncthreads();
    const long long start = (long long)blockIdx.x * kSortItems + tid;
#pragma unroll 4
    for (int r = 0; r < kSortRounds; r++) {
        const long long i = start + r * kSortThreads;
        if (i < n) atomicAdd(&h[(kin[i] >> shift) & 255u], 1u);
    }
    __syncthreads();
    counts[(long long)tid * nb + blockIdx.x] = h[tid];
}

// FIRST: the values are the indices (the keys' own pass writes none).  The
// block's pairs are put in digit order in shared memory and leave as runs of
// one digit, 16 pairs on average: writing each from where it was ranked
// touched a sector per pair (213 us for the first pass over 16.8 million
// particles, now 134).
template <bool FIRST>
__global__ void __launch_bounds__(kSortThreads, 4) k_radix_scatter(const uint32_t *__restrict__ kin,
                                                                      const uint32_t *__restrict__ vin, uint32_t *kout,
                                                                      uint32_t *vout, const long long *__restrict__ neff,
                                                                      int shift, const uint32_t *__restrict__ offs, int nb)
{
    __shared__ uint32_t wc[kSortWarps][256];  // per warp: digit counts, then first local place of each digit
    __shared__ uint32_t place[256];           // global place of a digit's run less its local one
    __shared__ uint32_t sk[kSortItems], sv[kSortItems];
    __shared__ uint32_t sh[32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const long long n = *neff, b0 = (long long)blockIdx.x * kSortItems;
    if (b0 >= n) return;
    const int cnt = (int)min((long long)kSortItems, n - b0);
#pragma unroll
    for (int w = 0; w < kSortWarps; w++) wc[w][tid] = 0;
    const int l0 = warp * (32 * kSortRounds) + lane;  // this thread's first entry of the block
    const unsigned lt = (1u << lane) - 1u;
    uint32_t k[kSortRounds];
    uint32_t rank[kSortRounds / 2];  // two 16-bit ranks (below 512) a word
#pragma unroll
    for (int r = 0; r < kSortRounds; r++) k[r] = l0 + 32 * r < cnt ? kin[b0 + l0 + 32 * r] : 0xffffffffu;
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kSortRounds; r++) {
        const uint32_t dg = (k[r] >> shift) & 255u;
        const bool valid = l0 + 32 * r < cnt;  // (the invalid lanes match among themselves)
        const unsigned peers = __match_any_sync(0xffffffffu, valid ? dg : 256u);
        const uint32_t before = valid ? wc[warp][dg] : 0u, mine = before + __popc(peers & lt);
        rank[r / 2] = r & 1 ? rank[r / 2] | mine << 16 : mine;
        __syncwarp();
        if (valid && lane == __ffs(peers) - 1) wc[warp][dg] = before + __popc(peers);
        __syncwarp();
    }
    __syncthreads();
    // digit tid: the block's count, its local start, the warps' starts in it
    uint32_t c[kSortWarps], sum = 0, tot;
#pragma unroll
    for (int w = 0; w < kSortWarps; w++) {
        c[w] = wc[w][tid];
        sum += c[w];
    }
    uint32_t run = block_excl_scan<kSortThreads>(sum, sh, tot);
    place[tid] = offs[(long long)tid * nb + blockIdx.x] - run;
#pragma unroll
    for (int w = 0; w < kSortWarps; w++) {
        wc[w][tid] = run;
        run += c[w];
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kSortRounds; r++) {
        const int l = l0 + 32 * r;
        if (l >= cnt) continue;
        const uint32_t at = wc[warp][(k[r] >> shift) & 255u] + ((rank[r / 2] >> (16 * (r & 1))) & 0xffffu);
        sk[at] = k[r];
        sv[at] = FIRST ? (uint32_t)(b0 + l) : vin[b0 + l];
    }
    __syncthreads();
    for (int l = tid; l < cnt; l += kSortThreads) {
        const uint32_t key = sk[l], pos = place[(key >> shift) & 255u] + l;
        kout[pos] = key;
        vout[pos] = sv[l];
    }
}

// ---------------------------------------------------------------------
// device-wide exclusive scan of u32 (reduce, scan of block sums, downsweep)
// ---------------------------------------------------------------------
__global__ void __launch_bounds__(1024) k_scan_reduce(const uint32_t *__restrict__ in, long long m, uint32_t *sums)
{
    __shared__ uint32_t sh[32];
    long long b0 = (long long)blockIdx.x * kScanItems + threadIdx.x * 4;
    uint32_t s = 0;
#pragma unroll
    for (int q = 0; q < 4; q++)
        if (b0 + q < m) s += in[b0 + q];
    uint32_t tot;
    block_excl_scan_1024(s, sh, tot);
    if (threadIdx.x == 0) sums[blockIdx.x] = tot;
}

__global__ void __launch_bounds__(1024) k_scan_down(const uint32_t *__restrict__ in, long long m, uint32_t *out,
                                                   const uint32_t *__restrict__ block_off)
{
    __shared__ uint32_t sh[32];
    long long b0 = (long long)blockIdx.x * kScanItems + threadIdx.x * 4;
    uint32_t v[4], s = 0;
#pragma unroll
    for (int q = 0; q < 4; q++) {
        v[q] = b0 + q < m ? in[b0 + q] : 0u;
        s += v[q];
    }
    uint32_t tot;
    uint32_t run = block_excl_scan_1024(s, sh, tot) + (block_off ? block_off[blockIdx.x] : 0u);
#pragma unroll
    for (int q = 0; q < 4; q++) {
        if (b0 + q < m) out[b0 + q] = run;
        run += v[q];
    }
}

size_t scan_scratch_words(long long m)
{
    size_t w = 0;
    while (m > kScanItems) {
        m = (m + kScanItems - 1) / kScanItems;
        w += (size_t)m + 32;
    }
    return w + 32;
}

// exclusive scan of m words, in may equal out
void scan_exclusive(const uint32_t *in, uint32_t *out, long long m, uint32_t *scratch, cudaStream_t st)
{
    if (m <= 0) return;
    if (m <= kScanItems) {
        note_launch();
        k_scan_down<<<1, 1024, 0, st>>>(in, m, out, nullptr);
        return;
    }
    long long nb = (m + kScanItems - 1) / kScanItems;
    uint32_t *sums = scratch;
    note_launch(2);
    k_scan_reduce<<<(int)nb, 1024, 0, st>>>(in, m, sums);
    scan_exclusive(sums, sums, nb, scratch + nb + 32, st);
    k_scan_down<<<(int)nb, 1024, 0, st>>>(in, m, out, sums);
}

// ---------------------------------------------------------------------
// host driver
// ---------------------------------------------------------------------
size_t sort_scratch_bytes(long long cap)
{
    long long nb = (cap + kSortItems - 1) / kSortItems;
    size_t w = 4 * (size_t)cap + 256 * (size_t)nb + scan_scratch_words(256 * nb) + 256;
    return w * sizeof(uint32_t);
}

// 8-bit digits covering the largest key, (ntiles << lb) for the dead
int radix_passes(long long ntiles, int lb)
{
    int bits = 0;
    while ((1ll << bits) <= (ntiles << lb)) bits++;
    return (bits + 7) / 8;
}

// sorts the first n entries (those at or past *dcount hold nothing): keys and
// permutation (new -> old) stay in scratch for sort_apply
SortResult sort_by_tile(const uint32_t *cell, long long n, const long long *dcount, const Grid &g, void *scratch,
                        cudaStream_t st)
{
    uint32_t *w = (uint32_t *)scratch;
    uint32_t *kA = w, *kB = w + n, *vA = w + 2 * n, *vB = w + 3 * n;
    const int nb = (int)((n + kSortItems - 1) / kSortItems);
    uint32_t *counts = w + 4 * n;
    uint32_t *sscr = counts + 256 * (long long)nb + 64;
    long long *neff = reinterpret_cast<long long *>(reinterpret_cast<uintptr_t>(counts + 256 * (long long)nb + 7) & ~uintptr_t(7));
    const int lb = g.tile_log2[0] + g.tile_log2[1] + g.tile_log2[2];
    const int passes = radix_passes(g.ntiles, lb);
    note_launch(2 * passes);
    for (int p = 0; p < passes; p++) {
        if (p == 0) k_make_keys<<<nb, kSortThreads, 0, st>>>(cell, dcount, n, g, kA, counts, nb, neff);
        else k_radix_hist<<<nb, kSortThreads, 0, st>>>(kA, neff, 8 * p, counts, nb);
        scan_exclusive(counts, counts, 256ll * nb, sscr, st);
        if (p == 0) k_radix_scatter<true><<<nb, kSortThreads, 0, st>>>(kA, nullptr, kB, vB, neff, 0, counts, nb);
        else k_radix_scatter<false><<<nb, kSortThreads, 0, st>>>(kA, vA, kB, vB, neff, 8 * p, counts, nb);
        std::swap(kA, kB);
        std::swap(vA, vB);
    }
    return {vA, kA, neff};
}

// ---------------------------------------------------------------------
// apply the permutation to the particle arrays (new[i] = old[perm[i]]), with
// the tile starts and the live count from the sorted keys
// ---------------------------------------------------------------------
// per thread: 2048 outputs a block, mostly from its own tiles' old range, eight
// independent reads at a time (one particle a thread, seven dependent pairs of
// reads: 607 us for 16.8 million particles in 3D, now 220)
constexpr int kPermuteItems = 8;

template <typename T>
__device__ __forceinline__ void move(const T *__restrict__ s, T *__restrict__ d, const uint32_t *from, long long i0,
                                     int cnt)
{
    T v[kPermuteItems];
#pragma unroll
    for (int k = 0; k < kPermuteItems; k++)
        if (k < cnt) v[k] = s[from[k]];
#pragma unroll
    for (int k = 0; k < kPermuteItems; k++)
        if (k < cnt) d[i0 + k * 256] = v[k];
}

__device__ __forceinline__ void move_state(const PartF32 &src, const PartF32 &dst, const uint32_t *from, long long i0,
                                           int cnt, int dim)
{
#pragma unroll
    for (int d = 0; d < 3; d++)
        if (d < dim) move(src.off[d], dst.off[d], from, i0, cnt);
}
__device__ __forceinline__ void move_state(const PartF64 &src, const PartF64 &dst, const uint32_t *from, long long i0,
                                           int cnt, int dim)
{
#pragma unroll
    for (int d = 0; d < 3; d++)
        if (d < dim) move(src.x[d], dst.x[d], from, i0, cnt);
}

template <class P_t>
__global__ void __launch_bounds__(256) k_permute(P_t src, P_t dst, SortResult r, long long ntiles, int lb,
                                                 uint32_t *starts, long long *dcount, int dim)
{
    const long long n = *r.neff;
    const long long i0 = (long long)blockIdx.x * (256 * kPermuteItems) + threadIdx.x;
    uint32_t from[kPermuteItems];
    int cnt = 0;  // this thread's live entries (the dead are sorted last)
#pragma unroll
    for (int k = 0; k < kPermuteItems; k++) {
        const long long i = i0 + k * 256;
        if (i > n) break;
        // entry i starts the tiles after its predecessor's (i == n: all that are left)
        const long long lo = i == 0 ? 0 : (long long)(r.key[i - 1] >> lb) + 1;
        const long long hi = i == n ? ntiles : (long long)(r.key[i] >> lb);
        for (long long t = lo; t <= hi && t <= ntiles; t++) {
            starts[t] = (uint32_t)i;
            if (t == ntiles) *dcount = i;
        }
        if (i < n && hi < ntiles) {
            from[k] = r.perm[i];
            cnt = k + 1;
        }
    }
    move(src.cell, dst.cell, from, i0, cnt);
    move_state(src, dst, from, i0, cnt, dim);
#pragma unroll
    for (int d = 0; d < 3; d++) move(src.u[d], dst.u[d], from, i0, cnt);
    if (src.tau) {
        move(src.tau, dst.tau, from, i0, cnt);
        move(src.id, dst.id, from, i0, cnt);
    }
}

template <class P_t>
void sort_apply(const P_t &src, const P_t &dst, const SortResult &r, long long n, const Grid &g, uint32_t *starts,
                long long *dcount, cudaStream_t st)
{
    const int lb = g.tile_log2[0] + g.tile_log2[1] + g.tile_log2[2];
    note_launch();
    k_permute<<<div_up(n + 1, 256 * kPermuteItems), 256, 0, st>>>(src, dst, r, g.ntiles, lb, starts, dcount, g.dim);
}
template void sort_apply<PartF32>(const PartF32 &, const PartF32 &, const SortResult &, long long, const Grid &,
                                  uint32_t *, long long *, cudaStream_t);
template void sort_apply<PartF64>(const PartF64 &, const PartF64 &, const SortResult &, long long, const Grid &,
                                  uint32_t *, long long *, cudaStream_t);

}  // namespace pic
