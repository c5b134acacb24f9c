// push_tile.cuh -- the tiled pushes (push_tile2d.cu, push_tile3d.cu; of the QED
// species push_tile.cu, push_qed_tile3d.cu) and their work items (push_tile.cu).
#pragma once
#include "push.cuh"
#include "sort.cuh"

namespace pic {

struct QedParams;

constexpr int kChunkMax = 1024;    // particles per work item at most (2D)
constexpr int kPushThreads = 256;  // threads per CTA of the 2D push (tiles of 8 x 8 cells: 128 on large grids)
constexpr int kChunk = 384;        // particles per work item at most (2D, QED species)
constexpr int kTileThreads = 128;  // threads per CTA of the QED species' pushes and the 3D push
constexpr int kTileMinBlocks = 6;  // CTAs per SM of the 2D QED pushes: 80 registers, 35 KB shared memory each (measured best)

struct TileItem {
    int tile, start, count, pad;
};

// 3D items: a 4^3 tile of the 8-ppc thermal workload in one item (512 +- 23
// particles); QED leptons: 256 measured best among 256-1024 on that workload
constexpr int kChunk3Max = 640;
constexpr int kChunk3 = 256;

// particles per work item at most, for n particles of a species on grid g
// (qed: photons and the leptons of the Monte Carlo)
int tile_chunk(const Grid &g, bool qed, long long n);
size_t tile_items_capacity(long long cap, long long ntiles);
// nitems (two words): all items, and those of the tiled push without QED, none
// where there are at most `least` particles an item (0: no such rule; see
// least_of in sim.cuh): the one-thread push runs instead
int tile_least(const Grid &g);
void build_tile_items(const uint32_t *starts, long long ntiles, int chunk, int least, uint32_t *cnt_scratch,
                      uint32_t *scan_scratch, TileItem *items, uint32_t *nitems, cudaStream_t st);
// nitems[1] for items that are there already
void launch_item_counts(const uint32_t *starts, long long ntiles, int least, uint32_t *nitems, cudaStream_t st);
// 2D, shape orders 2 and 4 (agg: the warp-aggregated deposit, order 2); and
// with a QED lepton species' Monte Carlo q fused in (order 2; q.on; the
// particles appended since the sort, and their event flags, are left to
// launch_push_qed_f32)
void launch_push_tile2d(const PartF32 &P, const TileItem *items, const uint32_t *nitems, long long max_items,
                        float *F, const Grid &g, const PushConst &pc, int *err, double *e_abs, cudaStream_t st,
                        bool agg);
void launch_push_qed_tile2d(const PartF32 &P, const TileItem *items, const uint32_t *nitems, long long max_items,
                            float *F, const Grid &g, const PushConst &pc, int *err, double *e_abs, cudaStream_t st,
                            const QedParams &q);
// the tiled photon push (2D, FP32; tiles of 8 or 16 cells): the photons of
// the work items, their pair Monte Carlo with q
void launch_push_photon_tile2d(const PartF32 &P, const TileItem *items, const uint32_t *nitems, long long max_items,
                               const float *F, const Grid &g, const PushConst &pc, const QedParams &q, int *err,
                               cudaStream_t st);
// work items for it over the photons appended since the sort ([*first, *P.dn),
// kChunk each)
size_t tail_items_capacity(long long cap);
void launch_tail_items(const PartF32 &P, const uint32_t *first, const Grid &g, TileItem *items, uint32_t *nitems,
                       cudaStream_t st);
// the surrogate's candidate conversions queued by the tiled photon push (q.cq)
void launch_photon_resolve(const QedParams &q, const PartF32 &P, int *err, cudaStream_t st);
// 3D, tiles of 4^3 cells (defer: a list of capacity >= the particle count,
// ndefer its device count; the particles the tiled kernel defers are pushed
// after it on the global path, with maybe_sparse all of them if *nitems is zero)
bool tile3d_push_supported(const Grid &g);
void launch_push_tile3d(const PartF32 &P, const TileItem *items, const uint32_t *nitems, long long max_items,
                        float *F, const Grid &g, const PushConst &pc, int *err, double *e_abs, uint32_t *defer,
                        uint32_t *ndefer, bool maybe_sparse, cudaStream_t st);
// and with a QED lepton species' Monte Carlo q fused in (q.on; every n_d a
// multiple of 4); nothing is deferred, and the particles appended since the
// sort are left to launch_push_qed_f32
bool tile3d_qed_push_supported(const Grid &g);
void launch_push_qed_tile3d(const PartF32 &P, const TileItem *items, const uint32_t *nitems, long long max_items,
                            float *F, const Grid &g, const PushConst &pc, int *err, double *e_abs, cudaStream_t st,
                            const QedParams &q);

}  // namespace pic
