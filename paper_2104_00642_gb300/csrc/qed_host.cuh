// qed_host.cuh -- host entry points of the QED module (qed.cu).
#pragma once
#include "../../include/pic.h"
#include "push.cuh"
#include "qed.cuh"

namespace pic {

size_t qed_table_bytes();
int qed_upload_tables(void *dev, QedTables *T, cudaStream_t st);
void qed_spectra(int p, double frac, double chi, double *F);
void launch_qed_eval(const QedTables &T, bool f64, int p, long long n, const double *chi, const double *r,
                     double *out, cudaStream_t st);
void launch_init_qed(long long first, long long n, uint64_t id0, uint64_t *id, double *tau, const uint32_t *key,
                     cudaStream_t st);
// A step's children.  Sources: the converting photons (first, when pairs), then
// the emitting species; targets: the photon species, and the pair's two.
constexpr int kSpawnSources = PIC_MAX_SPECIES;
// device state: the block counter (zero between launches), and per source the
// flags summed and the first place in each target species
struct SpawnCtl {
    unsigned done, pad;
    long long m[kSpawnSources], base[kSpawnSources][2];
};
template <class P_t>
struct SpawnSource {
    P_t p;               // (p.n: the host's bound on the count)
    const uint32_t *ev;  // event flags
    const void *evk;     // event data
    uint32_t *bsum;      // set by launch_spawn
};
template <class P_t>
struct SpawnTarget {
    P_t p;
    uint32_t *ev;
    long long *count, cap;
};
template <class P_t>
struct SpawnSet {
    int n, pairs, dim;
    uint32_t key[2], step;
    SpawnCtl *ctl;
    int *err;
    SpawnTarget<P_t> ph, el, po;
    SpawnSource<P_t> src[kSpawnSources];
};
// the children of the flagged particles, appended in the sources' order and in
// array order; scratch: a word for each kScanItems flags and one more per source
template <class P_t>
void launch_spawn(SpawnSet<P_t> &S, uint32_t *scratch, cudaStream_t st);
void launch_push_qed_f64(const PartF64 &P, double *F, const Grid &g, const PushConst &pc, const QedParams &q,
                         int *err, double *e_abs, cudaStream_t st);
void launch_push_photon_f64(const PartF64 &P, const double *F, const Grid &g, const PushConst &pc,
                            const QedParams &q, int *err, cudaStream_t st);
// one species' one-thread-per-particle push with QED (photon: launch_push_photon_f32)
struct QedPush {
    PartF32 P;
    PushConst pc;
    QedParams q;
    const uint32_t *first;
    int photon, nb;  // nb: set by the launch
};
// the pushes of several species (none with a network) in one launch
void launch_push_qed_set(QedPush *p, int n, float *F, const Grid &g, int *err, double *e_abs, cudaStream_t st);
// The pushes with a network (q.on, q.net).
// (first: see k_push_qed_f32 -- nullptr pushes every particle)
void launch_push_qed_f32(const PartF32 &P, float *F, const Grid &g, const PushConst &pc, const QedParams &q,
                         int *err, double *e_abs, cudaStream_t st, const uint32_t *first = nullptr);
// (tc: evaluate the pair network per CTA on the tcgen05 tensor cores instead
// of per warp with mma.sync)
void launch_push_photon_f32(const PartF32 &P, const float *F, const Grid &g, const PushConst &pc,
                            const QedParams &q, int *err, cudaStream_t st, bool tc);

}  // namespace pic
