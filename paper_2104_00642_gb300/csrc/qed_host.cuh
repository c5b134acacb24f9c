// qed_host.cuh -- host entry points of the QED module (qed.cu).
#pragma once
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
// places of a step's children (k_flag_sums): the block counter (zero between
// launches) and the first place in each target species
struct SpawnCtl {
    unsigned done, pad;
    long long base[2];
};
// the children of the flagged particles (q.ev), appended in array order;
// bsum: scan_blocks(n) + 1 words of scratch
template <class P_t>
void launch_spawn_photons(const P_t &parent, uint32_t *bsum, SpawnCtl *ctl, const QedParams &q, const P_t &ph,
                          uint32_t *ph_ev, long long *ph_count, long long ph_cap, int dim, int *err, cudaStream_t st);
template <class P_t>
void launch_spawn_pairs(const P_t &phot, uint32_t *bsum, SpawnCtl *ctl, const QedParams &q, const P_t &el,
                        uint32_t *el_ev, long long *el_count, long long el_cap, const P_t &po, uint32_t *po_ev,
                        long long *po_count, long long po_cap, int dim, int *err, cudaStream_t st);
void launch_push_qed_f64(const PartF64 &P, double *F, const Grid &g, const PushConst &pc, const QedParams &q,
                         int *err, double *e_abs, cudaStream_t st);
void launch_push_photon_f64(const PartF64 &P, const double *F, const Grid &g, const PushConst &pc,
                            const QedParams &q, int *err, cudaStream_t st);
// (first: see k_push_qed_f32 -- nullptr pushes every particle)
void launch_push_qed_f32(const PartF32 &P, float *F, const Grid &g, const PushConst &pc, const QedParams &q,
                         int *err, double *e_abs, cudaStream_t st, const uint32_t *first = nullptr);
// (tc: with the surrogate, evaluate the pair network per CTA on the tcgen05
// tensor cores instead of per warp with mma.sync)
// (first: see k_push_photon_f32 -- nullptr pushes every photon; tc is not
// taken with first)
void launch_push_photon_f32(const PartF32 &P, const float *F, const Grid &g, const PushConst &pc,
                            const QedParams &q, int *err, cudaStream_t st, bool tc, const uint32_t *first = nullptr);

}  // namespace pic
