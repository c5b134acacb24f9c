// diag.cuh -- FP64 diagnostics (diag.cu).
#pragma once
#include "pic_internal.cuh"
#include "push.cuh"

namespace pic {

// scratch of the reductions (zeroed once; one stream uses it); out: device doubles
size_t diag_scratch_doubles();
template <typename R>
void diag_field_energy(const R *F, const Grid &g, double *scratch, double *out2, cudaStream_t st);
void diag_kinetic_f32(const PartF32 &P, bool photon, double *scratch, double *out2, cudaStream_t st);
void diag_kinetic_f64(const PartF64 &P, bool photon, double *scratch, double *out2, cudaStream_t st);
void diag_rho_f32(const PartF32 &P, const Grid &g, double qw, double *rho, cudaStream_t st);
void diag_rho_f64(const PartF64 &P, const Grid &g, double qw, double *rho, cudaStream_t st);
template <typename R>
void diag_gauss(const R *F, const double *rho, const Grid &g, double rho_bg, const double *t1, const double *t2,
                double *scratch, double *out3, cudaStream_t st);
// one component between the padded array and the exchange layout of m[0] x
// m[1] x m[2] FP64 values (device buffers)
template <typename R>
void field_pack(const R *comp, const Grid &g, const long long *m, double *out, cudaStream_t st);
template <typename R>
void field_unpack(const double *in, const Grid &g, const long long *m, R *comp, cudaStream_t st);

}  // namespace pic
