// fdtd.cuh -- launchers of the field kernels (fdtd.cu).
#pragma once
#include "pic_internal.cuh"

namespace pic {

template <typename R>
void launch_update_E(R *F, const Grid &g, double h, bool twice, bool zeroJ, cudaStream_t st);
template <typename R>
void launch_update_B(R *F, const Grid &g, double h, const Laser &L, bool fold, cudaStream_t st);  // fold: of J, too
// 1D grids small enough for one block: the half steps between two pushes in
// one launch.  begin: E half and B half before a call's first push (J := 0);
// else the fold, B half, E half -- twice, J := 0 and B half again unless last
template <typename R>
bool fields_in_one_block(const Grid &g);
template <typename R>
void launch_fields_1d(R *F, const Grid &g, double h, bool begin, bool last, const Laser &L1, const Laser &L2,
                      cudaStream_t st);
void launch_fold_rho(double *rho, const Grid &g, cudaStream_t st);

}  // namespace pic
