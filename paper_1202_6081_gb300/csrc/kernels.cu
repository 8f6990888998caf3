// Explicit instantiations of the kernels' launchers.  Compiled once per lattice
// LBM_Q (27, 15), storage type LBM_T and group of kernels LBM_GROUP (STEP,
// INPLACE, STATE, ADJOINT), so that the units build in parallel (build.py).
#include "adjoint_kernels.cuh"

namespace lbm {
#define LBM_CAT_(a, b) a##b
#define LBM_CAT(a, b) LBM_CAT_(a, b)
LBM_CAT(LBM_INSTANTIATE_, LBM_GROUP)(, LBM_Q, LBM_T)
}  // namespace lbm
