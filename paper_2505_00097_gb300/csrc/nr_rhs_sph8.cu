// nr_rhs_sph8.cu -- right-hand-side kernels for spherical-like grids, 8th-order scheme.
#include "nr_rhs_kernels.cuh"

namespace nrk {

NRK_RHS_LAUNCH(sph8, FAM_SPH, 2, 8)

}  // namespace nrk
