// nr_rhs_sph.cu -- right-hand-side kernels for spherical-like grids, 4th-order scheme.
#include "nr_rhs_kernels.cuh"

namespace nrk {

NRK_RHS_LAUNCH(sph4, FAM_SPH, 2, 4)

}  // namespace nrk
