// nr_rhs_cyl8.cu -- right-hand-side kernels for cylindrical-like grids, 8th-order scheme.
#include "nr_rhs_kernels.cuh"

namespace nrk {

NRK_RHS_LAUNCH(cyl8, FAM_CYL, 1, 8)

}  // namespace nrk
