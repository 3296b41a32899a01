// nr_rhs_cyl.cu -- right-hand-side kernels for cylindrical-like grids, 4th-order scheme.
#include "nr_rhs_kernels.cuh"

namespace nrk {

NRK_RHS_LAUNCH(cyl4, FAM_CYL, 1, 4)

}  // namespace nrk
