// Instantiations: the persistent change-list kernel, block width 256, few rows per SM.
#define QE_SWEEP_INSTANTIATE
#include "qe_sweep.cuh"

namespace qe {
template cudaError_t launch_cd_rows_w<256, true> QE_SWEEP_ROWS_W_SIG;
}  // namespace qe
