// The register-pencil passes in FP64 (fft_fast.cuh).
#include "fft_fast.cuh"

namespace sbse {

int upload_reg_twiddles64() { return upload_pencil_twiddles(); }

SBSE_FAST_INST(double)
template void launch_plane_inv_orb<double>(const GridTables<double> &, double2 *, int, const double2 *, int, double *,
                                           cudaStream_t);

}  // namespace sbse
