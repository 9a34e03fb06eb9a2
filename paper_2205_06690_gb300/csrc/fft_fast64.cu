// The register-pencil passes in FP64 (fft_fast.cuh).
#include "fft_fast.cuh"

namespace sbse {

int upload_reg_twiddles64() { return upload_pencil_twiddles(); }

SBSE_FAST_INST(double)

}  // namespace sbse
