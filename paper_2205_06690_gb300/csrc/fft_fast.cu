// The register-pencil passes in FP32 (fft_fast.cuh).
#include "fft_fast.cuh"

namespace sbse {

int upload_reg_twiddles() {
  return upload_pencil_twiddles() == 0 && upload_reg_twiddles64() == 0 && upload_more_twiddles() == 0 ? 0 : -1;
}

SBSE_FAST_INST(float)

}  // namespace sbse
