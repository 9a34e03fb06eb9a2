// The register-pencil passes in FP32 (fft_fast.cuh) and the two sweeps of the FP32 orbitals.
#include "fft_fast.cuh"

namespace sbse {

int upload_reg_twiddles() {
  return upload_pencil_twiddles() == 0 && upload_pair_twiddles() == 0 && upload_reg_twiddles64() == 0 &&
                 upload_more_twiddles() == 0
             ? 0
             : -1;
}

SBSE_FAST_INST(float)

void launch_kin_planes(const GridTables<float> &g, const XfwdArgs<float> &a, cudaStream_t s) {
  count_launch(1);
  if (pair_size(g.N)) {
    launch_plane_kin2(g, a, s);
    return;
  }
  if (more_size(g.N)) {
    launch_more_kin(g, a, s);
    return;
  }
#define SBSE_CALL(n) FastOps<float>::kin<n>(g, a, s)
  SBSE_FAST_SWITCH(g.N, SBSE_CALL)
#undef SBSE_CALL
}

void launch_kin_z(const GridTables<float> &g, float2 *d, int n_items, const float2 *a_next, int L, float *dens,
                  cudaStream_t s, int *err) {
  count_launch(1);
  if (pair_size(g.N)) {
    launch_zkin2(g, d, n_items, a_next, L, dens, s, err);
    return;
  }
  if (more_size(g.N)) {
    launch_more_zkin(g, d, n_items, a_next, L, dens, s);
    return;
  }
#define SBSE_CALL(n) FastOps<float>::zkin<n>(g, d, n_items, a_next, L, dens, s)
  SBSE_FAST_SWITCH(g.N, SBSE_CALL)
#undef SBSE_CALL
}

}  // namespace sbse
