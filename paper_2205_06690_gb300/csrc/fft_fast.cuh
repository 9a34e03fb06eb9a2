// Three-pass 3D FFT round trip with register-resident pencils (fft_pencil.cuh) on the grid edges that the
// workloads use most, and the launchers of every such grid: further edges go to fft_more.cu, 80 and 96
// (FP32) to fft_split.cu. Included by one translation unit per precision.
#pragma once

#include "fft_pencil.cuh"

namespace sbse {

#define SBSE_FAST_SWITCH(N, CALL)      \
  switch (N) {                         \
    case 8: CALL(8); break;            \
    case 10: CALL(10); break;          \
    case 12: CALL(12); break;          \
    case 16: CALL(16); break;          \
    case 20: CALL(20); break;          \
    case 24: CALL(24); break;          \
    case 32: CALL(32); break;          \
    case 40: CALL(40); break;          \
    case 48: CALL(48); break;          \
    case 64: CALL(64); break;          \
    default: break;                    \
  }

template <typename T>
void launch_step_persistent(const GridTables<T> &g, const XfwdArgs<T> &fa, const XfwdArgs<T> &fp,
                            C2<T> *a_next, C2<T> *d, T *dens, int L, const StepQueue &q, int grid,
                            cudaStream_t s) {
#define SBSE_CALL(n) FastOps<T>::template step<n>(g, fa, fp, a_next, d, dens, L, q, grid, s)
  SBSE_FAST_SWITCH(g.N, SBSE_CALL)
#undef SBSE_CALL
  count_launch(1);
}

template <typename T> int step_resident_blocks(int N) {
  int r = 0;
#define SBSE_CALL(n) r = FastOps<T>::template resident_blocks<n>()
  SBSE_FAST_SWITCH(N, SBSE_CALL)
#undef SBSE_CALL
  return r;
}

template <typename T> int step_tiles_per_orbital(int N) {
  int r = 0;
#define SBSE_CALL(n) r = FastOps<T>::template tiles_per_orbital<n>()
  SBSE_FAST_SWITCH(N, SBSE_CALL)
#undef SBSE_CALL
  return r;
}

template <typename T> bool fast_supported(int N) {
  // FP64 pencils of 64 would not fit in the register file; 80 and 96 take the FP32 lane-pair
  // passes of fft_split.cu
  if (split_size(N)) return sizeof(T) == 4;
  for (int i = 0; i < kRegCount; ++i)
    if (kRegSizes[i] == N) return !(sizeof(T) == 8 && N > 48);
  return false;
}

template <typename T> void init_fast_kernels() {
#define SBSE_ATTR(n) set_attrs<T, n, true>()
  SBSE_ATTR(8); SBSE_ATTR(10); SBSE_ATTR(12); SBSE_ATTR(16); SBSE_ATTR(20);
  SBSE_ATTR(24); SBSE_ATTR(32); SBSE_ATTR(40); SBSE_ATTR(48);
  if constexpr (sizeof(T) == 4) set_attrs<T, 64, true>();
#undef SBSE_ATTR
  init_more_kernels<T>();
}

template <typename T> void launch_plane_fwd(const GridTables<T> &g, const XfwdArgs<T> &a, cudaStream_t s) {
  count_launch(1);
  if constexpr (sizeof(T) == 4) {
    if (split_size(g.N)) {
      launch_plane_fwd2(g, a, s);
      return;
    }
  }
  if (more_size(g.N)) {
    launch_more_fwd<T>(g, a, s);
    return;
  }
#define SBSE_CALL(n) FastOps<T>::template fwd<n>(g, a, s)
  SBSE_FAST_SWITCH(g.N, SBSE_CALL)
#undef SBSE_CALL
}

template <typename T> void launch_zcol(const GridTables<T> &g, C2<T> *d, int n_items, int mult, cudaStream_t s) {
  count_launch(1);
  if constexpr (sizeof(T) == 4) {
    if (split_size(g.N)) {
      launch_zcol2(g, d, n_items, mult, s);
      return;
    }
  }
  if (more_size(g.N)) {
    launch_more_z<T>(g, d, n_items, mult, s);
    return;
  }
#define SBSE_CALL(n) FastOps<T>::template z<n>(g, d, n_items, mult, s)
  SBSE_FAST_SWITCH(g.N, SBSE_CALL)
#undef SBSE_CALL
}

template <typename T>
void launch_plane_inv_orb(const GridTables<T> &g, C2<T> *d, int n_items, const C2<T> *a_next, int L,
                          T *dens, cudaStream_t s) {
  // A second kernel sums the density from the stored orbitals: in the inverse pass it needs one block per
  // pair and plane group working through the pair's L orbitals in turn, and N more registers, which spill
  // in FP64. 3 pairs on 16^3: 318 -> 16 + 5 us; 10 pairs on 40^3, 918 -> 560 + 73 us.
  const PoissonOut po{0, 0.0, 0.0, 0.0};
  count_launch(1);
  if (more_size(g.N)) {
    launch_more_inv<T>(g, d, n_items, nullptr, nullptr, nullptr, po, PI_PLAIN, s);
  } else {
#define SBSE_CALL(n) FastOps<T>::template inv<n>(g, d, n_items, nullptr, nullptr, nullptr, po, PI_PLAIN, s)
    SBSE_FAST_SWITCH(g.N, SBSE_CALL)
#undef SBSE_CALL
  }
  if (dens) launch_density<T>(g, d, a_next, n_items / L, L, dens, s);
}

template <typename T>
void launch_plane_inv_poisson(const GridTables<T> &g, C2<T> *d, int n_slots, const PoissonOut &po,
                              T *u_out, T *acc, C2<T> *em1_out, cudaStream_t s) {
  count_launch(1);
  if constexpr (sizeof(T) == 4) {
    if (split_size(g.N)) {
      launch_plane_inv2_poisson(g, d, n_slots, po, u_out, acc, em1_out, s);
      return;
    }
  }
  if (more_size(g.N)) {
    launch_more_inv<T>(g, d, n_slots, u_out, acc, em1_out, po, PI_POISSON, s);
    return;
  }
#define SBSE_CALL(n) FastOps<T>::template inv<n>(g, d, n_slots, u_out, acc, em1_out, po, PI_POISSON, s)
  SBSE_FAST_SWITCH(g.N, SBSE_CALL)
#undef SBSE_CALL
}

// grids of the persistent step kernel
template <typename T> bool step_supported(int N) { return fast_supported<T>(N) && !split_size(N) && !more_size(N); }

#define SBSE_FAST_INST(T)                                                                           \
  template void launch_step_persistent<T>(const GridTables<T> &, const XfwdArgs<T> &,              \
                                          const XfwdArgs<T> &, C2<T> *, C2<T> *, T *, int,         \
                                          const StepQueue &, int, cudaStream_t);                   \
  template int step_resident_blocks<T>(int);                                                       \
  template int step_tiles_per_orbital<T>(int);                                                     \
  template bool step_supported<T>(int);                                                            \
  template bool fast_supported<T>(int);                                                            \
  template void init_fast_kernels<T>();                                                            \
  template void launch_plane_fwd<T>(const GridTables<T> &, const XfwdArgs<T> &, cudaStream_t);     \
  template void launch_zcol<T>(const GridTables<T> &, C2<T> *, int, int, cudaStream_t);            \
  template void launch_plane_inv_poisson<T>(const GridTables<T> &, C2<T> *, int, const PoissonOut &, \
                                            T *, T *, C2<T> *, cudaStream_t);

}  // namespace sbse
