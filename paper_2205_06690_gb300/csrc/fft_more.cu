// The register-pencil passes (fft_pencil.cuh) on further grid edges: box-size sweeps at a fixed spacing ask
// for any edge with factors 2, 3, 5. The five passes of runtime radix (tdh_kernels.cu) that these sizes
// took spend their time on index arithmetic and shared-memory stages: 105 orbitals of 45^3 (15 pairs),
// a pass of 60 steps took 55.7 ms with them and takes 12.4 ms with these.
#include "fft_pencil.cuh"

namespace sbse {

bool more_size(int N) {
  return N == 18 || N == 25 || N == 27 || N == 30 || N == 36 || N == 45 || N == 50 || N == 54 || N == 60;
}

int upload_more_twiddles() { return upload_pencil_twiddles(); }

#define SBSE_MORE_SWITCH(N, CALL) \
  switch (N) {                    \
    case 18: CALL(18); break;     \
    case 25: CALL(25); break;     \
    case 27: CALL(27); break;     \
    case 30: CALL(30); break;     \
    case 36: CALL(36); break;     \
    case 45: CALL(45); break;     \
    case 50: CALL(50); break;     \
    case 54: CALL(54); break;     \
    case 60: CALL(60); break;     \
    default: break;               \
  }

namespace {
template <typename T, int N> void more_attrs() {
  if constexpr (!(sizeof(T) == 8 && N > 48)) set_attrs<T, N>();
}
}  // namespace

template <typename T> void init_more_kernels() {
#define SBSE_ATTR(n) more_attrs<T, n>()
  SBSE_ATTR(18); SBSE_ATTR(25); SBSE_ATTR(27); SBSE_ATTR(30); SBSE_ATTR(36); SBSE_ATTR(45);
  SBSE_ATTR(50); SBSE_ATTR(54); SBSE_ATTR(60);
#undef SBSE_ATTR
}

template <typename T> void launch_more_fwd(const GridTables<T> &g, const XfwdArgs<T> &a, cudaStream_t s) {
#define SBSE_CALL(n) FastOps<T>::template fwd<n>(g, a, s)
  SBSE_MORE_SWITCH(g.N, SBSE_CALL)
#undef SBSE_CALL
}

template <typename T> void launch_more_z(const GridTables<T> &g, C2<T> *d, int n_items, int mult, cudaStream_t s) {
#define SBSE_CALL(n) FastOps<T>::template z<n>(g, d, n_items, mult, s)
  SBSE_MORE_SWITCH(g.N, SBSE_CALL)
#undef SBSE_CALL
}

template <typename T>
void launch_more_inv(const GridTables<T> &g, C2<T> *d, int n_items, T *u_out, T *acc, C2<T> *em1_out, const PoissonOut &po,
                     int mode, cudaStream_t s) {
#define SBSE_CALL(n) FastOps<T>::template inv<n>(g, d, n_items, u_out, acc, em1_out, po, mode, s)
  SBSE_MORE_SWITCH(g.N, SBSE_CALL)
#undef SBSE_CALL
}

void launch_more_kin(const GridTables<float> &g, const XfwdArgs<float> &a, cudaStream_t s) {
#define SBSE_CALL(n) FastOps<float>::kin<n>(g, a, s)
  SBSE_MORE_SWITCH(g.N, SBSE_CALL)
#undef SBSE_CALL
}

void launch_more_zkin(const GridTables<float> &g, float2 *d, int n_items, const float2 *a_next, int L, float *dens,
                      cudaStream_t s) {
#define SBSE_CALL(n) FastOps<float>::zkin<n>(g, d, n_items, a_next, L, dens, s)
  SBSE_MORE_SWITCH(g.N, SBSE_CALL)
#undef SBSE_CALL
}

#define SBSE_MORE_INST(T)                                                                                        \
  template void init_more_kernels<T>();                                                                          \
  template void launch_more_fwd<T>(const GridTables<T> &, const XfwdArgs<T> &, cudaStream_t);                    \
  template void launch_more_z<T>(const GridTables<T> &, C2<T> *, int, int, cudaStream_t);                        \
  template void launch_more_inv<T>(const GridTables<T> &, C2<T> *, int, T *, T *, C2<T> *, const PoissonOut &, int, \
                                   cudaStream_t);
SBSE_MORE_INST(float)
SBSE_MORE_INST(double)

}  // namespace sbse
