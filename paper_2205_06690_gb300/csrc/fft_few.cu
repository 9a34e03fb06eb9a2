// Poisson round trips of few packed slots (potentials of a few pairs, hole-grid vectors), for which the
// thread-per-pencil kernels of fft_pencil.cuh leave most of the GPU idle: a warp then holds 32 pencils, there
// are fewer warps than SM sub-partitions, and a pass takes as long as one warp needs for its transforms
// (an FP64 warp instruction occupies its sub-partition's narrow pipe for about 64 clocks). Here four lanes of a
// warp share a pencil: N = 4 M, lane q holds the points 4 m + q, transforms M points in registers, and a
// radix-4 butterfly over two shuffles combines the four (decimation in time forward, in frequency
// backward, so the frequency layout k + M j needs no reordering). Four times the warps, each with about
// a third of the instructions; one plane per block. Figures at few_items below.
#include <math.h>

#include "fft_reg.cuh"
#include "bounds.cuh"
#include "kernels.h"
#include "passes.cuh"

namespace sbse {

namespace {

__constant__ float2 c_tqf[kRegTotal];
__constant__ double2 c_tqd[kRegTotal];
template <typename T> struct TwQ;
template <> struct TwQ<float> {
  __device__ __forceinline__ static float2 get(int i) { return c_tqf[i]; }
};
template <> struct TwQ<double> {
  __device__ __forceinline__ static double2 get(int i) { return c_tqd[i]; }
};

constexpr unsigned kAll = 0xffffffffu;

template <typename T> __device__ __forceinline__ C2<T> shfl_c(C2<T> v, int w) {
  return C2<T>{__shfl_xor_sync(kAll, v.x, w), __shfl_xor_sync(kAll, v.y, w)};
}

template <typename T, int M, int SIGN> __device__ __forceinline__ void fft_part(C2<T> (&v)[M]) {
  if constexpr (M == 4)
    dft_small<T, 4, SIGN, TwQ<T>>(v, 0, 4);
  else
    fft_reg<T, M, SIGN, TwQ<T>>(v);
}

// frequency block of lane q (lanes of a pencil: 8 apart): 0, 2, 1, 3
__device__ __forceinline__ int freq_block(int q) { return ((q & 1) << 1) | (q >> 1); }

// x[4 m + q] in v[m] -> X[k + M freq_block(q)] in v[k]; tw[k] = exp(-2 pi i k / N) in shared memory
template <typename T, int N> __device__ __forceinline__ void quad_fwd(C2<T> (&v)[N / 4], int q, const C2<T> *tw) {
  constexpr int M = N / 4;
  fft_part<T, M, -1>(v);
  const bool hi = q & 2, odd = q & 1;
#pragma unroll
  for (int k = 0; k < M; ++k) {
    C2<T> t = k > 0 ? cmul(v[k], tw[q * k]) : v[k];
    C2<T> o = shfl_c<T>(t, 16);
    t = hi ? csub(o, t) : cadd(t, o);
    if (q == 3) t = cmul_si(t, -1);
    o = shfl_c<T>(t, 8);
    v[k] = odd ? csub(o, t) : cadd(t, o);
  }
}

// the inverse of the layout change, unnormalised: X[k + M freq_block(q)] -> x[4 m + q]
template <typename T, int N> __device__ __forceinline__ void quad_inv(C2<T> (&v)[N / 4], int q, const C2<T> *tw) {
  constexpr int M = N / 4;
  const bool hi = q & 2, odd = q & 1;
#pragma unroll
  for (int k = 0; k < M; ++k) {
    C2<T> t = v[k], o = shfl_c<T>(t, 8);
    t = odd ? csub(o, t) : cadd(t, o);
    if (q == 3) t = cmul_si(t, +1);
    o = shfl_c<T>(t, 16);
    t = hi ? csub(o, t) : cadd(t, o);
    v[k] = k > 0 ? cmul(t, cconj(tw[q * k])) : t;
  }
  fft_part<T, M, +1>(v);
}

template <typename T, int N> constexpr size_t few_smem() { return ((size_t)N * (N + 1) + N) * sizeof(C2<T>); }

// block = one plane of one item: pre-operation, x and y transforms
template <typename T, int N>
__global__ void __launch_bounds__(4 * N) k_few_fwd(GView<T> g, XfwdArgs<T> a) {
  using C = C2<T>;
  constexpr int M = N / 4, LD = N + 1, NN = N * N, NT = 4 * N, UB = M < 8 ? M : 8;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C *S = reinterpret_cast<C *>(smem_raw), *tw = S + N * LD;
  const long long item = blockIdx.x / N, off = (long long)(blockIdx.x % N) * NN;
  (void)SBSE_IDX(item, a.n_items);
  for (int i = threadIdx.x; i < N; i += NT) tw[i] = g.tw[i];
  const PreopItem<T> it = preop_item<T>(g, a, item);
#pragma unroll 1
  for (int k0 = 0; k0 < M; k0 += UB) {
    C v[UB];
#pragma unroll
    for (int k = 0; k < UB; ++k)
      if (k0 + k < M) v[k] = preop_at<T>(g, it, off + threadIdx.x + (k0 + k) * NT);
#pragma unroll
    for (int k = 0; k < UB; ++k)
      if (k0 + k < M) S[(threadIdx.x / N + 4 * (k0 + k)) * LD + threadIdx.x % N] = v[k];
  }
  __syncthreads();
  const int lane = threadIdx.x & 31, q = lane >> 3, p = (threadIdx.x >> 5) * 8 + (lane & 7), fb = freq_block(q) * M;
  C v[M];
  C *row = S + p * LD;
#pragma unroll
  for (int m = 0; m < M; ++m) v[m] = row[4 * m + q];
  quad_fwd<T, N>(v, q, tw);
  __syncwarp();
#pragma unroll
  for (int k = 0; k < M; ++k) row[fb + k] = v[k];
  __syncthreads();
#pragma unroll
  for (int m = 0; m < M; ++m) v[m] = S[(4 * m + q) * LD + p];
  quad_fwd<T, N>(v, q, tw);
  C *out = a.out + item * g.ng + off + p;
#pragma unroll
  for (int k = 0; k < M; ++k) out[(fb + k) * N] = v[k];
}

// z columns: 8 consecutive columns per warp
constexpr int kFewZ = 64;
template <typename T, int N>
__global__ void __launch_bounds__(kFewZ) k_few_z(GView<T> g, C2<T> *data, int mult, int n_items) {
  using C = C2<T>;
  constexpr int M = N / 4, NN = N * N;
  __shared__ C tw[N];
  for (int i = threadIdx.x; i < N; i += kFewZ) tw[i] = g.tw[i];
  __syncthreads();
  const int lane = threadIdx.x & 31, q = lane >> 3, fb = freq_block(q) * M;
  const long long c = ((long long)blockIdx.x * (kFewZ / 32) + (threadIdx.x >> 5)) * 8 + (lane & 7);
  const long long item = c / NN;  // (NN is a multiple of the block's 16 columns)
  const int rem = (int)(c - item * NN), y = rem / N, x = rem - y * N;
  (void)SBSE_IDX(item, n_items);
  C *base = data + item * g.ng + rem;
  C v[M];
#pragma unroll
  for (int m = 0; m < M; ++m) v[m] = base[(long long)(4 * m + q) * NN];
  quad_fwd<T, N>(v, q, tw);
  const T inv_ng = T(1) / T(N * N * N);
  if (mult == Z_KINETIC) {
    const C mxy = cscale(cmul(g.kin[x], g.kin[y]), inv_ng);
#pragma unroll
    for (int k = 0; k < M; ++k) v[k] = cmul(v[k], cmul(mxy, g.kin[fb + k]));
  } else {
    const T gxy = g.k2[x] + g.k2[y];
    const bool half = mult == Z_HOLE_GRID && item + 1 < n_items;
#pragma unroll
    for (int k = 0; k < M; ++k) {
      const T G2 = gxy + g.k2[fb + k];
      v[k] = cscale(v[k], half ? T(0.5) * G2 * inv_ng : (G2 > T(0) ? T(4.0 * M_PI) * inv_ng / G2 : T(0)));
    }
  }
  quad_inv<T, N>(v, q, tw);
#pragma unroll
  for (int m = 0; m < M; ++m) base[(long long)(4 * m + q) * NN] = v[m];
}

// block = one plane of one item: y and x inverse transforms, then the unpacking of the slot's two
// potentials with the time integral and E - 1 (as in fft_pencil.cuh)
template <typename T, int N>
__global__ void __launch_bounds__(4 * N)
    k_few_inv(GView<T> g, const C2<T> *data, T *u_out, T *acc, C2<T> *em1_out, PoissonOut po) {
  using C = C2<T>;
  constexpr int M = N / 4, LD = N + 1, NN = N * N, NT = 4 * N;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C *S = reinterpret_cast<C *>(smem_raw), *tw = S + N * LD;
  const long long item = blockIdx.x / N, off = (long long)(blockIdx.x % N) * NN;
  for (int i = threadIdx.x; i < N; i += NT) tw[i] = g.tw[i];
  __syncthreads();
  const int lane = threadIdx.x & 31, q = lane >> 3, p = (threadIdx.x >> 5) * 8 + (lane & 7), fb = freq_block(q) * M;
  const C *base = data + item * g.ng + off;
  C v[M];
#pragma unroll
  for (int k = 0; k < M; ++k) v[k] = base[(fb + k) * N + p];
  quad_inv<T, N>(v, q, tw);
#pragma unroll
  for (int m = 0; m < M; ++m) S[(4 * m + q) * LD + p] = v[m];
  __syncthreads();
  C *row = S + p * LD;
#pragma unroll
  for (int k = 0; k < M; ++k) v[k] = row[fb + k];
  quad_inv<T, N>(v, q, tw);
  __syncwarp();
#pragma unroll
  for (int m = 0; m < M; ++m) row[4 * m + q] = v[m];
  __syncthreads();
  const T coef = (T)po.coef, tau = (T)po.tau_next;
  const bool keep = po.keep != 0.0;
#pragma unroll 2
  for (int k = 0; k < M; ++k) {
    const int l = threadIdx.x + k * NT;
    const C x = S[(threadIdx.x / N + 4 * k) * LD + threadIdx.x % N];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      if (2 * item + h >= po.n_out) break;
      const T val = h ? x.y : x.x;
      const long long o = (2 * item + h) * g.ng + off + l;
      if (u_out) u_out[o] = val;
      if (acc) acc[o] = (keep ? acc[o] : T(0)) + coef * val;
      if (em1_out) em1_out[o] = phase_em1<T>(val, tau);
    }
  }
}

#define SBSE_FEW_SWITCH(N, CALL) \
  switch (N) {                   \
    case 16: CALL(16); break;    \
    case 32: CALL(32); break;    \
    case 40: CALL(40); break;    \
    case 48: CALL(48); break;    \
    case 64: CALL(64); break;    \
    default: break;              \
  }

template <typename T, int N> void few_attrs() {
  if (few_smem<T, N>() > 48 * 1024) {
    raise_smem_limit((const void *)k_few_fwd<T, N>, few_smem<T, N>());
    raise_smem_limit((const void *)k_few_inv<T, N>, few_smem<T, N>());
  }
}

}  // namespace

// Whether n_items slots leave the thread-per-pencil passes short of warps (32 pencils each; the GPU has
// 608 SM sub-partitions). In FP32 a pass is latency-bound up to one warp per sub-partition (5 slots of
// 32^3, 160 warps: 11.3 + 4.6 + 5.1 -> 8.7 + 3.7 + 3.4 us). In FP64 the quartered pencils' extra
// instructions (about 1.5 times as many) count once a quarter of the sub-partitions are busy: 2 slots of
// 32^3, 64 warps: 32 + 31 + 41 -> 16 + 16 + 17 us; 5 slots of 40^3, 250 warps, were slower (fwd 62 -> 90,
// inv 165 -> 220 us). Edges: a warp holds 8 pencils, so multiples of 8, with a register transform of N / 4
// points (that leaves out 24, a 6-point transform, and 56, 72, 80 and 96, whose slots are seldom few).
template <typename T> bool few_items(int N, long long n_items) {
  if (N != 16 && N != 32 && N != 40 && N != 48 && N != 64) return false;
  return n_items * N * N / 32 < (sizeof(T) == 8 ? kSMs : 4 * kSMs);
}

int upload_few_twiddles() {
  float2 hf[kRegTotal];
  double2 hd[kRegTotal];
  for (int s = 0; s < kRegCount; ++s) {
    const int N = kRegSizes[s], off = reg_offset(N);
    for (int k = 0; k < N; ++k) {
      const double a = -2.0 * M_PI * (double)k / (double)N;
      hd[off + k] = make_double2(cos(a), sin(a));
      hf[off + k] = make_float2((float)cos(a), (float)sin(a));
    }
  }
#define SBSE_ATTR(n) (few_attrs<float, n>(), few_attrs<double, n>())
  SBSE_ATTR(16); SBSE_ATTR(32); SBSE_ATTR(40); SBSE_ATTR(48); SBSE_ATTR(64);
#undef SBSE_ATTR
  return cudaMemcpyToSymbol(c_tqf, hf, sizeof(hf)) == cudaSuccess && cudaMemcpyToSymbol(c_tqd, hd, sizeof(hd)) == cudaSuccess
             ? 0
             : -1;
}

template <typename T> void launch_few_fwd(const GridTables<T> &g, const XfwdArgs<T> &a, cudaStream_t s) {
#define SBSE_CALL(n) k_few_fwd<T, n><<<(unsigned)(a.n_items * n), 4 * n, few_smem<T, n>(), s>>>(view(g), a)
  SBSE_FEW_SWITCH(g.N, SBSE_CALL)
#undef SBSE_CALL
  count_launch(1);
}
template <typename T> void launch_few_z(const GridTables<T> &g, C2<T> *d, int n_items, int mult, cudaStream_t s) {
#define SBSE_CALL(n) k_few_z<T, n><<<(unsigned)(n_items * n * n / 16), kFewZ, 0, s>>>(view(g), d, mult, n_items)
  SBSE_FEW_SWITCH(g.N, SBSE_CALL)
#undef SBSE_CALL
  count_launch(1);
}
template <typename T>
void launch_few_inv(const GridTables<T> &g, C2<T> *d, int n_items, const PoissonOut &po, T *u_out, T *acc, C2<T> *em1_out,
                    cudaStream_t s) {
#define SBSE_CALL(n) \
  k_few_inv<T, n><<<(unsigned)(n_items * n), 4 * n, few_smem<T, n>(), s>>>(view(g), d, u_out, acc, em1_out, po)
  SBSE_FEW_SWITCH(g.N, SBSE_CALL)
#undef SBSE_CALL
  count_launch(1);
}

#define SBSE_FEW_INST(T)                                                                                    \
  template bool few_items<T>(int, long long);                                                               \
  template void launch_few_fwd<T>(const GridTables<T> &, const XfwdArgs<T> &, cudaStream_t);                \
  template void launch_few_z<T>(const GridTables<T> &, C2<T> *, int, int, cudaStream_t);                    \
  template void launch_few_inv<T>(const GridTables<T> &, C2<T> *, int, const PoissonOut &, T *, T *, C2<T> *, \
                                  cudaStream_t);
SBSE_FEW_INST(float)
SBSE_FEW_INST(double)

}  // namespace sbse
