// Three-pass 3D FFT round trip with compile-time N and register-resident pencils, used by the
// split-operator step of Eq. (10), the Poisson solves of Eq. (11) / q_ij and the exchange
// potentials of Eq. (1):
//   plane forward  : coalesced load of PPB z-planes with the fused pre-operation into shared
//                    memory (rows padded to N + 1), x FFT (thread per row), y FFT (thread per
//                    column), coalesced store
//   z column       : thread per (x, y) column, coalesced across x: forward z FFT, multiplier
//                    (kinetic propagator exp(-i |G|^2 dt / 2) or 4 pi / |G|^2, with 1/N^3),
//                    inverse z FFT, store
//   plane inverse  : y and x inverse FFTs, then the fused epilogue: plain store, store plus the
//                    induced density of all L orbitals of a pair (Eq. 11), or the Poisson
//                    unpacking with the damped time-integral accumulation of Eq. (13)
// Each element crosses HBM three times per round trip instead of five for the generic passes.
// Included by the translation units that instantiate it (each with its own twiddle tables).
#pragma once

#include <math.h>

#include <type_traits>

#include "fft_pair.cuh"

namespace sbse {


namespace {

__constant__ float2 c_twf[kRegTotal];
__constant__ double2 c_twd[kRegTotal];

template <typename T> struct TwP;  // twiddles of this translation unit
template <> struct TwP<float> {
  __device__ __forceinline__ static float2 get(int i) { return c_twf[i]; }
};
template <> struct TwP<double> {
  __device__ __forceinline__ static double2 get(int i) { return c_twd[i]; }
};

int upload_pencil_twiddles() {
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
  if (cudaMemcpyToSymbol(c_twf, hf, sizeof(hf)) != cudaSuccess) return -1;
  if (cudaMemcpyToSymbol(c_twd, hd, sizeof(hd)) != cudaSuccess) return -1;
  return 0;
}

// Loads of data that other blocks of the same launch may have written (persistent step kernel)
// bypass L1, which is not coherent across SMs.
template <bool COH, typename C> __device__ __forceinline__ C ldv(const C *p) {
  if constexpr (COH) return __ldcg(p);
  else return *p;
}

// planes per block: the largest divisor of N with <= 256 threads and <= 96 KB of shared memory
constexpr int plane_ppb(int N, int csize) {
  int best = 1;
  for (int d = 1; d <= N; ++d)
    if (N % d == 0 && d * N <= 256 && (long long)d * N * (N + 1) * csize <= 96 * 1024) best = d;
  return best;
}

template <typename T, int N> constexpr int kPPB = plane_ppb(N, (int)sizeof(C2<T>));
template <typename T, int N> constexpr size_t plane_smem() {
  return (size_t)kPPB<T, N> * N * (N + 1) * sizeof(C2<T>);
}

// ------------------------------------------------------------------------------------------

// One-dimensional kinetic operator F^-1 diag(kt) F of a pencil in registers (kt: a table of kin_tables.h)
template <int N> __device__ __forceinline__ void kin_pencil(float2 (&v)[N], const float2 *kt) {
  fft_reg<float, N, -1, TwP<float>>(v);
#pragma unroll
  for (int k = 0; k < N; ++k) v[k] = cmul(v[k], kt[k]);
  fft_reg<float, N, +1, TwP<float>>(v);
}
// the table of a sweep (`at`: kin_xy(N) or kin_z(N)); the caller synchronises
template <int N> __device__ __forceinline__ void load_kin(float2 *kt, const GView<float> &g, int at) {
  for (int i = threadIdx.x; i < N; i += blockDim.x) kt[i] = g.kin[at + i];
}

// The PPB planes starting at plane offset `off` (= z0 N^2) of `item`: the fused pre-operation, then the
// forward x and y FFTs, or with KIN (FP32 orbitals) the x and y kinetic operators; S is the block's
// shared tile
template <typename T, int N, bool PAIR, int PPB = kPPB<T, N>, bool KIN = false>
__device__ __forceinline__ void fwd_planes(const GView<T> &g, const XfwdArgs<T> &a, long long item,
                                           long long off, C2<T> *S, const C2<T> *kt = nullptr) {
  using C = C2<T>;
  constexpr int LD = N + 1, NN = N * N, NT = PPB * N;
  const PreopItem<T> it = preop_item<T>(g, a, item);
  // the thread's points lie in one column, PPB rows apart (NT = PPB N points per sweep of the block)
  C *srow = S + (threadIdx.x / N) * LD + threadIdx.x % N;
  if constexpr (PAIR) {
    // the hot pre-operation of the pair batch: loads of 8 points are issued before any is used;
    // the batch loop stays rolled (the unrolled one stalled on instruction fetch: 162 -> 156 us)
    constexpr int UB = 8;
    const C *dp = it.in + off, *ap = it.a + off, *pp = it.pv + off;
    const C *ep = it.em1 ? it.em1 + off : nullptr;
    // the deferred renormalisation is pending only in the step after a cleaning (cm1 != 0, the same for
    // the whole block): without one d enters unchanged, and FP64 saves a tenth of the pass
    auto sweep = [&](auto renorm) {
      constexpr bool RN = decltype(renorm)::value;
#pragma unroll 1
      for (int k0 = 0; k0 < N; k0 += UB) {
        C dv[UB], av[UB], pv[UB], ev[UB];
#pragma unroll
        for (int k = 0; k < UB; ++k) {
          if (k0 + k < N) {
            const int l = threadIdx.x + (k0 + k) * NT;
            dv[k] = dp[l];
            av[k] = ap[l];
            pv[k] = pp[l];
            ev[k] = ep ? ep[l] : C{T(0), T(0)};
          }
        }
#pragma unroll
        for (int k = 0; k < UB; ++k) {
          if (k0 + k < N) {
            srow[(k0 + k) * PPB * LD] =
                pair_phase<T>(pv[k], ev[k], av[k], RN ? renorm_value<T>(dv[k], av[k], it.cm1) : dv[k]);
          }
        }
      }
    };
    if (sizeof(T) == 4 || it.cm1 != T(0))
      sweep(std::true_type{});
    else
      sweep(std::false_type{});
  } else {
    // the other pre-operations, with the mode resolved outside the point loop so that each batch
    // of UB points issues all its loads before the first shared-memory store
    constexpr int UB = 8;
    auto run = [&](auto f) {
      // the batch loop is not unrolled: five variants of fully unrolled point loops overflowed the
      // instruction cache (no-instruction stalls)
#pragma unroll 1
      for (int k0 = 0; k0 < N; k0 += UB) {
        C v[UB];
#pragma unroll
        for (int k = 0; k < UB; ++k)
          if (k0 + k < N) v[k] = f(off + threadIdx.x + (k0 + k) * NT);
#pragma unroll
        for (int k = 0; k < UB; ++k) {
          if (k0 + k < N) srow[(k0 + k) * PPB * LD] = v[k];
        }
      }
    };
    if (it.mode == XF_PHASE_A) {
      run([&](long long i) { return cmul(it.pv[i], it.in[i]); });
    } else if (it.mode == XF_PACK_DN) {
      if (it.r1)
        run([&](long long i) { return C{it.r0[i], it.r1[i]}; });
      else
        run([&](long long i) { return C{it.r0[i], T(0)}; });
    } else if (it.mode == XF_PACK_PROD) {
      if (it.r2)
        run([&](long long i) { return C{it.r0[i] * it.r1[i], it.r2[i] * it.r3[i]}; });
      else
        run([&](long long i) { return C{it.r0[i] * it.r1[i], T(0)}; });
    } else {
      run([&](long long i) { return preop_at<T>(g, it, i); });
    }
  }
  __syncthreads();
  const int pl = threadIdx.x / N, q = threadIdx.x - pl * N;
  {
    C v[N];
    C *row = S + (pl * N + q) * LD;
#pragma unroll
    for (int x = 0; x < N; ++x) v[x] = row[x];
    if constexpr (KIN)
      kin_pencil<N>(v, kt);
    else
      fft_reg<T, N, -1, TwP<T>>(v);
#pragma unroll
    for (int x = 0; x < N; ++x) row[x] = v[x];
  }
  __syncthreads();
  {
    C v[N];
    const C *col = S + pl * N * LD + q;
#pragma unroll
    for (int y = 0; y < N; ++y) v[y] = col[y * LD];
    if constexpr (KIN)
      kin_pencil<N>(v, kt);
    else
      fft_reg<T, N, -1, TwP<T>>(v);
    C *out = a.out + item * g.ng + off + pl * NN + q;
#pragma unroll
    for (int y = 0; y < N; ++y) out[y * N] = v[y];
  }
}

// planes per block of the forward pass: the FP32 pair batch takes half the planes of the other
// passes (smaller blocks: five resident per SM instead of two, 15 warps instead of 12, to hide
// the L2 latency of its pre-operation's table loads)
template <typename T, int N, bool PAIR> constexpr int fwd_ppb() {
  return (PAIR && sizeof(T) == 4 && kPPB<T, N> % 2 == 0) ? kPPB<T, N> / 2 : kPPB<T, N>;
}
template <typename T, int N, bool PAIR> constexpr size_t fwd_smem() {
  return (size_t)fwd_ppb<T, N, PAIR>() * N * (N + 1) * sizeof(C2<T>);
}

// Planes per block where the usual blocks would leave half of the SMs without one (eta0 sets and pair
// batches of small systems): the smallest divisor of N that keeps three quarters of a warp's lanes busy.
// The transforms of a pencil are the same, so are the results. 3 pairs on 16^3 in FP64 (30 orbitals):
// forward pass 45 -> 24 us, inverse 318 (with the density) -> 16 + 5 us; 10 eta0 orbitals on 32^3 in FP32:
// 5.6 -> 5.1 us. At 120 blocks (eta0 on 48^3) the smaller blocks were slower (5.8 -> 9.2 us).
constexpr int few_ppb(int N, int most) {
  for (int d = 1; d < most; ++d)
    if (N % d == 0 && d * N >= 32 && 4 * d * N >= 3 * 32 * ((d * N + 31) / 32)) return d;
  return most;
}
template <typename T, int N> constexpr int kFew = few_ppb(N, kPPB<T, N>);
template <typename T, int N> constexpr size_t few_plane_smem() {
  return (size_t)kFew<T, N> * N * (N + 1) * sizeof(C2<T>);
}
constexpr long long kFewBlocks = kSMs / 2;
template <typename T, int N> constexpr bool few_planes(long long planes) {
  return kFew<T, N> < kPPB<T, N> && planes / kPPB<T, N> < kFewBlocks;
}

template <typename T, int N, bool PAIR, int PPB>
__global__ void __launch_bounds__(PPB * N) k_plane_fwd(GView<T> g, XfwdArgs<T> a, long long planes_total) {
  constexpr int NN = N * N;
  extern __shared__ unsigned char smem_raw[];
  // PPB divides N: the block's planes z0 .. z0 + PPB - 1 are contiguous inside one item
  const long long p0 = (long long)blockIdx.x * PPB;
  const long long item = p0 / N;
  (void)SBSE_IDX(p0 + PPB - 1, planes_total);
  (void)SBSE_IDX(item, a.n_items);
  fwd_planes<T, N, PAIR, PPB>(g, a, item, (p0 - item * N) * NN, reinterpret_cast<C2<T> *>(smem_raw));
}

// First sweep of the two-sweep split-operator step of the FP32 orbitals: the kinetic propagator is the
// product of one operator per axis, so the planes take the potential phase and the x and y operators, and
// the second sweep (k_zkin) the z operator. Two sweeps over the orbitals instead of the three of a 3D
// round trip. 15 pairs of 45^3: planes 82 us, z 14.5 us and density 13.6 us; the whole W 12.0 ms (three
// sweeps: 12.4 ms). Grids with lane-pair pencils (fft_split.cu) take theirs.
template <int N, bool PAIR, int PPB>
__global__ void __launch_bounds__(PPB * N) k_plane_kin(GView<float> g, XfwdArgs<float> a, long long planes_total) {
  constexpr int NN = N * N;
  extern __shared__ unsigned char smem_raw[];
  __shared__ float2 kt[N];
  load_kin<N>(kt, g, kin_xy(N));  // (read after the pre-operation's barrier)
  const long long p0 = (long long)blockIdx.x * PPB;
  const long long item = p0 / N;
  (void)SBSE_IDX(p0 + PPB - 1, planes_total);
  (void)SBSE_IDX(item, a.n_items);
  fwd_planes<float, N, PAIR, PPB, true>(g, a, item, (p0 - item * N) * NN, reinterpret_cast<float2 *>(smem_raw), kt);
}

// the density of a column of one orbital added to acc[z * stride] (first: assigned), eta0 loaded in batches
template <int N, bool COH>
__device__ __forceinline__ void add_density(const float2 (&v)[N], const float2 *ab, float *acc, int stride, bool first) {
  constexpr int UB = 16, NN = N * N;
#pragma unroll
  for (int z0 = 0; z0 < N; z0 += UB) {
    float2 a0[UB];
#pragma unroll
    for (int k = 0; k < UB; ++k)
      if (z0 + k < N) a0[k] = ldv<COH>(ab + (long long)(z0 + k) * NN);
#pragma unroll
    for (int k = 0; k < UB; ++k)
      if (z0 + k < N) {
        const float t = density_term<float>(a0[k], v[z0 + k]);
        float &d = acc[(z0 + k) * stride];
        d = first ? t : d + t;
      }
    asm volatile("" ::: "memory");  // keep the next batch's loads below this one (registers)
  }
}

// Second sweep: the z kinetic operator, a thread per (x, y) column. DENS: of each of the L orbitals of a pair
// (unit), summing the pair's induced density in shared memory.
constexpr int kZkT = 128;
template <int N, bool DENS>
__global__ void __launch_bounds__(kZkT)
    k_zkin(GView<float> g, float2 *data, const float2 *a_next, float *dens, int n_units, int L) {
  using C = float2;
  constexpr int NN = N * N;
  __shared__ C kt[N];
  __shared__ float D[DENS ? N * kZkT : 1];
  load_kin<N>(kt, g, kin_z(N));
  __syncthreads();
  const long long cols = (NN + blockDim.x - 1) / blockDim.x;  // blocks per unit
  const long long unit = blockIdx.x / cols;
  const int rem = (int)(blockIdx.x - unit * cols) * blockDim.x + threadIdx.x;
  if (rem >= NN) return;
  (void)SBSE_IDX(unit, n_units);
  const int n_orb = DENS ? L : 1;
  for (int ell = 0; ell < n_orb; ++ell) {
    C *base = data + (unit * n_orb + ell) * g.ng + rem;
    C v[N];
#pragma unroll
    for (int z = 0; z < N; ++z) v[z] = base[(long long)z * NN];
    kin_pencil<N>(v, kt);
#pragma unroll
    for (int z = 0; z < N; ++z) base[(long long)z * NN] = v[z];
    if constexpr (DENS) add_density<N, false>(v, a_next + (long long)ell * g.ng + rem, D + threadIdx.x, kZkT, ell == 0);
  }
  if constexpr (DENS) {
    float *db = dens + unit * g.ng + rem;
#pragma unroll 8
    for (int z = 0; z < N; ++z) db[(long long)z * NN] = D[z * kZkT + threadIdx.x];
  }
}

// one (x, y) column of one item: forward z FFT, multiplier, inverse z FFT (thread per column)
template <typename T, int N, bool COH>
__device__ __forceinline__ void zcol_column(const GView<T> &g, C2<T> *data, long long item, int rem,
                                            int mult) {
  using C = C2<T>;
  constexpr int NN = N * N;
  const int y = rem / N, x = rem - y * N;
  C *base = data + item * g.ng + rem;
  C v[N];
#pragma unroll
  for (int z = 0; z < N; ++z) v[z] = ldv<COH>(base + (long long)z * NN);
  fft_reg<T, N, -1, TwP<T>>(v);
  const T inv_ng = T(1) / T(N * N * N);
  if (mult == Z_KINETIC) {
    const C mxy = cscale(cmul(g.kin[x], g.kin[y]), inv_ng);
#pragma unroll
    for (int z = 0; z < N; ++z) v[z] = cmul(v[z], cmul(mxy, g.kin[z]));
  } else if (mult == Z_HOLE_GRID) {
    const T gxy = g.k2[x] + g.k2[y];
#pragma unroll
    for (int z = 0; z < N; ++z) v[z] = cscale(v[z], T(0.5) * (gxy + g.k2[z]) * inv_ng);
  } else {
    const T gxy = g.k2[x] + g.k2[y];
#pragma unroll
    for (int z = 0; z < N; ++z) {
      const T G2 = gxy + g.k2[z];
      v[z] = cscale(v[z], G2 > T(0) ? T(4.0 * M_PI) * inv_ng / G2 : T(0));
    }
  }
  fft_reg<T, N, +1, TwP<T>>(v);
#pragma unroll
  for (int z = 0; z < N; ++z) base[(long long)z * NN] = v[z];
}

template <typename T, int N>
__global__ void __launch_bounds__(128) k_zcol(GView<T> g, C2<T> *data, long long cols_total, int mult) {
  constexpr int NN = N * N;
  const long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= cols_total) return;
  const long long item = c / NN;
  if (mult == Z_HOLE_GRID && (item + 1) * NN == cols_total) mult = Z_POISSON;  // the last slot
  zcol_column<T, N, false>(g, data, item, (int)(c - item * NN), mult);
}

enum PlaneInvMode { PI_PLAIN = 0, PI_POISSON = 1 };

struct PlaneInvArgs {
  long long planes_total;  // planes of all items
  PoissonOut po;           // POISSON
};

// y then x inverse transforms of PPB planes held in shared memory
template <typename T, int N, bool COH = false>
__device__ __forceinline__ void plane_inverse(C2<T> *S, const C2<T> *src_item_plane0, int pl, int q) {
  using C = C2<T>;
  constexpr int LD = N + 1, NN = N * N;
  {
    C v[N];
    const C *col = src_item_plane0 + (long long)pl * NN + q;
#pragma unroll
    for (int y = 0; y < N; ++y) v[y] = ldv<COH>(col + y * N);
    fft_reg<T, N, +1, TwP<T>>(v);
    C *dst = S + pl * N * LD + q;
#pragma unroll
    for (int y = 0; y < N; ++y) dst[y * LD] = v[y];
  }
  __syncthreads();
  {
    C v[N];
    C *row = S + (pl * N + q) * LD;
#pragma unroll
    for (int x = 0; x < N; ++x) v[x] = row[x];
    fft_reg<T, N, +1, TwP<T>>(v);
#pragma unroll
    for (int x = 0; x < N; ++x) row[x] = v[x];
  }
  __syncthreads();
}

// y, x inverse FFTs of the planes z0 .. z0 + PPB - 1 of the L orbitals of `pair`, storing each and
// accumulating the induced density 2 sum_l (2 Re(conj(eta0_l) d_l) + |d_l|^2) (Eq. 11)
template <typename T, int N, bool COH>
__device__ __forceinline__ void inv_density_planes(const GView<T> &g, C2<T> *data, const C2<T> *a_next,
                                                   T *dens, int pair, int L, int z0, C2<T> *S) {
  using C = C2<T>;
  constexpr int PPB = kPPB<T, N>, LD = N + 1, NN = N * N, NT = PPB * N;
  const int pl = threadIdx.x / N, q = threadIdx.x - pl * N;
  T accd[N];
#pragma unroll
  for (int k = 0; k < N; ++k) accd[k] = T(0);
  for (int ell = 0; ell < L; ++ell) {
    const long long item = (long long)pair * L + ell;
    (void)SBSE_IDX((long long)z0 * NN + NN * PPB - 1, g.ng);  // the block's planes inside the item
    C *base = data + item * g.ng + (long long)z0 * NN;
    plane_inverse<T, N, COH>(S, base, pl, q);
    const C *ab = a_next + (long long)ell * g.ng + (long long)z0 * NN;
#pragma unroll
    for (int k = 0; k < N; ++k) {
      const int l = threadIdx.x + k * NT;
      const C dv = S[(threadIdx.x / N) * LD + threadIdx.x % N + k * PPB * LD];
      base[l] = dv;
      const C a0 = ldv<COH>(ab + l);
      accd[k] += density_term<T>(a0, dv);
    }
    __syncthreads();
  }
  T *db = dens + (long long)pair * g.ng + (long long)z0 * NN;
#pragma unroll
  for (int k = 0; k < N; ++k) db[threadIdx.x + k * NT] = accd[k];
}

// y, x inverse FFTs of the PPB planes at plane offset `off` of `item`, stored back in place
template <typename T, int N, bool COH, int PPB = kPPB<T, N>>
__device__ __forceinline__ void inv_plain_planes(const GView<T> &g, C2<T> *data, long long item,
                                                 long long off, C2<T> *S) {
  using C = C2<T>;
  constexpr int LD = N + 1, NT = PPB * N;
  const int pl = threadIdx.x / N, q = threadIdx.x - pl * N;
  C *base = data + item * g.ng + off;
  plane_inverse<T, N, COH>(S, base, pl, q);
#pragma unroll 4
  for (int k = 0; k < N; ++k) {
    const int l = threadIdx.x + k * NT;
    base[l] = S[(threadIdx.x / N) * LD + threadIdx.x % N + k * PPB * LD];
  }
}

template <typename T, int N, int MODE, int PPB = kPPB<T, N>>
__global__ void __launch_bounds__(PPB * N)
    k_plane_inv(GView<T> g, C2<T> *data, T *u_out, T *acc, C2<T> *em1_out, PlaneInvArgs pa) {
  using C = C2<T>;
  constexpr int LD = N + 1, NN = N * N, NT = PPB * N;
  extern __shared__ unsigned char smem_raw[];
  C *S = reinterpret_cast<C *>(smem_raw);
  const int pl = threadIdx.x / N, q = threadIdx.x - pl * N;
  const long long p0 = (long long)blockIdx.x * PPB;  // PPB divides N: all planes of one item
  const long long item = p0 / N;
  const long long off = (p0 - item * N) * NN;
  if (MODE == PI_PLAIN) {
    inv_plain_planes<T, N, false, PPB>(g, data, item, off, S);
    return;
  }
  C *base = data + item * g.ng + off;
  plane_inverse<T, N>(S, base, pl, q);
  // Poisson epilogue: unpack the two real potentials of the item, store u, accumulate the damped
  // time integral and store E - 1; the accumulator loads of a batch are issued together
  const T coef = (T)pa.po.coef, tau = (T)pa.po.tau_next;
  const bool keep = pa.po.keep != 0.0;
  const int n_h = (2 * item + 1 < pa.po.n_out) ? 2 : 1;
  constexpr int UB = 8;
#pragma unroll 1  // code size: the unrolled epilogue missed the instruction cache
  for (int k0 = 0; k0 < N; k0 += UB) {
    C v[UB];
    T old[UB][2];
#pragma unroll
    for (int k = 0; k < UB; ++k) {
      if (k0 + k >= N) break;
      const int l = threadIdx.x + (k0 + k) * NT;
      v[k] = S[(threadIdx.x / N) * LD + threadIdx.x % N + (k0 + k) * PPB * LD];
#pragma unroll
      for (int h = 0; h < 2; ++h)
        old[k][h] = (acc && keep && h < n_h) ? acc[(2 * item + h) * g.ng + off + l] : T(0);
    }
#pragma unroll
    for (int k = 0; k < UB; ++k) {
      if (k0 + k >= N) break;
      const int l = threadIdx.x + (k0 + k) * NT;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        if (h >= n_h) break;
        const T val = h ? v[k].y : v[k].x;
        const long long o = (2 * item + h) * g.ng + off + l;
        if (u_out) u_out[o] = val;
        if (acc) acc[o] = old[k][h] + coef * val;
        if (em1_out) em1_out[o] = phase_em1<T>(val, tau);
      }
    }
  }
}

// grids whose FP32 orbitals take the lane-pair sweeps (fft_split.cu): the persistent step does too
constexpr bool lane_pairs(int N) { return N == 32 || N == 48 || N == 64; }

// ------------------------------------------------------------------------------------------
// Persistent split-operator step: one launch advances the eta0 set and every pair's L orbitals by
// one step of Eq. (10) and writes each pair's induced density. Blocks claim tiles from a host-built
// queue; a tile waits (bounded) for the tiles it reads, whose queue positions are always earlier,
// so every awaited tile is held by a running block and the launch cannot deadlock. The queue
// pipelines pairs (forward tiles of pair j, z tiles of pair j-1, inverse tiles of pair j-2) so that
// the orbitals in flight stay in L2 between the passes (FP32: no z tiles of the pairs; the inverse tiles take
// the z operator).

__device__ __forceinline__ unsigned ld_acquire(const unsigned *p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// bounded wait for *p >= target (`limit` polls ~100 ns apart; the default 2^23 is about a second);
// false on timeout
__device__ __forceinline__ bool wait_geq(const unsigned *p, unsigned target, unsigned limit) {
  for (unsigned i = 0; i < limit; ++i) {
    if (ld_acquire(p) >= target) return true;
    __nanosleep(100);
  }
  return false;
}

// One tile with lane-pair pencils: its PPB planes, or its PPB N columns, in two halves
template <int N>
__device__ __forceinline__ void step_tile_pairs(const GView<float> &g, const XfwdArgs<float> &fa, const XfwdArgs<float> &fp,
                                                float2 *a_next, float2 *d, float *dens, int L, int4 it, float2 *S,
                                                const float2 *tab, const float2 *ztab) {
  using C = float2;
  constexpr int PPB = kPPB<float, N>, NN = N * N, NT = PPB * N, H = N / 2;
  static_assert(PPB % 2 == 0, "two halves of PPB / 2 planes");
  const int grp = threadIdx.x / (2 * N), tid = threadIdx.x - grp * 2 * N;
  if (it.x == SI_A_FWD || it.x == SI_P_FWD) {
#pragma unroll 1
    for (int half = 0; half < 2; ++half) {
      if (half) __syncthreads();
      const long long off = ((long long)it.z * PPB + half * (PPB / 2) + grp) * NN;
      C *tile = S + grp * N * (N + 1);
      if (it.x == SI_P_FWD)
        kin2_plane<N, true>(g, fp, it.y, off, tile, tab, tid);
      else
        kin2_plane<N, false>(g, fa, it.y, off, tile, tab, tid);
    }
    return;
  }
  const bool pair = it.x == SI_P_INV;
  if (!pair && it.x != SI_A_Z) return;
  const int lane = threadIdx.x & 31, s = lane >> 4, cw = (threadIdx.x >> 5) * 16 + (lane & 15);
  float *D = reinterpret_cast<float *>(S) + cw;
#pragma unroll 1
  for (int half = 0; half < 2; ++half) {
    const int rem = it.z * NT + half * (NT / 2) + cw;
    for (int l = 0; l < (pair ? L : 1); ++l) {
      C *base = (pair ? d + ((long long)it.y * L + l) * g.ng : a_next + (long long)it.y * g.ng) + rem;
      C v[H];
#pragma unroll
      for (int m = 0; m < H; ++m) v[m] = __ldcg(base + (long long)(2 * m + s) * NN);
      kin_roundtrip<N>(v, s, ztab);
#pragma unroll
      for (int m = 0; m < H; ++m) base[(long long)(2 * m + s) * NN] = v[m];
      if (pair) {
        const C *ab = a_next + (long long)l * g.ng + rem;
#pragma unroll
        for (int m = 0; m < H; ++m) {
          const float t = density_term<float>(__ldcg(ab + (long long)(2 * m + s) * NN), v[m]);
          float &acc = D[(2 * m + s) * (NT / 2)];
          acc = l ? acc + t : t;
        }
      }
    }
    if (pair)
#pragma unroll 8
      for (int m = 0; m < H; ++m)
        dens[(long long)it.y * g.ng + (long long)(2 * m + s) * NN + rem] = D[(2 * m + s) * (NT / 2)];
  }
}

template <typename T, int N>
__global__ void __launch_bounds__(kPPB<T, N> * N)
    k_step_persistent(GView<T> g, XfwdArgs<T> fa, XfwdArgs<T> fp, C2<T> *a_next, C2<T> *d, T *dens,
                      int L, StepQueue q) {
  using C = C2<T>;
  constexpr int PPB = kPPB<T, N>, NN = N * N, G = N / PPB, NT = PPB * N;
  extern __shared__ unsigned char smem_raw[];
  C *S = reinterpret_cast<C *>(smem_raw);
  __shared__ int4 cur;
  __shared__ int go;
  // FP32 takes the two sweeps of k_plane_kin and k_zkin (SI_A_Z, SI_P_INV: z operator on NT columns),
  // with lane pairs where the sweeps take them
  constexpr bool KIN = sizeof(T) == 4;
  constexpr bool LP = KIN && lane_pairs(N);
  constexpr int NK = LP ? 3 * N / 2 : KIN ? N : 1;
  __shared__ C kt[2 * NK];  // of the planes, and from NK of the z operator (read after the first tile's barrier)
  if constexpr (KIN) {
    for (int i = threadIdx.x; i < NK; i += blockDim.x) {
      kt[i] = g.kin[kin_xy(N) + i];
      kt[NK + i] = g.kin[kin_z(N) + i];
    }
  }
  const unsigned tgt = (q.epoch + 1) * (unsigned)G;
  for (;;) {
    if (threadIdx.x == 0) {
      const unsigned i = atomicAdd(q.claim, 1u) - q.claim_base;
      const int4 it = (i < (unsigned)q.n_items) ? q.items[i] : make_int4(-1, 0, 0, 0);
      bool ok = true;
      if (it.x == SI_A_Z) {
        ok = wait_geq(q.a_fwd + it.y, tgt, q.wait_limit);
      } else if (it.x == SI_A_INV) {
        ok = wait_geq(q.a_z + it.y, tgt, q.wait_limit);
      } else if (it.x == SI_P_Z) {
        ok = wait_geq(q.p_fwd + it.y, tgt, q.wait_limit);
      } else if (it.x == SI_P_INV) {
        ok = wait_geq(q.a_inv, (q.epoch + 1) * (unsigned)(L * G), q.wait_limit);
        const unsigned *before = KIN ? q.p_fwd : q.p_z;
        for (int l = 0; l < L && ok; ++l) ok = wait_geq(before + it.y * L + l, tgt, q.wait_limit);
      }
      if (!ok) atomicExch(q.err, 1);
      __threadfence();
      cur = it;
      go = ok ? 1 : 0;
    }
    __syncthreads();
    const int4 it = cur;
    if (it.x < 0) break;
    if (go) {
      if constexpr (LP) {
        step_tile_pairs<N>(g, fa, fp, a_next, d, dens, L, it, S, kt, kt + NK);
      } else if constexpr (KIN) {
        const int rem = it.z * NT + threadIdx.x;
        switch (it.x) {
          case SI_A_FWD: fwd_planes<T, N, false, PPB, true>(g, fa, it.y, (long long)it.z * PPB * NN, S, kt); break;
          case SI_P_FWD: fwd_planes<T, N, true, PPB, true>(g, fp, it.y, (long long)it.z * PPB * NN, S, kt); break;
          case SI_A_Z:
          case SI_P_INV: {
            const bool pair = it.x == SI_P_INV;
            float *D = reinterpret_cast<float *>(S);
            for (int l = 0; l < (pair ? L : 1); ++l) {
              C *base = (pair ? d + ((long long)it.y * L + l) * g.ng : a_next + (long long)it.y * g.ng) + rem;
              C v[N];
#pragma unroll
              for (int z = 0; z < N; ++z) v[z] = __ldcg(base + (long long)z * NN);
              kin_pencil<N>(v, kt + NK);
#pragma unroll
              for (int z = 0; z < N; ++z) base[(long long)z * NN] = v[z];
              if (pair) add_density<N, true>(v, a_next + (long long)l * g.ng + rem, D + threadIdx.x, NT, l == 0);
            }
            if (pair)
              for (int z = 0; z < N; ++z) dens[(long long)it.y * g.ng + (long long)z * NN + rem] = D[z * NT + threadIdx.x];
            break;
          }
          default: break;
        }
      } else {
        switch (it.x) {
          case SI_A_FWD: fwd_planes<T, N, false>(g, fa, it.y, (long long)it.z * PPB * NN, S); break;
          case SI_P_FWD: fwd_planes<T, N, true>(g, fp, it.y, (long long)it.z * PPB * NN, S); break;
          case SI_A_Z: zcol_column<T, N, true>(g, a_next, it.y, it.z * NT + threadIdx.x, Z_KINETIC); break;
          case SI_P_Z: zcol_column<T, N, true>(g, d, it.y, it.z * NT + threadIdx.x, Z_KINETIC); break;
          case SI_A_INV: inv_plain_planes<T, N, true>(g, a_next, it.y, (long long)it.z * PPB * NN, S); break;
          case SI_P_INV: inv_density_planes<T, N, true>(g, d, a_next, dens, it.y, L, it.z * PPB, S); break;
          default: break;
        }
      }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      __threadfence();
      unsigned *c = nullptr;
      if (it.x == SI_A_FWD) c = q.a_fwd + it.y;
      else if (it.x == SI_A_Z) c = KIN ? q.a_inv : q.a_z + it.y;
      else if (it.x == SI_A_INV) c = q.a_inv;
      else if (it.x == SI_P_FWD) c = q.p_fwd + it.y;
      else if (it.x == SI_P_Z) c = q.p_z + it.y;
      if (c) atomicAdd(c, 1u);
    }
  }
}

// ------------------------------------------------------------------------------------------
// dispatch over the compile-time sizes

template <typename T, int N, bool STEP = false> void set_attrs() {
  const int sm = (int)plane_smem<T, N>();
  if constexpr (STEP) cudaFuncSetAttribute(k_step_persistent<T, N>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm);
  const int sf = (int)few_plane_smem<T, N>();
  constexpr bool few = kFew<T, N> < kPPB<T, N> && few_plane_smem<T, N>() > 48 * 1024;
  auto limit = [](auto *k, int bytes) { cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes); };
  limit(k_plane_fwd<T, N, false, kPPB<T, N>>, sm);
  limit(k_plane_inv<T, N, PI_POISSON>, sm);
  if constexpr (few) limit(k_plane_fwd<T, N, false, kFew<T, N>>, sf);
  if constexpr (sizeof(T) == 4 && !lane_pairs(N)) {
    limit(k_plane_kin<N, false, kPPB<T, N>>, sm);
    limit(k_plane_kin<N, true, fwd_ppb<T, N, true>()>, (int)fwd_smem<T, N, true>());
    if constexpr (few) {
      limit(k_plane_kin<N, false, kFew<T, N>>, sf);
      limit(k_plane_kin<N, true, kFew<T, N>>, sf);
    }
  }
  if constexpr (sizeof(T) == 8) {
    limit(k_plane_fwd<T, N, true, kPPB<T, N>>, sm);
    limit(k_plane_inv<T, N, PI_PLAIN>, sm);
    if constexpr (few) {
      limit(k_plane_fwd<T, N, true, kFew<T, N>>, sf);
      limit(k_plane_inv<T, N, PI_PLAIN, kFew<T, N>>, sf);
    }
  }
}

template <typename T> struct FastOps {
  template <int N>
  static void step(const GridTables<T> &g, const XfwdArgs<T> &fa, const XfwdArgs<T> &fp, C2<T> *a_next,
                   C2<T> *d, T *dens, int L, const StepQueue &q, int grid, cudaStream_t s) {
    if constexpr (!(sizeof(T) == 8 && N > 48)) {
      k_step_persistent<T, N><<<grid, kPPB<T, N> * N, plane_smem<T, N>(), s>>>(view(g), fa, fp, a_next, d,
                                                                              dens, L, q);
    }
  }
  template <int N> static int resident_blocks() {
    if constexpr (!(sizeof(T) == 8 && N > 48)) {
      int per_sm = 0, dev = 0, sms = 0;
      cudaGetDevice(&dev);
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_step_persistent<T, N>, kPPB<T, N> * N,
                                                    plane_smem<T, N>());
      return per_sm * sms;
    }
    return 0;
  }
  template <int N> static int tiles_per_orbital() { return N / kPPB<T, N>; }
  // packing modes, and the FP64 orbitals
  template <int N> static void fwd(const GridTables<T> &g, const XfwdArgs<T> &a, cudaStream_t s) {
    if constexpr (!(sizeof(T) == 8 && N > 48)) {
      const long long planes = (long long)a.n_items * N;
      constexpr int PP = kPPB<T, N>, PF = kFew<T, N>;
      const bool few = few_planes<T, N>(planes);
      const unsigned blocks = (unsigned)(planes / (few ? PF : PP));
      if constexpr (sizeof(T) == 8) {
        if (a.mode == XF_PHASE_PAIR) {
          if (few)
            k_plane_fwd<T, N, true, PF><<<blocks, PF * N, few_plane_smem<T, N>(), s>>>(view(g), a, planes);
          else
            k_plane_fwd<T, N, true, PP><<<blocks, PP * N, plane_smem<T, N>(), s>>>(view(g), a, planes);
          return;
        }
      }
      if (few)
        k_plane_fwd<T, N, false, PF><<<blocks, PF * N, few_plane_smem<T, N>(), s>>>(view(g), a, planes);
      else
        k_plane_fwd<T, N, false, PP><<<blocks, PP * N, plane_smem<T, N>(), s>>>(view(g), a, planes);
    }
  }
  // the two sweeps of the FP32 orbitals
  template <int N> static void kin(const GridTables<T> &g, const XfwdArgs<T> &a, cudaStream_t s) {
    if constexpr (sizeof(T) == 4 && !lane_pairs(N)) {
      const long long planes = (long long)a.n_items * N;
      constexpr int P2 = fwd_ppb<T, N, true>(), PP = kPPB<T, N>, PF = kFew<T, N>;
      const bool pair = a.mode == XF_PHASE_PAIR;
      if (few_planes<T, N>(planes)) {
        const unsigned blocks = (unsigned)(planes / PF);
        if (pair) k_plane_kin<N, true, PF><<<blocks, PF * N, few_plane_smem<T, N>(), s>>>(view(g), a, planes);
        else k_plane_kin<N, false, PF><<<blocks, PF * N, few_plane_smem<T, N>(), s>>>(view(g), a, planes);
      } else if (pair) {
        k_plane_kin<N, true, P2><<<(unsigned)(planes / P2), P2 * N, fwd_smem<T, N, true>(), s>>>(view(g), a, planes);
      } else {
        k_plane_kin<N, false, PP><<<(unsigned)(planes / PP), PP * N, plane_smem<T, N>(), s>>>(view(g), a, planes);
      }
    }
  }
  template <int N>
  static void zkin(const GridTables<T> &g, C2<T> *d, int n_items, const C2<T> *a_next, int L, T *dens, cudaStream_t s) {
    if constexpr (sizeof(T) == 4 && !lane_pairs(N)) {
      constexpr long long per_unit = (N * N + kZkT - 1) / kZkT;
      // the density summed in the sweep needs one block per pair and 128 columns, working through L orbitals
      // in turn: below two blocks per SM a second kernel sums it from the stored orbitals
      if (dens && n_items / L * per_unit >= 2 * kSMs) {
        k_zkin<N, true><<<(unsigned)(n_items / L * per_unit), kZkT, 0, s>>>(view(g), d, a_next, dens, n_items / L, L);
        return;
      }
      const int nt = n_items * per_unit < kSMs ? 32 : kZkT;
      k_zkin<N, false><<<(unsigned)((long long)n_items * ((N * N + nt - 1) / nt)), nt, 0, s>>>(view(g), d, nullptr, nullptr,
                                                                                          n_items, 1);
      if (dens) launch_density<float>(g, d, a_next, n_items / L, L, dens, s);
    }
  }
  template <int N> static void z(const GridTables<T> &g, C2<T> *d, int n_items, int mult, cudaStream_t s) {
    if constexpr (!(sizeof(T) == 8 && N > 48)) {
      // threads per block: 128, or one warp where 128 would leave SMs without a block
      const long long cols = (long long)n_items * N * N;
      const int nt = cols < 128ll * kSMs ? 32 : 128;
      k_zcol<T, N><<<(unsigned)((cols + nt - 1) / nt), nt, 0, s>>>(view(g), d, cols, mult);
    }
  }
  // mode: PI_PLAIN (FP64 orbitals) or PI_POISSON
  template <int N>
  static void inv(const GridTables<T> &g, C2<T> *d, int n_items, T *u_out, T *acc, C2<T> *em1_out, const PoissonOut &po,
                  int mode, cudaStream_t s) {
    if constexpr (!(sizeof(T) == 8 && N > 48)) {
      const PlaneInvArgs pa{(long long)n_items * N, po};
      constexpr int PP = kPPB<T, N>, PF = kFew<T, N>;
      const unsigned blocks = (unsigned)(pa.planes_total / PP);
      if constexpr (sizeof(T) == 8) {
        if (mode == PI_PLAIN) {
          if (few_planes<T, N>(pa.planes_total))
            k_plane_inv<T, N, PI_PLAIN, PF><<<(unsigned)(pa.planes_total / PF), PF * N, few_plane_smem<T, N>(), s>>>(
                view(g), d, nullptr, nullptr, nullptr, pa);
          else
            k_plane_inv<T, N, PI_PLAIN><<<blocks, PP * N, plane_smem<T, N>(), s>>>(view(g), d, nullptr, nullptr, nullptr, pa);
          return;
        }
      }
      k_plane_inv<T, N, PI_POISSON><<<blocks, PP * N, plane_smem<T, N>(), s>>>(view(g), d, u_out, acc, em1_out, pa);
    }
  }
};

}  // namespace

}  // namespace sbse
