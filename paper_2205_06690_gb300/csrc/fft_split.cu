// Lane-pair passes (FP32). N = 80 and 96: the split-operator step of Eq. (10), the Poisson solves of
// Eq. (11) / q_ij and the exchange potentials of Eq. (1) on the paper-scale grids (the 520-electron
// system of Sec. III sits on ~0.85M points, 96^3 here). N = 32, 48 and 64: the split-operator step.
//
// A pencil of N points is too long for one thread's registers next to the epilogue's state (80, 96), or
// leaves room for too few warps to hide the loads (48: 12 warps per SM), so it is split over a lane pair (l, l ^ 16) of one warp: N = 2H, each lane holds H points, transforms
// them with the register FFT of length H, and one radix-2 butterfly across the pair (operands
// swapped by warp shuffles) completes the transform. Forward transforms take the pencil
// interleaved (lane s holds x[2m + s]) and return it in two quarter blocks (decimation in time);
// inverse transforms take the blocks and return the interleaved order (decimation in frequency),
// so no pass needs a reordering step. A warp transforms 16 pencils; 16 consecutive lanes always
// touch 16 consecutive grid points or rows of a padded shared-memory tile (conflict-free, 128-byte
// global segments).
//
// The split-operator step (Eq. 10) takes two sweeps over the orbitals: the kinetic propagator is
// the product of three one-dimensional operators (one per axis), so
//   plane kinetic : one z-plane per block (2N threads): fused pre-operation (potential phase), the
//                   x and then the y operator (forward FFT, exp(-i dt k^2 / 2) / N, inverse FFT)
//   z kinetic     : 16 columns per warp: the z operator, and for the pair batch the induced density
//                   of the pair's L orbitals (Eq. 11)
// The Poisson solves (4 pi / |G|^2 does not factor over the axes) keep the 3D round trip:
//   plane forward : pre-operation (packing), x FFTs in the padded tile, y FFTs stored to global
//   z columns     : forward z FFT, 4 pi / |G|^2 with 1/N^3, inverse z FFT
//   plane inverse : y then x inverse FFTs, then the unpacking with the damped time-integral
//                   accumulation of Eq. (13) and E - 1 of the next step
// Blocks are ordered plane-major (plane outer, item inner), so the tables read beside the orbitals
// (eta0 of each stochastic orbital, the potential phases, E - 1 of each pair) are the same z-slice
// for consecutive blocks and stay in L2 even when the whole table set does not fit there.
#include "fft_pair.cuh"

namespace sbse {

namespace {

template <int N> constexpr size_t split_smem() { return (size_t)N * (N + 1) * sizeof(float2); }
template <int N> constexpr size_t split_density_smem() { return split_smem<N>() + (size_t)N * N * sizeof(float); }

// ------------------------------------------------------------------------------------------
// plane forward pass of the three-pass round trip (Poisson packing of densities and pair
// products): block = (plane z, item), 2N threads; x FFTs in the tile, y FFTs stored to global

template <int N>
__global__ void __launch_bounds__(2 * N, N == 96 ? 2 : 3) k_plane_fwd2(GView<float> g, XfwdArgs<float> a, int n_items) {
  using C = float2;
  constexpr int LD = N + 1, NN = N * N, H = N / 2, Q = H / 2;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C *S = reinterpret_cast<C *>(smem_raw);
  const int z = (int)(blockIdx.x / (unsigned)n_items);
  const long long item = (long long)blockIdx.x - (long long)z * n_items;
  const long long off = (long long)z * NN;
  preop_plane<N, false>(g, a, item, off, S, threadIdx.x);
  __syncthreads();
  const int lane = threadIdx.x & 31, s = lane >> 4, p = (threadIdx.x >> 5) * 16 + (lane & 15);
  {  // x transforms, pencil p = row p of the tile, in place
    C v[H];
    C *row = S + p * LD;
#pragma unroll
    for (int m = 0; m < H; ++m) v[m] = row[2 * m + s];
    fft2_dit<N, -1>(v, s);
    __syncwarp();
#pragma unroll
    for (int j = 0; j < Q; ++j) {
      row[s * Q + j] = v[j];
      row[H + s * Q + j] = v[Q + j];
    }
  }
  __syncthreads();
  {  // y transforms, pencil p = column p, stored to global
    C v[H];
    const C *col = S + p;
#pragma unroll
    for (int m = 0; m < H; ++m) v[m] = col[(2 * m + s) * LD];
    fft2_dit<N, -1>(v, s);
    (void)SBSE_IDX(off + p + (long long)(N - 1) * N, g.ng);
    C *out = a.out + item * g.ng + off + p;
#pragma unroll
    for (int j = 0; j < Q; ++j) {
      out[(s * Q + j) * N] = v[j];
      out[(H + s * Q + j) * N] = v[Q + j];
    }
  }
}

// ------------------------------------------------------------------------------------------
// First sweep of the two-sweep split-operator step. The kinetic propagator of Eq. (10) is
// exp(-i dt |G|^2 / 2) = prod_axes exp(-i dt k_a^2 / 2), so in real space it is the product of three
// one-dimensional operators F_a^-1 K_a F_a, one per axis, which commute. This pass applies the
// potential phase (the pre-operation) and the x and y operators to one z-plane held in shared
// memory (kin_roundtrip along each axis); the second sweep applies the z operator. One HBM round trip
// per sweep: two per step instead of the three of a 3D FFT round trip. 36 pairs of 48^3 x 10 orbitals:
// 160 + 119 us (three thread-per-pencil sweeps: 147 + 113 + 113; the same two sweeps with a thread per pencil:
// 208 + 157, held by 12 warps per SM); 10 pairs of 32^3: 14.1 us for the planes.

// Mixed grids that took three thread-per-pencil sweeps before and two since (W of 10 pairs x 10 orbitals, three
// against two): 20^3 6.5 -> 4.1 ms per 100 steps, 24^3 7.1 -> 4.6, 40^3 (streamed before) 13.1 -> 11.2; with lane
// pairs 32^3 8.0 -> 5.5, 64^3 46.8 -> 33.4.

// blocks per SM that the registers should allow: N points of a lane pair per thread pair
constexpr int kin2_blocks(int N) { return N == 96 ? 2 : N == 80 ? 3 : N == 64 ? 5 : N == 48 ? 8 : 12; }

template <int N, bool PAIR>
__global__ void __launch_bounds__(2 * N, kin2_blocks(N)) k_plane_kin2(GView<float> g, XfwdArgs<float> a, int n_items) {
  constexpr int NN = N * N, H = N / 2;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int z = (int)(blockIdx.x / (unsigned)n_items);
  const long long item = (long long)blockIdx.x - (long long)z * n_items;
  __shared__ float2 tab[3 * H];
  for (int i = threadIdx.x; i < 3 * H; i += blockDim.x) tab[i] = g.kin[kin_xy(N) + i];
  kin2_plane<N, PAIR>(g, a, item, (long long)z * NN, reinterpret_cast<float2 *>(smem_raw), tab, threadIdx.x);
}

// Second sweep: the z operator on 64 columns of one item (PLAIN) or of each of the L orbitals of a
// pair (DENS), which also sums the pair's induced density 2 sum_l (2 Re(conj(eta0_l) d_l) +
// |d_l|^2) (Eq. 11) in shared memory and writes it.
constexpr int kZDPitch = 80;  // density rows of 64 columns padded so the two half-warps miss each other's banks

template <int N, bool DENS>
__global__ void __launch_bounds__(128, N >= 80 ? 3 : DENS || N == 64 ? 4 : 6) k_zkin2(GView<float> g, float2 *data, const float2 *a_next, float *dens,
                                                  int n_units, int L) {
  using C = float2;
  constexpr int NN = N * N, H = N / 2, UB = 16;
  __shared__ float D[DENS ? N * kZDPitch : 1];
  __shared__ C tab[3 * H];
  for (int i = threadIdx.x; i < 3 * H; i += blockDim.x) tab[i] = g.kin[kin_z(N) + i];
  __syncthreads();
  const int cs = (int)(blockIdx.x / (unsigned)n_units);
  const int unit = (int)blockIdx.x - cs * n_units;
  const int lane = threadIdx.x & 31, s = lane >> 4, cw = (threadIdx.x >> 5) * 16 + (lane & 15);
  const int rem = cs * 64 + cw;
  const int n_orb = DENS ? L : 1;
  (void)SBSE_IDX(rem, NN);
  for (int ell = 0; ell < n_orb; ++ell) {
    const long long item = DENS ? (long long)unit * L + ell : unit;
    (void)SBSE_IDX(item, (long long)n_units * n_orb);
    C *base = data + item * g.ng + rem;
    C v[H];
#pragma unroll
    for (int m = 0; m < H; ++m) v[m] = base[(long long)(2 * m + s) * NN];
    kin_roundtrip<N>(v, s, tab);
#pragma unroll
    for (int m = 0; m < H; ++m) base[(long long)(2 * m + s) * NN] = v[m];
    if constexpr (DENS) {
      const C *ab = a_next + (long long)ell * g.ng + rem;
#pragma unroll
      for (int m0 = 0; m0 < H; m0 += UB) {
        C a0[UB];
#pragma unroll
        for (int k = 0; k < UB; ++k)
          if (m0 + k < H) a0[k] = ab[(long long)(2 * (m0 + k) + s) * NN];
#pragma unroll
        for (int k = 0; k < UB; ++k) {
          if (m0 + k < H) {
            const C dv = v[m0 + k];
            const float t = density_term<float>(a0[k], dv);
            float &acc = D[(2 * (m0 + k) + s) * kZDPitch + cw];
            acc = ell ? acc + t : t;
          }
        }
        // keep the loads of the next batch below this one (hoisting them all costs registers)
        asm volatile("" ::: "memory");
      }
    }
  }
  if constexpr (DENS) {
    float *db = dens + (long long)unit * g.ng + rem;
#pragma unroll 8
    for (int m = 0; m < H; ++m) db[(long long)(2 * m + s) * NN] = D[(2 * m + s) * kZDPitch + cw];
  }
}

// The same sweep for the pair batch with the columns of the next orbital staged in shared memory
// by one bulk tensor copy (N z-rows x ZT_CW columns) while the current orbital is transformed, so
// the column loads no longer stall the warps. ZT_CW = 32 columns (two warps) per block keep the
// stage (24 KB at N = 96) and the density rows small enough for five blocks per SM.
constexpr int kZtCw = 32;
constexpr int kZtPitch = kZtCw + 16;  // density rows: the two half-warps' rows fall on different banks

// dynamic shared memory of the staged z sweep: the stage and the density rows, plus the slack that
// lets the kernel start the stage on a 128-byte boundary (the alignment a tensor copy's shared
// destination needs; the dynamic region itself follows the static variables)
constexpr unsigned kZtAlign = 128;
template <int N> constexpr size_t ztma_smem() {
  return (size_t)N * kZtCw * sizeof(float2) + (size_t)N * kZtPitch * sizeof(float) + kZtAlign;
}

__device__ __forceinline__ void tma_load_3d(void *dst, const CUtensorMap *map, int x, int y, int z, uint64_t *bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(
          tma_smem_addr(dst)),
      "l"((uint64_t)(uintptr_t)map), "r"(x), "r"(y), "r"(z), "r"(tma_smem_addr(bar))
      : "memory");
}

template <int N>
__global__ void __launch_bounds__(2 * kZtCw, N >= 80 ? 5 : N == 64 ? 7 : 10)
    k_zkin2_tma(const __grid_constant__ CUtensorMap dmap, GView<float> g, float2 *data, const float2 *a_next,
                float *dens, int n_units, int L, int *err) {
  using C = float2;
  constexpr int NN = N * N, H = N / 2, UB = N >= 80 ? 48 : N / 2;
  constexpr unsigned kStage = (unsigned)N * kZtCw * sizeof(C);
  extern __shared__ __align__(16) unsigned char smem_raw[];
  unsigned char *smem = smem_raw + ((kZtAlign - (tma_smem_addr(smem_raw) & (kZtAlign - 1))) & (kZtAlign - 1));
  C *St = reinterpret_cast<C *>(smem);                    // [z][column], 128-byte aligned
  float *D = reinterpret_cast<float *>(smem + kStage);    // [z][kZtPitch]
  __shared__ C tab[3 * H];
  __shared__ __align__(8) uint64_t bar;
  const int cs = (int)(blockIdx.x / (unsigned)n_units);
  const int unit = (int)blockIdx.x - cs * n_units;
  const long long item0 = (long long)unit * L;
  if (tma_smem_addr(St) & (kZtAlign - 1)) {  // never expected: report instead of issuing the copy
    if (threadIdx.x == 0) atomicExch(err, 1);
    return;
  }
  if (threadIdx.x == 0) {
    tma_bar_init(&bar, 1);
    tma_bar_expect(&bar, kStage);
    tma_load_3d(St, &dmap, 2 * cs * kZtCw, 0, (int)item0, &bar);
  }
  for (int i = threadIdx.x; i < 3 * H; i += blockDim.x) tab[i] = g.kin[kin_z(N) + i];
  __syncthreads();
  const int lane = threadIdx.x & 31, s = lane >> 4, cw = (threadIdx.x >> 5) * 16 + (lane & 15);
  const int rem = cs * kZtCw + cw;
  (void)SBSE_IDX(rem, NN);
  (void)SBSE_IDX(item0 + L - 1, (long long)n_units * L);
  int failed = -1;  // the orbital whose copy did not land in time
  for (int ell = 0; ell < L; ++ell) {
    if (!__syncthreads_and(tma_bar_wait(&bar, (unsigned)(ell & 1)))) {
      failed = ell;
      break;
    }
    C v[H];
#pragma unroll
    for (int m = 0; m < H; ++m) v[m] = St[(2 * m + s) * kZtCw + cw];
    __syncthreads();  // every thread holds its columns: the stage can take the next orbital
    if (threadIdx.x == 0 && ell + 1 < L) {
      tma_fence_proxy();
      tma_bar_expect(&bar, kStage);
      tma_load_3d(St, &dmap, 2 * cs * kZtCw, 0, (int)(item0 + ell + 1), &bar);
    }
    kin_roundtrip<N>(v, s, tab);
    C *base = data + (item0 + ell) * g.ng + rem;
#pragma unroll
    for (int m = 0; m < H; ++m) base[(long long)(2 * m + s) * NN] = v[m];
    const C *ab = a_next + (long long)ell * g.ng + rem;
#pragma unroll
    for (int m0 = 0; m0 < H; m0 += UB) {
      C a0[UB];
#pragma unroll
      for (int k = 0; k < UB; ++k)
        if (m0 + k < H) a0[k] = ab[(long long)(2 * (m0 + k) + s) * NN];
#pragma unroll
      for (int k = 0; k < UB; ++k) {
        if (m0 + k < H) {
          const C dv = v[m0 + k];
          const float t = density_term<float>(a0[k], dv);
          float &acc = D[(2 * (m0 + k) + s) * kZtPitch + cw];
          acc = ell ? acc + t : t;
        }
      }
      asm volatile("" ::: "memory");
    }
  }
  if (failed >= 0) {
    if (threadIdx.x == 0) {
      atomicExch(err, 1);
      tma_bar_wait(&bar, (unsigned)(failed & 1));  // the copy still in flight: a bounded chance to land
    }
    __syncthreads();
    return;
  }
  __syncthreads();
  float *db = dens + (long long)unit * g.ng + rem;
#pragma unroll 8
  for (int m = 0; m < H; ++m) db[(long long)(2 * m + s) * NN] = D[(2 * m + s) * kZtPitch + cw];
}

// ------------------------------------------------------------------------------------------
// z columns: 64 columns per block of 128 threads (NN is a multiple of 64 for N = 80, 96)

template <int N>
__global__ void __launch_bounds__(128, 4) k_zcol2(GView<float> g, float2 *data, int mult, int n_items) {
  using C = float2;
  constexpr int NN = N * N, H = N / 2, Q = H / 2;
  const int lane = threadIdx.x & 31, s = lane >> 4;
  const long long c = (long long)blockIdx.x * 64 + (threadIdx.x >> 5) * 16 + (lane & 15);
  const long long item = c / NN;
  const int rem = (int)(c - item * NN), y = rem / N, x = rem - y * N;
  (void)SBSE_IDX(item, n_items);
  C *base = data + item * g.ng + rem;
  C v[H];
#pragma unroll
  for (int m = 0; m < H; ++m) v[m] = base[(long long)(2 * m + s) * NN];
  fft2_dit<N, -1>(v, s);
  const float inv_ng = 1.f / (float)(N * N * N);
  if (mult == Z_KINETIC) {
    const C mxy = cscale(cmul(g.kin[x], g.kin[y]), inv_ng);
#pragma unroll
    for (int j = 0; j < Q; ++j) {
      v[j] = cmul(v[j], cmul(mxy, g.kin[s * Q + j]));
      v[Q + j] = cmul(v[Q + j], cmul(mxy, g.kin[H + s * Q + j]));
    }
  } else {
    const float gxy = g.k2[x] + g.k2[y];
#pragma unroll
    for (int j = 0; j < Q; ++j) {
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const float G2 = gxy + g.k2[h * H + s * Q + j];
        const float f = G2 > 0.f ? float(4.0 * M_PI) * inv_ng / G2 : 0.f;
        v[h * Q + j] = cscale(v[h * Q + j], f);
      }
    }
  }
  fft2_dif<N, +1>(v, s);
#pragma unroll
  for (int m = 0; m < H; ++m) base[(long long)(2 * m + s) * NN] = v[m];
}

// ------------------------------------------------------------------------------------------
// plane inverse pass of the Poisson round trip: block = (plane z, packed slot). y then x inverse
// FFTs of the plane, then the epilogue: the two real potentials of the slot, u, the damped time
// integral of Eq. (13) and E - 1 for the next step.

template <int N>
__global__ void __launch_bounds__(2 * N, N == 96 ? 2 : 3) k_plane_inv2(GView<float> g, float2 *data, float *u_out,
                                                                       float *acc, float2 *em1_out, int n_units,
                                                                       PoissonOut po) {
  using C = float2;
  constexpr int LD = N + 1, NN = N * N, NT = 2 * N, H = N / 2, Q = H / 2, KP = NN / NT;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C *S = reinterpret_cast<C *>(smem_raw);
  const int z = (int)(blockIdx.x / (unsigned)n_units);
  const long long item = (long long)blockIdx.x - (long long)z * n_units;
  const long long off = (long long)z * NN;
  const int lane = threadIdx.x & 31, s = lane >> 4, p = (threadIdx.x >> 5) * 16 + (lane & 15);
  (void)SBSE_IDX(off + p + (long long)(N - 1) * N, g.ng);
  (void)SBSE_IDX(2 * item + 1, 2ll * n_units);  // the slot's two densities
  {  // y inverse FFTs from global (frequency blocks) into the tile (interleaved rows)
    C v[H];
    const C *col = data + item * g.ng + off + p;
#pragma unroll
    for (int j = 0; j < Q; ++j) {
      v[j] = col[(s * Q + j) * N];
      v[Q + j] = col[(H + s * Q + j) * N];
    }
    fft2_dif<N, +1>(v, s);
#pragma unroll
    for (int m = 0; m < H; ++m) S[(2 * m + s) * LD + p] = v[m];
  }
  __syncthreads();
  {  // x inverse FFTs in the tile
    C v[H];
    C *row = S + p * LD;
#pragma unroll
    for (int j = 0; j < Q; ++j) {
      v[j] = row[s * Q + j];
      v[Q + j] = row[H + s * Q + j];
    }
    fft2_dif<N, +1>(v, s);
    __syncwarp();
#pragma unroll
    for (int m = 0; m < H; ++m) row[2 * m + s] = v[m];
  }
  __syncthreads();
  const float coef = (float)po.coef, tau = (float)po.tau_next;
  const bool keep = po.keep != 0.0;
  const int n_h = (2 * item + 1 < po.n_out) ? 2 : 1;
  const int y0 = threadIdx.x / N;
  const C *srow = S + y0 * LD + (threadIdx.x - y0 * N);
  constexpr int UB = 8;
#pragma unroll 1
  for (int k0 = 0; k0 < KP; k0 += UB) {
    C v[UB];
    float old[UB][2];
#pragma unroll
    for (int k = 0; k < UB; ++k) {
      if (k0 + k >= KP) break;
      const int l = threadIdx.x + (k0 + k) * NT;
      v[k] = srow[2 * (k0 + k) * LD];
#pragma unroll
      for (int h = 0; h < 2; ++h)
        old[k][h] = (acc && keep && h < n_h) ? acc[(2 * item + h) * g.ng + off + l] : 0.f;
    }
#pragma unroll
    for (int k = 0; k < UB; ++k) {
      if (k0 + k >= KP) break;
      const int l = threadIdx.x + (k0 + k) * NT;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        if (h >= n_h) break;
        const float val = h ? v[k].y : v[k].x;
        const long long o = (2 * item + h) * g.ng + off + l;
        if (u_out) u_out[o] = val;
        if (acc) acc[o] = old[k][h] + coef * val;
        if (em1_out) em1_out[o] = phase_em1<float>(val, tau);
      }
    }
  }
}

template <int N> void set_split_attrs() {
  const int sm = (int)split_smem<N>();
  if constexpr (N >= 80) {
    cudaFuncSetAttribute(k_plane_fwd2<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm);
    cudaFuncSetAttribute(k_plane_inv2<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm);
  }
  cudaFuncSetAttribute(k_plane_kin2<N, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm);
  cudaFuncSetAttribute(k_plane_kin2<N, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm);
}

template <int N> void fwd2(const GridTables<float> &g, const XfwdArgs<float> &a, cudaStream_t s) {
  k_plane_fwd2<N><<<(unsigned)a.n_items * N, 2 * N, split_smem<N>(), s>>>(view(g), a, a.n_items);
}

template <int N> void kin2(const GridTables<float> &g, const XfwdArgs<float> &a, cudaStream_t s) {
  const unsigned blocks = (unsigned)a.n_items * N;
  if (a.mode == XF_PHASE_PAIR)
    k_plane_kin2<N, true><<<blocks, 2 * N, split_smem<N>(), s>>>(view(g), a, a.n_items);
  else
    k_plane_kin2<N, false><<<blocks, 2 * N, split_smem<N>(), s>>>(view(g), a, a.n_items);
}

template <int N> void zcol2(const GridTables<float> &g, float2 *d, int n_items, int mult, cudaStream_t s) {
  static_assert((N * N) % 64 == 0, "z pass blocks hold 64 whole columns");
  const unsigned blocks = (unsigned)((long long)n_items * N * N / 64);
  k_zcol2<N><<<blocks, 128, 0, s>>>(view(g), d, mult, n_items);
}

template <int N>
void zkin2(const GridTables<float> &g, float2 *d, int n_items, const float2 *a_next, int L, float *dens,
           cudaStream_t s, int *err) {
  const int units = dens ? n_items / L : n_items;
  if (dens && (long long)units * (N * N / kZtCw) < 4 * kSMs) {
    // a block works through its pair's L orbitals in turn: where that leaves most of the SMs' schedulers
    // without a warp, a second kernel sums the density from the stored orbitals (10 pairs x 4 orbitals of 32^3:
    // 5.5 + 5.7 us; 36 pairs of 48^3 take 119 us in one sweep)
    k_zkin2<N, false><<<(unsigned)n_items * (N * N / 64), 128, 0, s>>>(view(g), d, nullptr, nullptr, n_items, 1);
    launch_density<float>(g, d, a_next, units, L, dens, s);
    return;
  }
  if (dens && err) {
    // d as n_items orbitals x N z-planes x 2 N^2 floats; boxes of 2 ZT_CW floats x N planes x 1
    CUtensorMap map;
    const uint64_t dims[3] = {(uint64_t)2 * N * N, (uint64_t)N, (uint64_t)n_items};
    const uint64_t strides[2] = {(uint64_t)N * N * sizeof(float2), (uint64_t)g.ng * sizeof(float2)};
    const uint32_t box[3] = {2u * kZtCw, (uint32_t)N, 1u};
    if (make_tensor_map_f32(&map, d, 3, dims, strides, box, false)) {
      raise_smem_limit((const void *)k_zkin2_tma<N>, ztma_smem<N>());
      const unsigned blocks = (unsigned)units * (N * N / kZtCw);
      k_zkin2_tma<N><<<blocks, 2 * kZtCw, ztma_smem<N>(), s>>>(map, view(g), d, a_next, dens, units, L, err);
      return;
    }
  }
  const unsigned blocks = (unsigned)units * (N * N / 64);
  if (dens)
    k_zkin2<N, true><<<blocks, 128, 0, s>>>(view(g), d, a_next, dens, units, L);
  else
    k_zkin2<N, false><<<blocks, 128, 0, s>>>(view(g), d, nullptr, nullptr, units, 1);
}

template <int N>
void inv2(const GridTables<float> &g, float2 *d, int n_units, float *u_out, float *acc, float2 *em1_out,
          const PoissonOut &po, cudaStream_t s) {
  k_plane_inv2<N><<<(unsigned)n_units * N, 2 * N, split_smem<N>(), s>>>(view(g), d, u_out, acc, em1_out, n_units,
                                                                      po);
}

}  // namespace

bool split_size(int N) { return N == 80 || N == 96; }
bool pair_size(int N) { return N == 32 || N == 48 || N == 64; }

int upload_split_twiddles() { return upload_pair_twiddles(); }

void init_split_kernels() {
  set_split_attrs<32>();
  set_split_attrs<48>();
  set_split_attrs<64>();
  set_split_attrs<80>();
  set_split_attrs<96>();
}

void launch_plane_fwd2(const GridTables<float> &g, const XfwdArgs<float> &a, cudaStream_t s) {
  if (g.N == 80) fwd2<80>(g, a, s);
  else if (g.N == 96) fwd2<96>(g, a, s);
}

void launch_zcol2(const GridTables<float> &g, float2 *d, int n_items, int mult, cudaStream_t s) {
  if (g.N == 80) zcol2<80>(g, d, n_items, mult, s);
  else if (g.N == 96) zcol2<96>(g, d, n_items, mult, s);
}

void launch_plane_inv2_poisson(const GridTables<float> &g, float2 *d, int n_slots, const PoissonOut &po,
                               float *u_out, float *acc, float2 *em1_out, cudaStream_t s) {
  if (g.N == 80) inv2<80>(g, d, n_slots, u_out, acc, em1_out, po, s);
  else if (g.N == 96) inv2<96>(g, d, n_slots, u_out, acc, em1_out, po, s);
}

#define SBSE_PAIR_SWITCH(N, CALL) \
  switch (N) {                    \
    case 32: CALL(32); break;     \
    case 48: CALL(48); break;     \
    case 64: CALL(64); break;     \
    case 80: CALL(80); break;     \
    case 96: CALL(96); break;     \
    default: break;               \
  }

void launch_plane_kin2(const GridTables<float> &g, const XfwdArgs<float> &a, cudaStream_t s) {
#define SBSE_CALL(n) kin2<n>(g, a, s)
  SBSE_PAIR_SWITCH(g.N, SBSE_CALL)
#undef SBSE_CALL
}

void launch_zkin2(const GridTables<float> &g, float2 *d, int n_items, const float2 *a_next, int L, float *dens,
                  cudaStream_t s, int *err) {
#define SBSE_CALL(n) zkin2<n>(g, d, n_items, a_next, L, dens, s, err)
  SBSE_PAIR_SWITCH(g.N, SBSE_CALL)
#undef SBSE_CALL
}

}  // namespace sbse
