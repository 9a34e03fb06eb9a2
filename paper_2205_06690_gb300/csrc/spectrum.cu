// Absorption spectrum of the exciton matrix A by a Chebyshev expansion (Sec. II.C, electron-hole
// basis: the paragraph after Eq. 18): sigma(omega) = omega <f0| delta_s(A - omega) |f0> with the
// dipole start vector f0_ia = <phi_a| x |phi_i>, so that only the residues R_n = <f0|T_n(A~)|f0> of
// repeated applications of the scaled A are needed.
//
//   dipoles   : one block per (i, a), FP64 grid sum with x measured from the box centre
//   scaling   : Gershgorin bounds [lo, hi] of A, A~ = (A - c) / w, c = (lo + hi) / 2,
//               w = 1.01 (hi - lo) / 2
//   recursion : v_0 = f0, v_1 = A~ f0, v_{n+1} = 2 A~ v_n - v_{n-1} (one cooperative launch, a warp
//               per row of A), then R_n = f0 . v_n
//   spectrum  : with K = n_terms Chebyshev-Gauss nodes x_k = cos(pi (k + 1/2) / K),
//               D_k = sum_n (2 - delta_n0) R_n T_n(x_k) and
//               sigma(omega) = omega / K sum_k G_s(c + w x_k - omega) D_k, G_s a normalised Gaussian.
// Everything is FP64 (A is FP64 in both precision modes).
#include <math.h>

#include "gemm_nt.cuh"
#include "kernels.h"

namespace sbse {

namespace {

constexpr int kSpT = 256;

__device__ __forceinline__ double block_sum_fixed(double v, double *red) {
  red[threadIdx.x] = v;
  __syncthreads();
  for (int w = blockDim.x / 2; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
    __syncthreads();
  }
  const double s = red[0];
  __syncthreads();
  return s;
}

// f0[i n_c + a] = dV sum_r phi_c[a](r) x(r) phi_o[i](r)
__global__ void __launch_bounds__(kSpT)
    k_dipole(const double *phi_o, const double *phi_c, int n_c, int N, double h, double box, int axis, double dV,
             double *f0) {
  __shared__ double red[kSpT];
  const int i = blockIdx.x / n_c, a = blockIdx.x - i * n_c;
  const long long ng = (long long)N * N * N;
  const double *pi = phi_o + (long long)i * ng, *pa = phi_c + (long long)a * ng;
  // coordinates from a table: two FP64 instructions per point instead of five (511 -> 247 us for 512
  // pairs on 48^3)
  extern __shared__ double xs[];
  for (int i = threadIdx.x; i < N; i += kSpT) xs[i] = h * (double)i - 0.5 * box;
  __syncthreads();
  double s = 0.0;
  const int NN = N * N;
#pragma unroll 4
  for (int r = threadIdx.x; r < (int)ng; r += kSpT) {
    const int idx = axis == 0 ? r % N : (axis == 1 ? (r / N) % N : r / NN);
    s = fma(pi[r], pa[r] * xs[idx], s);
  }
  s = block_sum_fixed(s, red);
  if (threadIdx.x == 0) f0[blockIdx.x] = s * dV;
}

// a vector entry as it is stored: every NaN as the one with this payload, so that none equals kUnset
constexpr unsigned long long kUnset = ~0ull;
__device__ __forceinline__ double entry(double v) { return v == v ? v : __longlong_as_double(0x7ff8000000000000ll); }

// cw = {c, w} from the Gershgorin discs of the rows of A (a warp per row), and v_0 = f0
constexpr int kInitT = 1024;
__global__ void __launch_bounds__(kInitT) k_cheb_init(const double *A, int n, const double *f0, double *cw, double *v0) {
  __shared__ double slo[kInitT / 32], shi[kInitT / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  double lo = INFINITY, hi = -INFINITY;
  for (int r = warp; r < n; r += kInitT / 32) {
    double rad = 0.0;
    for (int j = lane; j < n; j += 32)
      if (j != r) rad += fabs(A[(long long)r * n + j]);
    for (int q = 16; q > 0; q >>= 1) rad += __shfl_xor_sync(0xffffffffu, rad, q);
    const double d = A[(long long)r * n + r];
    lo = fmin(lo, d - rad);
    hi = fmax(hi, d + rad);
  }
  for (int r = threadIdx.x; r < n; r += kInitT) v0[r] = entry(f0[r]);
  if (lane == 0) {
    slo[warp] = lo;
    shi[warp] = hi;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < kInitT / 32; ++w) {
      lo = fmin(lo, slo[w]);
      hi = fmax(hi, shi[w]);
    }
    cw[0] = 0.5 * (lo + hi);
    cw[1] = 1.01 * 0.5 * (hi - lo);
  }
}

// The recursion with a stride of S terms, in one cooperative launch: v_{t+S} = 2 T_S(A~) v_t - v_{t-S}
// advances the S vectors of a round by one matrix (S = 1: A~ itself). Every v_t is kept as row t of `hist`.
// A warp per row of the matrix (rows stay in the SM's L1), the round's vectors staged in shared memory.
// The rows of hist are filled with an all-ones bit pattern first (a NaN that `entry` never lets through), and a
// block waits for the entries of the round themselves, so a round costs one store-to-load trip through L2
// and S dot products (FP64-bound: about 1 us each for 512 rows), and no barrier. 4095 terms of a 512 x 512
// A took 25.6 ms as separate launches, 23.9 ms with a grid barrier per term, 13.0 ms with S = 1, and take
// 7.4 ms with S = 4 including the two products that make T_4(A~). Every wait is bounded; one that runs
// out sets *err and the block leaves.
constexpr unsigned kPollLimit = 1u << 21;

// mat: A with cw = {c, w} (S = 1, mat = A, scaled on the fly), or T_S(A~) with cw = null. STAGED: the round's
// vectors in shared memory, and (rows) the first row of each warp as well.
template <int S, bool STAGED>
__global__ void k_cheb_run(const double *mat, int n, const double *cw, double *hist, int n_terms, int *err, int rows) {
  extern __shared__ double sv[];  // the round's S vectors, then (rows) a row per warp
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  const double c = cw ? cw[0] : 0.0, iw = cw ? 1.0 / cw[1] : 1.0;
  const int r0 = blockIdx.x * nw + warp, stride = gridDim.x * nw;
  constexpr int LG = 32 / S;       // lanes that hold the same vector's sum after the reduce-scatter
  const int mine = lane / LG;      // this lane's vector
  double v_old = 0.0;              // v_{t-S} of row r0 (first lane of each group)
  double *own = sv + (long long)(S + warp) * n;
  if (STAGED && rows && r0 < n)
    for (int j = lane; j < n; j += 32) own[j] = mat[(long long)r0 * n + j];  // read by the same lane only
  for (int t = 0; t + S < n_terms; t += S) {
    const double *cur = hist + (long long)t * n;
    bool ok = true;
    // kLoads entries per thread in flight, the unset ones loaded again together (one at a time, a round of
    // 512 rows with S = 4 took 9.1 us)
    constexpr int kLoads = 4 * S;
    for (int j0 = threadIdx.x; j0 < S * n; j0 += kLoads * blockDim.x) {
      unsigned long long bits[kLoads];
#pragma unroll
      for (int u = 0; u < kLoads; ++u) bits[u] = j0 + u * blockDim.x < S * n ? kUnset : 0;
      bool some = true;
      for (unsigned i = 0; i < kPollLimit && some; ++i) {
        some = false;
#pragma unroll
        for (int u = 0; u < kLoads; ++u)
          if (bits[u] == kUnset)
            asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(bits[u]) : "l"(cur + j0 + u * blockDim.x) : "memory");
#pragma unroll
        for (int u = 0; u < kLoads; ++u) some = some || bits[u] == kUnset;
      }
      ok = ok && !some;
#pragma unroll
      for (int u = 0; u < kLoads; ++u)
        if (STAGED && j0 + u * blockDim.x < S * n) sv[j0 + u * blockDim.x] = __longlong_as_double((long long)bits[u]);
    }
    if (!__syncthreads_and(ok)) {
      if (threadIdx.x == 0) atomicExch(err, 1);
      return;
    }
    for (int r = r0; r < n; r += stride) {
      double s[S];
#pragma unroll
      for (int u = 0; u < S; ++u) s[u] = 0.0;
      const double *row = mat + (long long)r * n;
      if (STAGED && rows && r == r0) {
#pragma unroll 4
        for (int j = lane; j < n; j += 32) {
          const double m = own[j];
#pragma unroll
          for (int u = 0; u < S; ++u) s[u] = fma(m, sv[u * n + j], s[u]);
        }
      } else {
#pragma unroll 4
        for (int j = lane; j < n; j += 32) {
          const double m = row[j];
#pragma unroll
          for (int u = 0; u < S; ++u) s[u] = fma(m, STAGED ? sv[u * n + j] : __ldcg(cur + (long long)u * n + j), s[u]);
        }
      }
      // reduce-scatter over the vectors, then the sum over the lanes of a group
#pragma unroll
      for (int w = 16, k = S / 2; k > 0; w >>= 1, k >>= 1)
#pragma unroll
        for (int u = 0; u < k; ++u) {
          const bool up = (lane & w) != 0;
          const double give = up ? s[u] : s[u + k], keep = up ? s[u + k] : s[u];
          s[u] = keep + __shfl_xor_sync(0xffffffffu, give, w);
        }
#pragma unroll
      for (int w = LG / 2; w > 0; w >>= 1) s[0] += __shfl_xor_sync(0xffffffffu, s[0], w);
      const int tn = t + S + mine;
      if (lane % LG == 0 && tn < n_terms) {
        const double vr = STAGED ? sv[mine * n + r] : __ldcg(cur + (long long)mine * n + r);
        const double at = cw ? (s[0] - c * vr) * iw : s[0];
        // v_{t-S}; at the start T_{|m-S|}: v_S = T_S v_0, and v_{S+m} subtracts v_{S-m}
        double before;
        if (t == 0)
          before = mine == 0 ? at : (STAGED ? sv[(S - mine) * n + r] : __ldcg(hist + (long long)(S - mine) * n + r));
        else
          before = r == r0 ? v_old : __ldcg(hist + (long long)(t - S + mine) * n + r);
        const double v = entry(2.0 * at - before);
        asm volatile("st.relaxed.gpu.global.f64 [%0], %1;" ::"l"(hist + (long long)tn * n + r), "d"(v) : "memory");
        if (r == r0) v_old = vr;
      }
    }
    __syncthreads();  // the staged vectors are rewritten in the next round
  }
}

// entries of A~ = (A - c) / w, and of a plain matrix; rows m, columns k (left) or rows k, columns n (right)
struct LoadScaled {
  const double *A, *cw;
  int n;
  __device__ double at(long long r, long long c) const {
    const double a = A[r * n + c];
    return (r == c ? a - cw[0] : a) / cw[1];
  }
};
struct LoadPlain {
  const double *A;
  int n;
  __device__ double at(long long r, long long c) const { return A[r * n + c]; }
};
template <class M> struct Left {
  M m;
  __device__ double operator()(int r, long long k) const { return m.at(r, k); }
};
template <class M> struct Right {
  M m;
  __device__ double operator()(int c, long long k) const { return m.at(k, c); }
};

// out = 2 sum of the chunks' products - 1: T_2 of the matrix that was squared
__global__ void k_cheb_square(const double *part, int chunks, int n, double *out) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x, nn = (long long)n * n;
  if (i >= nn) return;
  double s = 0.0;
  for (int c = 0; c < chunks; ++c) s += part[(long long)c * nn + i];
  out[i] = 2.0 * s - (i / n == i % n ? 1.0 : 0.0);
}

// the vectors before the first round: y = M x (times 2 minus x with `third`), a warp per row
template <class M> __global__ void __launch_bounds__(kSpT) k_cheb_first(M m, int n, const double *x, double *y, int third) {
  const int r = blockIdx.x * (kSpT / 32) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (r >= n) return;
  double s = 0.0;
  for (int j = lane; j < n; j += 32) s = fma(m.at(r, j), x[j], s);
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane == 0) y[r] = entry(third ? 2.0 * s - x[r] : s);
}

constexpr int kStride = 4, kSqChunks = 4;
// Rounds of four terms where the two n^3 products that they need (about n^3 / 1.5e5 us) cost less than the
// round trips saved (about 2 us per term).
bool cheb_strided(int n, int n_terms) { return n_terms >= 64 && (double)n * n * n < 1.5e5 * n_terms; }

// R_t = f0 . v_t, a warp per term
__global__ void __launch_bounds__(kSpT) k_cheb_residues(const double *hist, const double *f0, int n, int n_terms, double *R) {
  const int t = blockIdx.x * (kSpT / 32) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (t >= n_terms) return;
  double s = 0.0;
  for (int j = lane; j < n; j += 32) s = fma(f0[j], hist[(long long)t * n + j], s);
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane == 0) R[t] = s;
}

// cosine table tab[j] = cos(pi j / (2 K)), j < 4 K: T_n(x_k) = cos(pi n (2 k + 1) / (2 K)) is an entry of it
__global__ void k_cos_table(int K, double *tab) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j < 4 * K) tab[j] = cospi((double)j / (2.0 * (double)K));
}

// D_k = sum_n (2 - delta_n0) R_n T_n(x_k): a block per node, the threads share the terms (before: one
// thread per node evaluating a cosine per term, 3.2 ms at 4096 terms; this kernel 77 us)
__global__ void __launch_bounds__(kSpT) k_cheb_density(const double *R, int K, const double *tab, double *D) {
  __shared__ double red[kSpT];
  const unsigned k = blockIdx.x, period = 4u * (unsigned)K;
  const unsigned odd = 2u * k + 1u;
  const unsigned step = (unsigned)(((unsigned long long)kSpT * odd) % period);
  unsigned j = (unsigned)(((unsigned long long)threadIdx.x * odd) % period);
  double s = 0.0;
  for (int n = threadIdx.x; n < K; n += kSpT) {
    s = fma(n == 0 ? R[0] : 2.0 * R[n], tab[j], s);
    j += step;
    if (j >= period) j -= period;
  }
  s = block_sum_fixed(s, red);
  if (threadIdx.x == 0) D[k] = s;
}

// sigma_j = omega_j / K sum_k G_s(c + w x_k - omega_j) D_k: a block per frequency (before: a thread, four
// blocks for 400 frequencies, 8.9 ms; here 54 us). Gaussians below the smallest FP64 number are not evaluated.
__global__ void __launch_bounds__(kSpT)
    k_sigma(const double *D, int K, const double *tab, const double *cw, const double *omega, int n_omega, double s,
            double *sigma) {
  __shared__ double red[kSpT];
  const double c = cw[0], w = cw[1], norm = 1.0 / (s * sqrt(2.0 * M_PI));
  for (int j = blockIdx.x; j < n_omega; j += gridDim.x) {
    const double om = omega[j];
    double acc = 0.0;
    for (int k = threadIdx.x; k < K; k += kSpT) {
      const double e = (c + w * tab[2 * k + 1] - om) / s;
      const double q = e * e;
      acc = fma(q > 1500.0 ? 0.0 : exp(-0.5 * q), D[k], acc);  // (a D that is not finite stays one)
    }
    acc = block_sum_fixed(acc, red);
    if (threadIdx.x == 0) sigma[j] = om * norm * acc / (double)K;
  }
}

}  // namespace

size_t sigma_work_doubles(int K) { return 5 * (size_t)K; }  // D, then the cosine table

size_t spectrum_work_bytes(int n, int n_terms, int n_omega, bool squares) {
  // f0, cw, the vectors (n_terms x n), R, D and its cosine table, omega, sigma; T_2, T_4 and the chunks of
  // their products
  const size_t nn = squares && cheb_strided(n, n_terms) ? (size_t)n * n : 0;
  return sizeof(double) * ((size_t)n + 2 + (size_t)n * n_terms + (size_t)n_terms + sigma_work_doubles(n_terms) +
                           2 * (size_t)n_omega + (2 + kSqChunks) * nn);
}

SpectrumBufs spectrum_bufs(double *work, int n, int n_terms, int n_omega, bool squares) {
  SpectrumBufs b{};
  b.f0 = work;
  b.cw = b.f0 + n;
  b.hist = b.cw + 2;
  b.R = b.hist + (size_t)n * n_terms;
  b.D = b.R + n_terms;
  b.omega = b.D + sigma_work_doubles(n_terms);
  b.sigma = b.omega + n_omega;
  b.squares = squares && cheb_strided(n, n_terms) ? b.sigma + n_omega : nullptr;
  return b;
}

void launch_sigma_from_residues(const double *R, int K, const double *cw, const double *omega, int n_omega,
                                double s, double *D, double *sigma, cudaStream_t st) {
  double *tab = D + K;
  k_cos_table<<<(unsigned)((4 * K + kSpT - 1) / kSpT), kSpT, 0, st>>>(K, tab);
  k_cheb_density<<<K, kSpT, 0, st>>>(R, K, tab, D);
  k_sigma<<<n_omega < 65535 ? n_omega : 65535, kSpT, 0, st>>>(D, K, tab, cw, omega, n_omega, s, sigma);
  count_launch(3);
}

bool launch_absorption(const SpectrumBufs &b, const double *phi_o, const double *phi_c, int n_o, int n_c, int N,
                       double h, double box, double dV, const double *A, int axis, int n_terms, double s,
                       int n_omega, int *err, cudaStream_t st) {
  int n = n_o * n_c;
  k_dipole<<<n, kSpT, (size_t)N * sizeof(double), st>>>(phi_o, phi_c, n_c, N, h, box, axis, dV, b.f0);
  cudaMemsetAsync(b.hist, 0xff, (size_t)n * n_terms * sizeof(double), st);
  k_cheb_init<<<1, kInitT, 0, st>>>(A, n, b.f0, b.cw, b.hist);
  count_launch(2);
  const bool strided = b.squares != nullptr;
  const double *mat = A, *cw = b.cw;
  if (strided) {
    // T_2 = 2 A~ A~ - 1, T_4 = 2 T_2 T_2 - 1; v_1 = A~ v_0, v_2 = T_2 v_0, v_3 = 2 T_2 v_1 - v_1
    const long long nn = (long long)n * n;
    double *t2 = b.squares, *t4 = t2 + nn, *part = t4 + nn;
    const long long kc = ((n + kSqChunks - 1) / kSqChunks + kGemmBK - 1) / kGemmBK * kGemmBK;
    const int chunks = (int)((n + kc - 1) / kc);
    dim3 grid((unsigned)chunks, (n + kGemmBM - 1) / kGemmBM, (n + kGemmBN - 1) / kGemmBN);
    const LoadScaled a{A, b.cw, n};
    const LoadPlain p2{t2, n};
    const unsigned rows = (unsigned)((n + kSpT / 32 - 1) / (kSpT / 32)), flat = (unsigned)((nn + kSpT - 1) / kSpT);
    k_gemm_nt_part<double><<<grid, kGemmThreads, 0, st>>>(n, n, n, kc, Left<LoadScaled>{a}, Right<LoadScaled>{a}, part);
    k_cheb_square<<<flat, kSpT, 0, st>>>(part, chunks, n, t2);
    k_gemm_nt_part<double><<<grid, kGemmThreads, 0, st>>>(n, n, n, kc, Left<LoadPlain>{p2}, Right<LoadPlain>{p2}, part);
    k_cheb_square<<<flat, kSpT, 0, st>>>(part, chunks, n, t4);
    double *v = b.hist;
    k_cheb_first<<<rows, kSpT, 0, st>>>(a, n, v, v + n, 0);
    k_cheb_first<<<rows, kSpT, 0, st>>>(p2, n, v, v + 2 * n, 0);
    k_cheb_first<<<rows, kSpT, 0, st>>>(p2, n, v + n, v + 3 * n, 1);
    count_launch(7);
    mat = t4;
    cw = nullptr;
  }
  // four rows (warps) per block while that leaves an SM free for each block
  int dev = 0, sms = 0, per_sm = 0;
  int threads = n > 32 ? 128 : strided ? 512 : 1024;  // (512: the registers of four vectors)
  unsigned blocks = n <= 32 ? 1u : (unsigned)((n + 3) / 4);
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return false;
  if (blocks > (unsigned)sms) {
    threads = 512;
    blocks = (unsigned)((n + 15) / 16);
  }
  if (blocks > (unsigned)sms) blocks = (unsigned)sms;
  const size_t vec = (size_t)n * sizeof(double), vecs = (strided ? kStride : 1) * vec, most = 200 * 1024;
  const bool staged = vecs <= most;  // else the vectors are read from L2
  int rows = staged && vecs + threads / 32 * vec <= most;
  const size_t sm = staged ? vecs + (rows ? threads / 32 * vec : 0) : 0;
  const void *fn = strided ? (staged ? (const void *)k_cheb_run<kStride, true> : (const void *)k_cheb_run<kStride, false>)
                           : (staged ? (const void *)k_cheb_run<1, true> : (const void *)k_cheb_run<1, false>);
  if (sm > 48 * 1024) raise_smem_limit(fn, sm);
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, threads, sm) != cudaSuccess || per_sm < 1) return false;
  double *hist = b.hist;
  void *args[] = {&mat, &n, &cw, &hist, &n_terms, &err, &rows};
  if (cudaLaunchCooperativeKernel(fn, dim3(blocks), dim3(threads), args, sm, st) != cudaSuccess) return false;
  k_cheb_residues<<<(n_terms + kSpT / 32 - 1) / (kSpT / 32), kSpT, 0, st>>>(b.hist, b.f0, n, n_terms, b.R);
  count_launch(2);
  launch_sigma_from_residues(b.R, n_terms, b.cw, b.omega, n_omega, s, b.D, b.sigma, st);
  return true;
}

}  // namespace sbse
