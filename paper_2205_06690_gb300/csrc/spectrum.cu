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

// a vector entry as it is stored: a NaN of all ones as another one, so that none equals kUnset (an integer test: an
// FP64 comparison would lengthen the chain of a term)
constexpr unsigned long long kUnset = ~0ull;
__device__ __forceinline__ double entry(double v) {
  return (unsigned long long)__double_as_longlong(v) == kUnset ? __longlong_as_double(0x7ff8000000000000ll) : v;
}

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

// The recursion in one cooperative launch: v_{t+1} = 2 A~ v_t - v_{t-1}, A~ = (A - c) / w scaled on the fly, every
// v_t kept as row t of `hist`. A warp per row of the matrix, the vector staged in shared memory.
// The rows of hist are filled with an all-ones bit pattern first (a NaN that `entry` never lets through), and a
// block waits for the entries of v_t themselves, so a term costs one store-to-load trip through L2
// and a dot product per row (FP64-bound: about 0.5 us for 512 rows), and no barrier. 4095 terms of a 512 x 512
// A took 25.6 ms as separate launches, 23.9 ms with a grid barrier per term, and take about 15 ms. Every wait is
// bounded; one that runs out sets *err and the block leaves.
// (Rounds of four terms with T_4 of the matrix took 7.4 ms, but lost precision: the rounding of T_4's entries is the
// same in every round, and near the zeros of sin 4 theta, inside the spectrum, the recursion amplifies it. Residues
// were on average 1.5 and up to 8 times as far from 64 bits.)
constexpr unsigned kPollLimit = 1u << 21;

// staged: the vector in shared memory
__global__ void k_cheb_run(const double *A, int n, const double *cw, double *hist, int n_terms, int *err, int staged) {
  extern __shared__ double sv[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  const double c = cw[0], iw = 1.0 / cw[1];
  const int r0 = blockIdx.x * nw + warp, stride = gridDim.x * nw;
  double v_old = 0.0;  // v_{t-2} of row r0, kept by its lane 0
  for (int t = 1; t < n_terms; ++t) {
    const double *cur = hist + (long long)(t - 1) * n;
    bool ok = true;
    for (int j = threadIdx.x; j < n; j += blockDim.x) {
      unsigned long long bits = kUnset;
      for (unsigned i = 0; i < kPollLimit && bits == kUnset; ++i)
        asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(bits) : "l"(cur + j) : "memory");
      ok = ok && bits != kUnset;
      if (staged) sv[j] = __longlong_as_double((long long)bits);
    }
    if (!__syncthreads_and(ok)) {
      if (threadIdx.x == 0) atomicExch(err, 1);
      return;
    }
    for (int r = r0; r < n; r += stride) {
      const double *row = A + (long long)r * n;
      double s = 0.0, s2 = 0.0;
      int j = lane;
#pragma unroll 4
      for (; j + 32 < n; j += 64) {
        s = fma(row[j], staged ? sv[j] : __ldcg(cur + j), s);
        s2 = fma(row[j + 32], staged ? sv[j + 32] : __ldcg(cur + j + 32), s2);
      }
      if (j < n) s = fma(row[j], staged ? sv[j] : __ldcg(cur + j), s);
      s += s2;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      if (lane == 0) {
        const double vr = staged ? sv[r] : __ldcg(cur + r);
        const double at = (s - c * vr) * iw;
        const double before = t == 1 ? at : r == r0 ? v_old : __ldcg(cur - n + r);  // v_1 = A~ v_0
        asm volatile("st.relaxed.gpu.global.f64 [%0], %1;" ::"l"(hist + (long long)t * n + r), "d"(entry(2.0 * at - before))
                     : "memory");
        if (r == r0) v_old = vr;
      }
    }
    __syncthreads();  // the staged vector is rewritten in the next term
  }
}

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

size_t spectrum_work_bytes(int n, int n_terms, int n_omega) {
  // f0, cw, the vectors (n_terms x n), R, D and its cosine table, omega, sigma
  return sizeof(double) * ((size_t)n + 2 + (size_t)n * n_terms + (size_t)n_terms + sigma_work_doubles(n_terms) +
                           2 * (size_t)n_omega);
}

SpectrumBufs spectrum_bufs(double *work, int n, int n_terms, int n_omega) {
  SpectrumBufs b{};
  b.f0 = work;
  b.cw = b.f0 + n;
  b.hist = b.cw + 2;
  b.R = b.hist + (size_t)n * n_terms;
  b.D = b.R + n_terms;
  b.omega = b.D + sigma_work_doubles(n_terms);
  b.sigma = b.omega + n_omega;
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
  // four rows (warps) per block while that leaves an SM free for each block
  int dev = 0, sms = 0, per_sm = 0;
  int threads = n > 32 ? 128 : 1024;
  unsigned blocks = n <= 32 ? 1u : (unsigned)((n + 3) / 4);
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return false;
  if (blocks > (unsigned)sms) {
    threads = 512;
    blocks = (unsigned)((n + 15) / 16);
  }
  if (blocks > (unsigned)sms) blocks = (unsigned)sms;
  const size_t vec = (size_t)n * sizeof(double);
  int staged = vec <= 200 * 1024;  // else the vector is read from L2
  const size_t sm = staged ? vec : 0;
  if (sm > 48 * 1024) raise_smem_limit((const void *)k_cheb_run, sm);
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_cheb_run, threads, sm) != cudaSuccess || per_sm < 1)
    return false;
  const double *cw = b.cw;
  double *hist = b.hist;
  void *args[] = {&A, &n, &cw, &hist, &n_terms, &err, &staged};
  if (cudaLaunchCooperativeKernel((const void *)k_cheb_run, dim3(blocks), dim3(threads), args, sm, st) != cudaSuccess) return false;
  k_cheb_residues<<<(n_terms + kSpT / 32 - 1) / (kSpT / 32), kSpT, 0, st>>>(b.hist, b.f0, n, n_terms, b.R);
  count_launch(2);
  launch_sigma_from_residues(b.R, n_terms, b.cw, b.omega, n_omega, s, b.D, b.sigma, st);
  return true;
}

}  // namespace sbse
