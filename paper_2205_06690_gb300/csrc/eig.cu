// Lowest eigenvalues of the real symmetric Tamm-Dancoff matrix A (Eq. 1), in FP64 on the device:
// Householder reduction to tridiagonal form (one thread-block cluster, the matrix in its distributed
// shared memory) followed by Sturm-sequence multisection, one block per requested eigenvalue.
#include <cooperative_groups.h>
#include <math.h>

#include "kernels.h"

namespace sbse {

namespace cg = cooperative_groups;

__device__ double block_sum(double v, double *red) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  __syncthreads();
  if (lane == 0) red[w] = v;
  __syncthreads();
  double s = 0.0;
  if (threadIdx.x < 32) {
    s = (threadIdx.x < (blockDim.x >> 5)) ? red[threadIdx.x] : 0.0;
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (threadIdx.x == 0) red[32] = s;
  }
  __syncthreads();
  return red[32];
}

// Householder reduction of A (n x n, row-major, symmetric) to the diagonal dg[n] and off-diagonal
// of[n-1] by one thread-block cluster. H = I - beta v v^T maps A[k+1:, k] onto alpha e_1; the trailing
// block becomes A' - v w^T - w v^T with p = beta A' v, K = beta v.p / 2, w = p - K v.
// Rows are dealt to the CTAs in turn (row i to CTA i mod size: even shares while the trailing block
// shrinks) and stay in their shared memory (INSMEM; else in global memory, L2-resident, overwritten).
// Two exchanges a step, each CTA writing its entries into every CTA's copy through distributed shared
// memory: the column x, from which all CTAs form v alike, and p. The rank-2 update of step k - 1 is
// applied in the sweep that forms p of step k, so a row is read once per step.
// Bound: 3 m^2 FP64 multiply-adds per step over the cluster's SMs (1.6 per clock and SM) and the latency
// of two cluster barriers and two block sums. One block of 1024 threads took 64.2 ms at n = 512 and
// 2.58 ms at n = 128; the cluster of 16 takes 4.96 ms and 0.58 ms. A grid-wide barrier over all SMs
// would cut the arithmetic further but costs several times a cluster barrier, about what it saves.
// refl != null: the Householder vector of step k is stored in row k of refl (entries k+1 .. n-1)
// and its beta in betas[k] (0 where the step is the identity), for the back-transformation of
// eigenvectors.
// An FP64 instruction holds its SM sub-partition for about 64 clocks whatever the warp's active lanes, so
// the scalars (square root, division) are formed by one thread and the sums by one warp per
// sub-partition.
constexpr int kTriThreads = 512;

__host__ __device__ inline int tri_rows(int n, int cs) { return (n + cs - 1) / cs; }
// shared memory beyond the rows: x, v, the previous v and w, p (n each) and the scalars
__host__ __device__ inline size_t tri_vec_doubles(int n) { return 5 * (size_t)n + 8; }

// partial sums of a_i b_i, o <= i < n, into red[0..3] (first four warps); the caller synchronises
__device__ __forceinline__ void tri_dot(const double *a, const double *b, int o, int n, double *red) {
  if (threadIdx.x < 128) {
    double s = 0.0;
    for (int i = o + threadIdx.x; i < n; i += 128) s = fma(a[i], b[i], s);
    for (int q = 16; q > 0; q >>= 1) s += __shfl_xor_sync(0xffffffffu, s, q);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  }
}

template <bool INSMEM>
__global__ void __launch_bounds__(kTriThreads)
    k_tridiag(const double *Ain, double *Ag, int n, double *dg, double *of, double *refl, double *betas) {
  extern __shared__ double sm[];
  cg::cluster_group cl = cg::this_cluster();
  const int cs = (int)cl.num_blocks(), rank = (int)cl.block_rank();
  double *x = sm, *v = x + n, *vp = v + n, *wp = vp + n, *p = wp + n, *red = p + n;  // red: 4 sums, beta, K
  double *rows = INSMEM ? red + 8 : Ag;
  // row i (owned: i % cs == rank)
  auto row = [&](int i) { return INSMEM ? rows + (size_t)(i / cs) * n : rows + (size_t)i * n; };
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
  for (int i = rank + cs * warp; i < n; i += cs * nw) {
    double *r = row(i);
    for (int j = lane; j < n; j += 32) r[j] = Ain[(size_t)i * n + j];
  }
  for (int i = tid; i < n; i += blockDim.x) vp[i] = wp[i] = 0.0;
  cl.sync();  // (also orders the CTA's own rows)
  for (int k = 0; k + 2 < n; ++k) {
    const int o = k + 1;
    const int first = o + ((rank - o) % cs + cs) % cs;  // first owned row >= o
    // column k below the diagonal with the pending update, written to every CTA's x
    if (warp == 0) {
      const double vk = vp[k], wk = wp[k];
      for (int i = first + lane * cs; i < n; i += 32 * cs) {
        const double xi = fma(-wp[i], vk, fma(-vp[i], wk, row(i)[k]));
        for (int dst = 0; dst < cs; ++dst) *cl.map_shared_rank(x + i, dst) = xi;
      }
    } else if (warp == 1 && lane == 0 && k % cs == rank) {
      dg[k] = fma(-2.0 * vp[k], wp[k], row(k)[k]);
    }
    cl.sync();
    tri_dot(x, x, o, n, red);
    for (int i = o + tid; i < n; i += blockDim.x) v[i] = x[i];
    __syncthreads();
    if (tid == 0) {
      const double sigma = (red[0] + red[1]) + (red[2] + red[3]), x0 = x[o];
      double alpha = x0, beta = 0.0;
      if (!(sigma - x0 * x0 <= 0.0)) {  // else the step is the identity (beta = 0)
        alpha = x0 >= 0.0 ? -sqrt(sigma) : sqrt(sigma);
        beta = 1.0 / (sigma - x0 * alpha);  // 2 / |v|^2
        v[o] = x0 - alpha;
      }
      red[4] = beta;
      if (rank == 0) {
        of[k] = alpha;
        if (betas) betas[k] = beta;
      }
    }
    __syncthreads();
    const double beta = red[4];
    if (refl && k % cs == rank && beta != 0.0)
      for (int i = o + tid; i < n; i += blockDim.x) refl[(size_t)k * n + i] = v[i];
    // the pending update of the owned rows and p = beta A' v, one warp per row
    for (int i = first + cs * warp; i < n; i += cs * nw) {
      double *r = row(i);
      const double vi = vp[i], wi = wp[i];
      double s = 0.0;
      for (int j = o + lane; j < n; j += 32) {
        const double aij = fma(-wi, vp[j], fma(-vi, wp[j], r[j]));
        r[j] = aij;
        s = fma(aij, v[j], s);
      }
      for (int q = 16; q > 0; q >>= 1) s += __shfl_xor_sync(0xffffffffu, s, q);
      if (lane < cs) *cl.map_shared_rank(p + i, lane) = beta * s;
    }
    cl.sync();
    tri_dot(v, p, o, n, red);
    __syncthreads();
    if (tid == 0) red[5] = 0.5 * beta * ((red[0] + red[1]) + (red[2] + red[3]));
    __syncthreads();
    const double K = red[5];
    for (int i = o + tid; i < n; i += blockDim.x) {  // a step that is the identity leaves v = w = 0 pending
      const double vi = beta != 0.0 ? v[i] : 0.0;
      vp[i] = vi;
      wp[i] = fma(-K, vi, p[i]);
    }
    __syncthreads();
  }
  // the last 2 x 2 block, with the pending update
  if (tid == 0) {
    const int a = n - 2, b = n - 1;
    if (a % cs == rank) dg[a] = fma(-2.0 * vp[a], wp[a], row(a)[a]);
    if (b % cs == rank) {
      dg[b] = fma(-2.0 * vp[b], wp[b], row(b)[b]);
      of[a] = fma(-wp[b], vp[a], fma(-vp[b], wp[a], row(b)[a]));
    }
  }
  cl.sync();  // no CTA leaves while another may still write into its shared memory
}

// The same reduction by one block with the matrix in global memory, for sizes whose five vectors do not
// fit the shared memory of a cluster's CTAs (n > kTriMaxN).
constexpr int kEigThreads = 1024;
constexpr int kTriMaxN = 5000;

__global__ void __launch_bounds__(kEigThreads)
    k_tridiag_block(double *A, int n, double *dg, double *of, double *refl, double *betas) {
  extern __shared__ double sm[];
  double *v = sm;
  double *p = v + n;
  double *red = p + n;  // 33 doubles
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
  for (int k = 0; k + 2 < n; ++k) {
    const int m = n - k - 1;
    const int o = k + 1;
    double ss = 0.0;
    for (int i = tid; i < m; i += blockDim.x) {
      const double x = A[(long long)(o + i) * n + k];
      v[i] = x;
      ss += x * x;
    }
    const double sigma = block_sum(ss, red);
    const double x0 = v[0];
    if (sigma - x0 * x0 <= 0.0) {  // column already reduced
      if (tid == 0) {
        dg[k] = A[(long long)k * n + k];
        of[k] = x0;
        if (betas) betas[k] = 0.0;
      }
      __syncthreads();
      continue;
    }
    const double alpha = (x0 >= 0.0) ? -sqrt(sigma) : sqrt(sigma);
    const double beta = 1.0 / (sigma - x0 * alpha);  // 2 / |v|^2
    __syncthreads();
    if (tid == 0) v[0] = x0 - alpha;
    __syncthreads();
    if (refl) {
      for (int i = tid; i < m; i += blockDim.x) refl[(long long)k * n + o + i] = v[i];
      if (tid == 0) betas[k] = beta;
    }
    // p = beta A' v, one warp per row (coalesced across the row)
    for (int i = warp; i < m; i += nw) {
      const double *row = A + (long long)(o + i) * n + o;
      double s = 0.0;
      for (int j = lane; j < m; j += 32) s += row[j] * v[j];
      for (int q = 16; q > 0; q >>= 1) s += __shfl_xor_sync(0xffffffffu, s, q);
      if (lane == 0) p[i] = beta * s;
    }
    __syncthreads();
    double vp = 0.0;
    for (int i = tid; i < m; i += blockDim.x) vp += v[i] * p[i];
    const double K = 0.5 * beta * block_sum(vp, red);
    for (int i = tid; i < m; i += blockDim.x) p[i] -= K * v[i];  // p <- w
    __syncthreads();
    const long long mm = (long long)m * m;
    for (long long l = tid; l < mm; l += blockDim.x) {
      const int i = (int)(l / m), j = (int)(l - (long long)i * m);
      A[(long long)(o + i) * n + o + j] -= v[i] * p[j] + p[i] * v[j];
    }
    if (tid == 0) {
      dg[k] = A[(long long)k * n + k];
      of[k] = alpha;
    }
    __syncthreads();
  }
  if (tid == 0) {
    if (n >= 2) {
      dg[n - 2] = A[(long long)(n - 2) * n + n - 2];
      of[n - 2] = A[(long long)(n - 1) * n + n - 2];
    }
    dg[n - 1] = A[(long long)(n - 1) * n + n - 1];
  }
}

// k_tridiag on the largest cluster that its shared memory and the device allow (16 CTAs need the
// opt-in; small matrices take fewer, with at least 8 rows each)
static void launch_tridiag(const double *A, double *Aw, int n, double *dg, double *of, double *refl, double *betas,
                           cudaStream_t s) {
  if (n > kTriMaxN) {
    const size_t sm = (2 * (size_t)n + 34) * sizeof(double);
    raise_smem_limit((const void *)k_tridiag_block, sm);
    cudaMemcpyAsync(Aw, A, (size_t)n * n * sizeof(double), cudaMemcpyDeviceToDevice, s);
    k_tridiag_block<<<1, kEigThreads, sm, s>>>(Aw, n, dg, of, refl, betas);
    count_launch(1);
    return;
  }
  for (int cs = 16; cs >= 1; cs >>= 1) {
    if (cs > 1 && n < 8 * cs) continue;
    const size_t vec = tri_vec_doubles(n) * sizeof(double);
    const size_t full = vec + (size_t)tri_rows(n, cs) * n * sizeof(double);
    const bool in = full <= 200 * 1024;
    const void *fn = in ? (const void *)k_tridiag<true> : (const void *)k_tridiag<false>;
    const size_t smem = in ? full : vec;
    if (smem > 48 * 1024) raise_smem_limit(fn, smem);
    if (cs > 8 && cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) {
      cudaGetLastError();
      continue;
    }
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)cs);
    cfg.blockDim = dim3(kTriThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = (unsigned)cs;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    int fit = 0;
    if (cs > 1 && (cudaOccupancyMaxActiveClusters(&fit, fn, &cfg) != cudaSuccess || fit < 1)) {
      cudaGetLastError();
      continue;
    }
    if (in)
      cudaLaunchKernelEx(&cfg, k_tridiag<true>, A, Aw, n, dg, of, refl, betas);
    else
      cudaLaunchKernelEx(&cfg, k_tridiag<false>, A, Aw, n, dg, of, refl, betas);
    count_launch(1);
    return;
  }
}

// The tridiagonal scaled by a power of two to norm <= 1, for the Sturm counts: ds = diagonal, es =
// squared off-diagonal, kept at or above 1e-40 (a change of 1e-20 of the norm in the off-diagonal, far
// below rounding) so that a decoupled matrix never makes the recurrence vanish.
// Number of eigenvalues below x from the sign changes of the principal minors,
// p_i = (d_i - x) p_{i-1} - e_{i-1}^2 p_{i-2} (a zero minor takes the sign opposite to the one before, as
// the zero pivot of the quotient form counts as negative). Every four steps the pair is rescaled by a
// power of two (|d - x| <= 2 and the floor on e^2 keep four steps far inside the exponent range). Three
// FP64 instructions per step and no division: the quotient form's division made the chain several
// times longer.
__device__ __forceinline__ int sturm_count(const double *ds, const double *es, int n, double x) {
  // the sign and the zero test read the bit pattern: an FP64 comparison costs as much as a product
  double p0 = 1.0, p1 = ds[0] - x;
  auto zero = [](double p) { return ((__double2hiint(p) << 1) | __double2loint(p)) == 0; };
  int neg = zero(p1) ? 1 : (int)((unsigned)__double2hiint(p1) >> 31), c = neg;  // neg: sign of the latest minor
  int i = 1;
  auto step = [&](int q) {
    const double p2 = fma(ds[q] - x, p1, -(es[q - 1] * p0));
    const int ng = zero(p2) ? 1 - neg : (int)((unsigned)__double2hiint(p2) >> 31);
    c += ng ^ neg;
    neg = ng;
    p0 = p1;
    p1 = p2;
  };
  for (; i + 3 < n; i += 4) {
#pragma unroll
    for (int u = 0; u < 4; ++u) step(i + u);
    // scale by 2^-e, e the exponent of the larger of the two
    const int e0 = (__double2hiint(p0) >> 20) & 0x7ff, e1 = (__double2hiint(p1) >> 20) & 0x7ff;
    const double sc = __hiloint2double((2046 - max(max(e0, e1), 1)) << 20, 0);
    p0 *= sc;
    p1 *= sc;
  }
  for (; i < n; ++i) step(i);
  return c;
}

// (j+1)-th smallest eigenvalue by multisection: one block per eigenvalue, each thread counts the
// eigenvalues below one of 128 interior points of the bracket, which shrinks 129-fold per round (a warp
// on each of the SM's sub-partitions costs no more time than one warp). Eight warps of eight
// eigenvalues on one SM with the quotient form took 5.9 ms for ten eigenvalues at n = 512, this 0.58 ms;
// at n = 128, 1.48 ms and 0.15 ms.
// A tridiagonal with an entry that is not finite has no eigenvalues: NaN (fmin and fmax pass over a NaN, so
// bounds and norm do not show it).
constexpr int kBisT = 128;
__global__ void __launch_bounds__(kBisT) k_bisect(const double *dg, const double *of, int n, int k, double *ev) {
  extern __shared__ double sm[];
  __shared__ double bound[3][kBisT / 32];
  double *ds = sm, *es = sm + n;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, j = blockIdx.x;
  double lo = dg[0], hi = dg[0], nrm = 0.0;
  bool finite = true;
  for (int i = threadIdx.x; i < n; i += kBisT) {
    const double d = dg[i];
    finite = finite && fabs(d) < INFINITY && (i == n - 1 || fabs(of[i]) < INFINITY);
    const double r = (i > 0 ? fabs(of[i - 1]) : 0.0) + (i < n - 1 ? fabs(of[i]) : 0.0);
    lo = fmin(lo, d - r);
    hi = fmax(hi, d + r);
    nrm = fmax(nrm, fabs(d) + r);
  }
  for (int q = 16; q > 0; q >>= 1) {
    lo = fmin(lo, __shfl_xor_sync(0xffffffffu, lo, q));
    hi = fmax(hi, __shfl_xor_sync(0xffffffffu, hi, q));
    nrm = fmax(nrm, __shfl_xor_sync(0xffffffffu, nrm, q));
  }
  if (lane == 0) {
    bound[0][warp] = lo;
    bound[1][warp] = hi;
    bound[2][warp] = nrm;
  }
  if (!__syncthreads_and(finite)) {
    if (threadIdx.x == 0) ev[j] = NAN;
    return;
  }
  for (int w = 0; w < kBisT / 32; ++w) {
    lo = fmin(lo, bound[0][w]);
    hi = fmax(hi, bound[1][w]);
    nrm = fmax(nrm, bound[2][w]);
  }
  if (nrm == 0.0) {  // the zero matrix (the floor on e^2 below is relative to the norm)
    if (threadIdx.x == 0) ev[j] = 0.0;
    return;
  }
  int ex = 0;
  if (nrm < INFINITY) frexp(nrm, &ex);
  for (int i = threadIdx.x; i < n; i += kBisT) {
    ds[i] = ldexp(dg[i], -ex);
    if (i < n - 1) {
      const double e = ldexp(of[i], -ex);
      es[i] = fmax(e * e, 1e-40);
    }
  }
  __syncthreads();
  lo = ldexp(lo, -ex) - 1e-12;
  hi = ldexp(hi, -ex) + 1e-12;
  for (int it = 0; it < 64; ++it) {
    const double w = (hi - lo) / (kBisT + 1.0);
    const double x = lo + (threadIdx.x + 1) * w;
    const bool below = (x > lo && x < hi) ? (sturm_count(ds, es, n, x) <= j) : (x <= lo);
    const int m = __syncthreads_count(below);  // threads 0..m-1 have at most j eigenvalues below their point
    const double nlo = (m == 0) ? lo : lo + m * w;
    const double nhi = (m == kBisT) ? hi : lo + (m + 1) * w;
    if (!(nhi - nlo < hi - lo)) break;  // no further progress in floating point
    lo = nlo;
    hi = nhi;
  }
  if (threadIdx.x == 0) ev[j] = ldexp(0.5 * (lo + hi), ex);
}

static void launch_bisect(const double *dg, const double *of, int n, int k, double *ev, cudaStream_t s) {
  const size_t sm = 2 * (size_t)n * sizeof(double);
  if (sm > 48 * 1024) raise_smem_limit((const void *)k_bisect, sm);
  k_bisect<<<k, kBisT, sm, s>>>(dg, of, n, k, ev);
  count_launch(1);
}

size_t eig_work_bytes(int n) { return (size_t)n * n * sizeof(double) + 2 * (size_t)n * sizeof(double); }

// A (device, n x n) is copied into work and reduced there; the lowest k eigenvalues go to evals_dev.
int launch_eig_lowest(double *A, int n, int k, double *evals_dev, double *work, cudaStream_t s) {
  double *Aw = work;
  double *dg = Aw + (long long)n * n;
  double *of = dg + n;
  if (n >= 3) {
    launch_tridiag(A, Aw, n, dg, of, nullptr, nullptr, s);
  } else {
    // n <= 2: the matrix is already tridiagonal
    cudaMemcpyAsync(dg, A, sizeof(double), cudaMemcpyDeviceToDevice, s);
    if (n == 2) {
      cudaMemcpyAsync(dg + 1, A + 3, sizeof(double), cudaMemcpyDeviceToDevice, s);
      cudaMemcpyAsync(of, A + 2, sizeof(double), cudaMemcpyDeviceToDevice, s);
    }
  }
  launch_bisect(dg, of, n, k, evals_dev, s);
  return 0;
}

// ---- eigenvectors: inverse iteration on the tridiagonal T, then x = Q y with the stored reflectors

// (T - lam I) = P L U by Gaussian elimination with partial pivoting (row interchanges between
// neighbours); U has the diagonal d, first and second superdiagonals e, f; mult and piv record
// the elimination for the right-hand sides. tiny replaces exact zero pivots.
__device__ void tri_factor(const double *dg, const double *of, int n, double lam, double tiny, double *d,
                           double *e, double *f, double *mult, unsigned char *piv) {
  double b = dg[0] - lam, c = n > 1 ? of[0] : 0.0;
  for (int i = 0; i + 1 < n; ++i) {
    const double a = of[i], bn = dg[i + 1] - lam, cn = (i + 2 < n) ? of[i + 1] : 0.0;
    if (fabs(b) >= fabs(a)) {
      if (b == 0.0) b = tiny;
      const double m = a / b;
      piv[i] = 0;
      d[i] = b;
      e[i] = c;
      f[i] = 0.0;
      mult[i] = m;
      b = bn - m * c;
      c = cn;
    } else {
      const double m = b / a;
      piv[i] = 1;
      d[i] = a;
      e[i] = bn;
      f[i] = cn;
      mult[i] = m;
      b = c - m * bn;
      c = -m * cn;
    }
  }
  d[n - 1] = (b == 0.0) ? tiny : b;
}

// r <- (T - lam I)^-1 r with the factors of tri_factor
__device__ void tri_solve(int n, const double *d, const double *e, const double *f, const double *mult,
                          const unsigned char *piv, double *r) {
  for (int i = 0; i + 1 < n; ++i) {
    if (piv[i]) {
      const double t = r[i];
      r[i] = r[i + 1];
      r[i + 1] = t;
    }
    r[i + 1] -= mult[i] * r[i];
  }
  r[n - 1] /= d[n - 1];
  if (n >= 2) r[n - 2] = (r[n - 2] - e[n - 2] * r[n - 1]) / d[n - 2];
  for (int i = n - 3; i >= 0; --i) r[i] = (r[i] - e[i] * r[i + 1] - f[i] * r[i + 2]) / d[i];
}

// eigenvectors Y[j][.] of T for the ascending eigenvalues ev[j], j < k (one block): three inverse
// iterations each from a fixed start vector; a vector whose eigenvalue is within 1e-3 |T| of an
// earlier one is orthogonalised against that cluster after every iteration.
__global__ void __launch_bounds__(256)
    k_tri_vectors(const double *dg, const double *of, int n, int k, const double *ev, double *Y,
                  double *fac /* 4 n doubles + n bytes */) {
  __shared__ double red[33];
  double *d = fac, *e = d + n, *f = e + n, *mult = f + n;
  unsigned char *piv = reinterpret_cast<unsigned char *>(mult + n);
  double nrm = 0.0;
  for (int i = 0; i < n; ++i)
    nrm = fmax(nrm, fabs(dg[i]) + (i > 0 ? fabs(of[i - 1]) : 0.0) + (i + 1 < n ? fabs(of[i]) : 0.0));
  const double tiny = 2.2e-16 * (nrm + 1e-300);
  for (int j = 0; j < k; ++j) {
    double *y = Y + (long long)j * n;
    if (threadIdx.x == 0) tri_factor(dg, of, n, ev[j], tiny, d, e, f, mult, piv);
    for (int i = threadIdx.x; i < n; i += blockDim.x) y[i] = 1.0 + 0.5 * sin(1.0 + i);  // fixed start
    __syncthreads();
    for (int it = 0; it < 3; ++it) {
      if (threadIdx.x == 0) tri_solve(n, d, e, f, mult, piv, y);
      __syncthreads();
      for (int q = j - 1; q >= 0 && ev[j] - ev[q] < 1e-3 * nrm; --q) {  // cluster: Gram-Schmidt
        const double *yq = Y + (long long)q * n;
        double s = 0.0;
        for (int i = threadIdx.x; i < n; i += blockDim.x) s += yq[i] * y[i];
        s = block_sum(s, red);
        for (int i = threadIdx.x; i < n; i += blockDim.x) y[i] -= s * yq[i];
        __syncthreads();
      }
      double s = 0.0;
      for (int i = threadIdx.x; i < n; i += blockDim.x) s += y[i] * y[i];
      const double inv = 1.0 / sqrt(block_sum(s, red));
      for (int i = threadIdx.x; i < n; i += blockDim.x) y[i] *= inv;
      __syncthreads();
    }
  }
}

// x_j = H_0 H_1 ... H_{n-3} y_j (one block per eigenvector), sign fixed so that the component of
// largest magnitude is positive; X row-major n x k
__global__ void __launch_bounds__(256)
    k_tri_backtransform(const double *refl, const double *betas, int n, int k, const double *Y, double *X) {
  extern __shared__ double sy[];
  __shared__ double red[33];
  const int j = blockIdx.x;
  for (int i = threadIdx.x; i < n; i += blockDim.x) sy[i] = Y[(long long)j * n + i];
  __syncthreads();
  for (int kk = n - 3; kk >= 0; --kk) {
    const double beta = betas[kk];
    if (beta == 0.0) continue;
    const double *v = refl + (long long)kk * n;
    double s = 0.0;
    for (int i = kk + 1 + threadIdx.x; i < n; i += blockDim.x) s += v[i] * sy[i];
    s = beta * block_sum(s, red);
    for (int i = kk + 1 + threadIdx.x; i < n; i += blockDim.x) sy[i] -= s * v[i];
    __syncthreads();
  }
  // sign: the largest-magnitude component positive (first index on ties)
  double best = -1.0;
  int arg = n;
  for (int i = threadIdx.x; i < n; i += blockDim.x)
    if (fabs(sy[i]) > best) {
      best = fabs(sy[i]);
      arg = i;
    }
  __shared__ double bv[256];
  __shared__ int bi[256];
  bv[threadIdx.x] = best;
  bi[threadIdx.x] = arg;
  __syncthreads();
  for (int w = blockDim.x / 2; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w) {
      const double o = bv[threadIdx.x + w];
      const int oi = bi[threadIdx.x + w];
      if (o > bv[threadIdx.x] || (o == bv[threadIdx.x] && oi < bi[threadIdx.x])) {
        bv[threadIdx.x] = o;
        bi[threadIdx.x] = oi;
      }
    }
    __syncthreads();
  }
  const double sg = (bi[0] < n && sy[bi[0]] < 0.0) ? -1.0 : 1.0;
  for (int i = threadIdx.x; i < n; i += blockDim.x) X[(long long)i * k + j] = sg * sy[i];
}

size_t eig_vectors_work_bytes(int n, int k) {
  return eig_work_bytes(n) + ((size_t)n * n + n + (size_t)k * n + 4 * (size_t)n) * sizeof(double) + n + 16;
}

// lowest k eigenvalues and their eigenvectors (row-major n x k, device) of A (device, n x n)
int launch_eig_vectors(const double *A, int n, int k, double *evals_dev, double *evecs_dev, double *work,
                       cudaStream_t s) {
  double *Aw = work;
  double *dg = Aw + (long long)n * n;
  double *of = dg + n;
  double *refl = of + n;
  double *betas = refl + (long long)n * n;
  double *Y = betas + n;
  double *fac = Y + (long long)k * n;
  cudaMemsetAsync(betas, 0, (size_t)n * sizeof(double), s);
  if (n >= 3) {
    launch_tridiag(A, Aw, n, dg, of, refl, betas, s);
  } else {
    cudaMemcpyAsync(dg, A, sizeof(double), cudaMemcpyDeviceToDevice, s);
    if (n == 2) {
      cudaMemcpyAsync(dg + 1, A + 3, sizeof(double), cudaMemcpyDeviceToDevice, s);
      cudaMemcpyAsync(of, A + 2, sizeof(double), cudaMemcpyDeviceToDevice, s);
    }
  }
  launch_bisect(dg, of, n, k, evals_dev, s);
  k_tri_vectors<<<1, 256, 0, s>>>(dg, of, n, k, evals_dev, Y, fac);
  k_tri_backtransform<<<k, 256, (size_t)n * sizeof(double), s>>>(refl, betas, n, k, Y, evecs_dev);
  count_launch(2);
  return 0;
}

}  // namespace sbse
