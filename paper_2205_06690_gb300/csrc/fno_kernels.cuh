// Kernels of the Fourier layers (fno.cu): truncated transforms by folded sums, the per-mode channel
// mix, the pointwise layer and the weight gradients.
//
// The kept modes of an axis come in pairs +-k and the samples in pairs x, N - x, so every truncated
// transform is summed over half the samples (even and odd parts) for half the modes (cosine and sine
// sums A, B give F(k) = A - i B and F(-k) = A + i B): a quarter of the multiply-adds of the direct sum.
// fold[p (m + 1) + k] = (cos, sin)(2 pi p k / N), p <= N / 2, k <= m. Kept index j of a full axis: k for
// j < m, k - 2m for j >= m (see kept()).
#pragma once

#include <cuda_bf16.h>

namespace sbse {

constexpr int kFoT = 128;
constexpr int kFoRows = 64;  // rows of a plane transformed along x at a time

inline int fo_rows(int N) { return N < kFoRows ? N : kFoRows; }
inline size_t fo_tab_bytes(int N, int m) { return (size_t)(N / 2 + 1) * (m + 1) * sizeof(float2); }
inline size_t fo_fwd_smem(int N, int m) {
  return fo_tab_bytes(N, m) + (size_t)N * m * sizeof(float2) + (size_t)fo_rows(N) * (N + 1) * sizeof(float);
}
inline size_t fo_inv_smem(int N, int m) {
  return fo_tab_bytes(N, m) + (size_t)N * m * sizeof(float2) + 2 * (size_t)(m + 1) * m * sizeof(float2);
}

// Forward x and y transforms of one real N x N plane (block = plane of in[..][y][x]) to
// out[plane][2m][m]. The plane is read once and nothing but the kept modes is written; bound by
// instruction issue (68 % of its slots, 18 % of DRAM). 128 fields of 64^3, m = 12: 103 us (separate x and y kernels of
// direct sums over the grid: 293 + 300 us).
__global__ void __launch_bounds__(kFoT)
    k_fo_fwd_xy(const float *in, float2 *out, int N, int m, const float2 *fold) {
  extern __shared__ __align__(16) unsigned char fo_smem[];
  const int H = N / 2, m1 = m + 1, RC = N < kFoRows ? N : kFoRows, ld = N + 1;
  float2 *tab = reinterpret_cast<float2 *>(fo_smem);
  float2 *T = tab + (H + 1) * m1;
  float *rows = reinterpret_cast<float *>(T + N * m);
  for (int i = threadIdx.x; i < (H + 1) * m1; i += kFoT) tab[i] = fold[i];
  const float *src = in + (long long)blockIdx.x * N * N;
  constexpr int RT = 4, KT = 3;
  for (int r0 = 0; r0 < N; r0 += RC) {
    const int rc = min(RC, N - r0);
    __syncthreads();
    for (int i = threadIdx.x; i < rc * N; i += kFoT) rows[(i / N) * ld + i % N] = src[(long long)r0 * N + i];
    __syncthreads();
    const int RG = (rc + RT - 1) / RT, KG = (m + KT - 1) / KT;
    for (int it = threadIdx.x; it < RG * KG; it += kFoT) {
      const int rg = it % RG, kg = it / RG;
      const float *row[RT];
      int kx[KT];
      float re[RT][KT], im[RT][KT];
#pragma unroll
      for (int i = 0; i < RT; ++i) row[i] = rows + min(rg + i * RG, rc - 1) * ld;
#pragma unroll
      for (int j = 0; j < KT; ++j) kx[j] = min(kg * KT + j, m - 1);
#pragma unroll
      for (int i = 0; i < RT; ++i)
#pragma unroll
        for (int j = 0; j < KT; ++j) {
          re[i][j] = row[i][0];
          im[i][j] = 0.f;
        }
      for (int p = 1; 2 * p < N; ++p) {
        float2 w[KT];
#pragma unroll
        for (int j = 0; j < KT; ++j) w[j] = tab[p * m1 + kx[j]];
#pragma unroll
        for (int i = 0; i < RT; ++i) {
          const float a = row[i][p], b = row[i][N - p], e = a + b, o = a - b;
#pragma unroll
          for (int j = 0; j < KT; ++j) {
            re[i][j] = fmaf(e, w[j].x, re[i][j]);
            im[i][j] = fmaf(-o, w[j].y, im[i][j]);
          }
        }
      }
      if (N % 2 == 0) {
#pragma unroll
        for (int i = 0; i < RT; ++i)
#pragma unroll
          for (int j = 0; j < KT; ++j) re[i][j] = fmaf(row[i][H], tab[H * m1 + kx[j]].x, re[i][j]);
      }
#pragma unroll
      for (int i = 0; i < RT; ++i)
#pragma unroll
        for (int j = 0; j < KT; ++j)
          if (rg + i * RG < rc && kg * KT + j < m)
            T[(r0 + rg + i * RG) * m + kg * KT + j] = make_float2(re[i][j], im[i][j]);
    }
  }
  __syncthreads();
  constexpr int YT = 2;
  const int YG = (m1 + YT - 1) / YT;
  float2 *dst = out + (long long)blockIdx.x * 2 * m * m;
  for (int it = threadIdx.x; it < m * YG; it += kFoT) {
    const int kx = it % m, kg = it / m;
    float2 A[YT], Bs[YT];
    int k[YT];
    const float2 t0 = T[kx];
#pragma unroll
    for (int j = 0; j < YT; ++j) {
      k[j] = min(kg * YT + j, m);
      A[j] = t0;
      Bs[j] = make_float2(0.f, 0.f);
    }
    for (int p = 1; 2 * p < N; ++p) {
      const float2 a = T[p * m + kx], b = T[(N - p) * m + kx];
      const float ex = a.x + b.x, ey = a.y + b.y, ox = a.x - b.x, oy = a.y - b.y;
#pragma unroll
      for (int j = 0; j < YT; ++j) {
        const float2 w = tab[p * m1 + k[j]];
        A[j].x = fmaf(ex, w.x, A[j].x);
        A[j].y = fmaf(ey, w.x, A[j].y);
        Bs[j].x = fmaf(ox, w.y, Bs[j].x);
        Bs[j].y = fmaf(oy, w.y, Bs[j].y);
      }
    }
#pragma unroll
    for (int j = 0; j < YT; ++j) {
      const int kk = kg * YT + j;
      if (kk > m) continue;
      if (N % 2 == 0) {
        const float c = tab[H * m1 + kk].x;
        A[j].x = fmaf(T[H * m + kx].x, c, A[j].x);
        A[j].y = fmaf(T[H * m + kx].y, c, A[j].y);
      }
      if (kk < m) dst[kk * m + kx] = make_float2(A[j].x + Bs[j].y, A[j].y - Bs[j].x);
      if (kk > 0) dst[(2 * m - kk) * m + kx] = make_float2(A[j].x - Bs[j].y, A[j].y + Bs[j].x);
    }
  }
}

// Forward z transform, in[o][N][inner] -> out[o][2m][inner]: thread per (o, i) and group of kZk modes
// (gridDim.y), the samples read coalesced over i from L2.
constexpr int kZk = 7;
__global__ void __launch_bounds__(kFoT)
    k_fo_fwd_z(const float2 *in, float2 *out, long long cols, int inner, int N, int m, const float2 *fold) {
  const long long t = (long long)blockIdx.x * kFoT + threadIdx.x;
  if (t >= cols) return;
  const long long o = t / inner;
  const int i = (int)(t - o * inner), H = N / 2, m1 = m + 1, k0 = blockIdx.y * kZk;
  const float2 *src = in + o * N * inner + i;
  float2 A[kZk], Bs[kZk];
  const float2 t0 = src[0];
#pragma unroll
  for (int j = 0; j < kZk; ++j) {
    A[j] = t0;
    Bs[j] = make_float2(0.f, 0.f);
  }
#pragma unroll 2
  for (int p = 1; 2 * p < N; ++p) {
    const float2 a = src[(long long)p * inner], b = src[(long long)(N - p) * inner];
    const float ex = a.x + b.x, ey = a.y + b.y, ox = a.x - b.x, oy = a.y - b.y;
#pragma unroll
    for (int j = 0; j < kZk; ++j) {
      const float2 w = fold[p * m1 + min(k0 + j, m)];
      A[j].x = fmaf(ex, w.x, A[j].x);
      A[j].y = fmaf(ey, w.x, A[j].y);
      Bs[j].x = fmaf(ox, w.y, Bs[j].x);
      Bs[j].y = fmaf(oy, w.y, Bs[j].y);
    }
  }
  const float2 h = N % 2 == 0 ? src[(long long)H * inner] : make_float2(0.f, 0.f);
  float2 *dst = out + o * 2 * m * inner + i;
#pragma unroll
  for (int j = 0; j < kZk; ++j) {
    const int k = k0 + j;
    if (k > m) continue;
    const float c = fold[H * m1 + k].x;
    const float ax = fmaf(h.x, c, A[j].x), ay = fmaf(h.y, c, A[j].y);
    if (k < m) dst[(long long)k * inner] = make_float2(ax + Bs[j].y, ay - Bs[j].x);
    if (k > 0) dst[(long long)(2 * m - k) * inner] = make_float2(ax - Bs[j].y, ay + Bs[j].x);
  }
}

// Inverse z transform, in[o][2m][inner] -> out[o][N][inner]: thread per (o, i) and group of kZz sample
// pairs z, N - z. P = G(k) + G(-k), M = G(k) - G(-k): out(+-z) = sum_k P cos +- i M sin.
constexpr int kZz = 4;
__global__ void __launch_bounds__(kFoT)
    k_fo_inv_z(const float2 *in, float2 *out, long long cols, int inner, int N, int m, const float2 *fold) {
  const long long t = (long long)blockIdx.x * kFoT + threadIdx.x;
  if (t >= cols) return;
  const long long o = t / inner;
  const int i = (int)(t - o * inner), H = N / 2, m1 = m + 1, p0 = blockIdx.y * kZz;
  const float2 *src = in + o * 2 * m * inner + i;
  float2 A[kZz], Bs[kZz];
  const float2 g0 = src[0];
#pragma unroll
  for (int j = 0; j < kZz; ++j) {
    A[j] = g0;
    Bs[j] = make_float2(0.f, 0.f);
  }
#pragma unroll 4
  for (int k = 1; k <= m; ++k) {
    const float2 g = k < m ? src[(long long)k * inner] : make_float2(0.f, 0.f), q = src[(long long)(2 * m - k) * inner];
    const float px = g.x + q.x, py = g.y + q.y, mx = g.x - q.x, my = g.y - q.y;
#pragma unroll
    for (int j = 0; j < kZz; ++j) {
      const float2 w = fold[min(p0 + j, H) * m1 + k];
      A[j].x = fmaf(px, w.x, A[j].x);
      A[j].y = fmaf(py, w.x, A[j].y);
      Bs[j].x = fmaf(mx, w.y, Bs[j].x);
      Bs[j].y = fmaf(my, w.y, Bs[j].y);
    }
  }
  float2 *dst = out + o * N * inner + i;
#pragma unroll
  for (int j = 0; j < kZz; ++j) {
    const int p = p0 + j;
    if (p > H) continue;
    dst[(long long)p * inner] = make_float2(A[j].x - Bs[j].y, A[j].y + Bs[j].x);
    if (p > 0 && 2 * p < N) dst[(long long)(N - p) * inner] = make_float2(A[j].x + Bs[j].y, A[j].y - Bs[j].x);
  }
}

// Inverse y and x transforms of one plane of kept modes in[plane][2m][m] to a real N x N plane:
// out = scale sum_kx c_kx Re(t_kx e^{i 2 pi kx x / N}), c_0 = 1, c_kx = 2 (hermitian) or 1. The row
// modes t stay in shared memory; lanes take consecutive x, so both halves of a row are written in
// whole segments. 128 fields of 64^3, m = 12: 74 us (before: 429 + 300 us).
__global__ void __launch_bounds__(kFoT)
    k_fo_inv_xy(const float2 *in, float *out, int N, int m, int hermitian, float scale, const float2 *fold) {
  extern __shared__ __align__(16) unsigned char fo_smem[];
  const int H = N / 2, m1 = m + 1;
  float2 *tab = reinterpret_cast<float2 *>(fo_smem);
  float2 *T = tab + (H + 1) * m1;
  float2 *P = T + N * m, *M = P + m1 * m;
  for (int i = threadIdx.x; i < (H + 1) * m1; i += kFoT) tab[i] = fold[i];
  const float2 *src = in + (long long)blockIdx.x * 2 * m * m;
  for (int i = threadIdx.x; i < m1 * m; i += kFoT) {
    const int k = i / m, kx = i - k * m;
    const float2 g = k < m ? src[k * m + kx] : make_float2(0.f, 0.f);
    const float2 q = k > 0 ? src[(2 * m - k) * m + kx] : make_float2(0.f, 0.f);
    P[i] = make_float2(g.x + q.x, g.y + q.y);
    M[i] = make_float2(g.x - q.x, g.y - q.y);
  }
  __syncthreads();
  constexpr int YT = 2;
  const int YG = (H + YT) / YT;  // pairs p = 0 .. H
  for (int it = threadIdx.x; it < m * YG; it += kFoT) {
    const int kx = it % m, pg = it / m;
    float2 A[YT], Bs[YT];
    int p[YT];
#pragma unroll
    for (int j = 0; j < YT; ++j) {
      p[j] = min(pg * YT + j, H);
      A[j] = P[kx];
      Bs[j] = make_float2(0.f, 0.f);
    }
    for (int k = 1; k <= m; ++k) {
      const float2 a = P[k * m + kx], b = M[k * m + kx];
#pragma unroll
      for (int j = 0; j < YT; ++j) {
        const float2 w = tab[p[j] * m1 + k];
        A[j].x = fmaf(a.x, w.x, A[j].x);
        A[j].y = fmaf(a.y, w.x, A[j].y);
        Bs[j].x = fmaf(b.x, w.y, Bs[j].x);
        Bs[j].y = fmaf(b.y, w.y, Bs[j].y);
      }
    }
    const float c = kx > 0 && hermitian ? 2.f * scale : scale;
#pragma unroll
    for (int j = 0; j < YT; ++j) {
      const int q = pg * YT + j;
      if (q > H) continue;
      T[q * m + kx] = make_float2(c * (A[j].x - Bs[j].y), c * (A[j].y + Bs[j].x));
      if (q > 0 && 2 * q < N) T[(N - q) * m + kx] = make_float2(c * (A[j].x + Bs[j].y), c * (A[j].y - Bs[j].x));
    }
  }
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, NP = (N + 1) / 2;
  float *dst = out + (long long)blockIdx.x * N * N;
  constexpr int RT = 8;
  for (int r0 = warp * RT; r0 < N; r0 += (kFoT / 32) * RT)
    for (int p0 = 0; p0 < NP; p0 += 32) {
      const int p = p0 + lane, pc = min(p, NP - 1);
      float E[RT], O[RT];
#pragma unroll
      for (int i = 0; i < RT; ++i) E[i] = O[i] = 0.f;
      for (int kx = 0; kx < m; ++kx) {
        const float2 w = tab[pc * m1 + kx];
#pragma unroll
        for (int i = 0; i < RT; ++i) {
          const float2 t = T[min(r0 + i, N - 1) * m + kx];
          E[i] = fmaf(t.x, w.x, E[i]);
          O[i] = fmaf(t.y, w.y, O[i]);
        }
      }
#pragma unroll
      for (int i = 0; i < RT; ++i)
        if (p < NP && r0 + i < N) {
          dst[(long long)(r0 + i) * N + p] = E[i] - O[i];
          if (p > 0) dst[(long long)(r0 + i) * N + N - p] = E[i] + O[i];
        }
    }
  if (N % 2 == 0)  // the column x = N / 2, its own mirror image
    for (int r = threadIdx.x; r < N; r += kFoT) {
      float s = 0.f;
      for (int kx = 0; kx < m; ++kx) s = fmaf(T[r * m + kx].x, tab[H * m1 + kx].x, s);
      dst[(long long)r * N + H] = s;
    }
}

// ---- per-mode channel mix ---------------------------------------------------------------------------
// A block takes kMxModes adjacent modes: the spectra F[b][c][mode] are read as segments of adjacent
// modes into shared memory, a warp takes one mode, and its lanes the output channels, so the weights
// R[mode][ci][co] are read once, in whole rows (one thread per output read them with a stride of C^2
// entries: 102 us at 6912 modes x 32 x 32, batch 4, here 39 us; 28 MB of weights).
constexpr int kMxModes = 8, kMxT = 32 * kMxModes, kMxB = 4;  // kMxB batch entries share one read of R

inline size_t mix_tile_bytes(int B, int C) { return (size_t)B * C * (kMxModes + 1) * sizeof(float2); }

__device__ __forceinline__ void mix_load(const float2 *g, float2 *s, int rows, int mode0, int nm, int modes, int m,
                                         const float *kxscale) {
  for (int i = threadIdx.x; i < rows * kMxModes; i += kMxT) {
    const int r = i / kMxModes, q = i % kMxModes;
    float2 v = make_float2(0.f, 0.f);
    if (q < nm) {
      v = g[(long long)r * modes + mode0 + q];
      if (kxscale) {
        const float f = kxscale[(mode0 + q) % m];
        v.x *= f;
        v.y *= f;
      }
    }
    s[r * (kMxModes + 1) + q] = v;
  }
}
__device__ __forceinline__ void mix_store(float2 *g, const float2 *s, int rows, int mode0, int nm, int modes) {
  for (int i = threadIdx.x; i < rows * kMxModes; i += kMxT) {
    const int r = i / kMxModes, q = i % kMxModes;
    if (q < nm) g[(long long)r * modes + mode0 + q] = s[r * (kMxModes + 1) + q];
  }
}

// Complex entries of the parameter vector start on any float: with an odd channel count its pairs are not
// aligned to their size, and are then read and written by halves.
__device__ __forceinline__ __nv_bfloat162 load_pair(const __nv_bfloat16 *p, bool aligned) {
  return aligned ? *reinterpret_cast<const __nv_bfloat162 *>(p) : __halves2bfloat162(p[0], p[1]);
}

// G[b][co][mode] = sum_ci F[b][ci][mode] R[mode][ci][co]
__global__ void __launch_bounds__(kMxT)
    k_fo_mix(const float2 *F, const __nv_bfloat16 *R, float2 *G, int B, int C, int modes, bool aligned) {
  extern __shared__ __align__(16) unsigned char fo_smem[];
  float2 *sF = reinterpret_cast<float2 *>(fo_smem), *sG = sF + B * C * (kMxModes + 1);
  const int mode0 = blockIdx.x * kMxModes, nm = min(kMxModes, modes - mode0);
  mix_load(F, sF, B * C, mode0, nm, modes, 1, nullptr);
  __syncthreads();
  const int q = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (q < nm) {
    const __nv_bfloat16 *Rm = R + 2ll * (mode0 + q) * C * C;
    for (int co = lane; co < C; co += 32)
      for (int b0 = 0; b0 < B; b0 += kMxB) {
        const int nb = min(kMxB, B - b0);
        float re[kMxB], im[kMxB];
#pragma unroll
        for (int b = 0; b < kMxB; ++b) re[b] = im[b] = 0.f;
#pragma unroll 8
        for (int ci = 0; ci < C; ++ci) {
          const float2 w = __bfloat1622float2(load_pair(Rm + 2 * (ci * C + co), aligned));
#pragma unroll
          for (int b = 0; b < kMxB; ++b) {
            const float2 x = sF[((b0 + min(b, nb - 1)) * C + ci) * (kMxModes + 1) + q];
            re[b] += x.x * w.x - x.y * w.y;
            im[b] += x.x * w.y + x.y * w.x;
          }
        }
#pragma unroll
        for (int b = 0; b < kMxB; ++b)
          if (b < nb) sG[((b0 + b) * C + co) * (kMxModes + 1) + q] = make_float2(re[b], im[b]);
      }
  }
  __syncthreads();
  mix_store(G, sG, B * C, mode0, nm, modes);
}

// Backward of the mix in one pass over dG' = kxscale dG: dR[mode][ci][co] = sum_b conj(F[b][ci]) dG'[b][co]
// and dF[b][ci][mode] = sum_co conj(R[mode][ci][co]) dG'[b][co]; lanes along co, the sum over co by a warp
// reduction would cost 10 shuffles per term, so dF is summed with lanes along ci from a transposed copy
// of the mode's weights in shared memory. add: dR holds the sum over earlier batch entries.
__global__ void __launch_bounds__(kMxT)
    k_fo_mix_back(const float2 *F, const float2 *dG, const __nv_bfloat16 *R, float *dR, float2 *dF, int B, int C, int modes,
                  int m, const float *kxscale, int add, bool aligned, bool aligned_d) {
  extern __shared__ __align__(16) unsigned char fo_smem[];
  float2 *sF = reinterpret_cast<float2 *>(fo_smem), *sG = sF + B * C * (kMxModes + 1);
  __nv_bfloat162 *sR = reinterpret_cast<__nv_bfloat162 *>(sG + B * C * (kMxModes + 1));
  const int mode0 = blockIdx.x * kMxModes, nm = min(kMxModes, modes - mode0);
  mix_load(F, sF, B * C, mode0, nm, modes, 1, nullptr);
  mix_load(dG, sG, B * C, mode0, nm, modes, m, kxscale);
  __syncthreads();
  const int q = threadIdx.x >> 5, lane = threadIdx.x & 31;
  __nv_bfloat162 *Rt = sR + (size_t)q * C * (C + 1);  // [co][ci], rows padded
  if (q < nm) {
    const long long base = (long long)(mode0 + q) * C * C;
    for (int ci = 0; ci < C; ++ci)
      for (int co = lane; co < C; co += 32) {
        Rt[co * (C + 1) + ci] = load_pair(R + 2 * (base + ci * C + co), aligned);
        float *r = dR + 2 * (base + ci * C + co);
        float re = add ? r[0] : 0.f, im = add ? r[1] : 0.f;
        for (int b = 0; b < B; ++b) {
          const float2 f = sF[(b * C + ci) * (kMxModes + 1) + q], g = sG[(b * C + co) * (kMxModes + 1) + q];
          re += f.x * g.x + f.y * g.y;
          im += f.x * g.y - f.y * g.x;
        }
        if (aligned_d) {
          *reinterpret_cast<float2 *>(r) = make_float2(re, im);
        } else {
          r[0] = re;
          r[1] = im;
        }
      }
  }
  __syncthreads();  // F is no longer needed: its tile takes dF
  if (q < nm)
    for (int ci = lane; ci < C; ci += 32)
      for (int b0 = 0; b0 < B; b0 += kMxB) {
        const int nb = min(kMxB, B - b0);
        float re[kMxB], im[kMxB];
#pragma unroll
        for (int b = 0; b < kMxB; ++b) re[b] = im[b] = 0.f;
#pragma unroll 4
        for (int co = 0; co < C; ++co) {
          const float2 w = __bfloat1622float2(Rt[co * (C + 1) + ci]);
#pragma unroll
          for (int b = 0; b < kMxB; ++b) {
            const float2 x = sG[((b0 + min(b, nb - 1)) * C + co) * (kMxModes + 1) + q];
            re[b] += w.x * x.x + w.y * x.y;  // conj(w) x
            im[b] += w.x * x.y - w.y * x.x;
          }
        }
#pragma unroll
        for (int b = 0; b < kMxB; ++b)
          if (b < nb) sF[((b0 + b) * C + ci) * (kMxModes + 1) + q] = make_float2(re[b], im[b]);
      }
  __syncthreads();
  mix_store(dF, sF, B * C, mode0, nm, modes);
}

// ---- pointwise layers -------------------------------------------------------------------------------
// One thread per kPw adjacent-by-stride points with the C input channels in registers (CP = C padded to
// a compiled size; the padding's weights are zero) and the weights as shared-memory broadcasts of four.
// FP32 multiply-adds (C^2 per point) and the activations' traffic bound it; with a runtime channel
// count the inputs sat in local memory. 64^3, C = 32, batch 4: forward 132 us
// without and 141 us with U (310 us before), backward 140 us (270 us, and 116 us for the activation).
constexpr int kPw = 2, kPwT = 128;

template <int CP, bool TRANS>
__device__ __forceinline__ void pw_weights(const __nv_bfloat16 *W, float *ws, int C) {
  for (int i = threadIdx.x; i < CP * CP; i += kPwT) {
    const int o = i / CP, k = i - o * CP;  // ws[out][in]
    ws[i] = (o < C && k < C) ? __bfloat162float(TRANS ? W[k * C + o] : W[o * C + k]) : 0.f;
  }
}

// U[b][co][r] = S + sum_ci W[co][ci] V[b][ci][r] + bias[co]; Vn = GELU(U) (act) or U; U may be null
template <int CP>
__global__ void __launch_bounds__(kPwT)
    k_fo_pointwise(const float *S, const float *V, const __nv_bfloat16 *W, const float *bias, float *U, float *Vn, int C,
                   long long ng, int act) {
  __shared__ __align__(16) float ws[CP * CP];
  pw_weights<CP, false>(W, ws, C);
  __syncthreads();
  const long long r0 = (long long)blockIdx.x * (kPwT * kPw) + threadIdx.x, b = blockIdx.y;
  float v[kPw][CP];
  bool in[kPw];
#pragma unroll
  for (int u = 0; u < kPw; ++u) {
    const long long r = r0 + u * kPwT;
    in[u] = r < ng;
#pragma unroll
    for (int c = 0; c < CP; ++c) v[u][c] = (in[u] && c < C) ? V[(b * C + c) * ng + r] : 0.f;
  }
  // outputs in groups of four: the group's loads are in flight together (one at a time, their latency was
  // the bound)
  for (int c0 = 0; c0 < C; c0 += 4) {
    float s[4][kPw];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int co = min(c0 + q, C - 1);
#pragma unroll
      for (int u = 0; u < kPw; ++u) s[q][u] = in[u] ? S[(b * C + co) * ng + r0 + u * kPwT] : 0.f;
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int co = min(c0 + q, C - 1);
      const float bi = bias[co];
#pragma unroll
      for (int u = 0; u < kPw; ++u) s[q][u] += bi;
#pragma unroll
      for (int c = 0; c < CP; c += 4) {
        const float4 w = *reinterpret_cast<const float4 *>(ws + co * CP + c);
#pragma unroll
        for (int u = 0; u < kPw; ++u) {
          s[q][u] = fmaf(w.x, v[u][c], s[q][u]);
          s[q][u] = fmaf(w.y, v[u][c + 1], s[q][u]);
          s[q][u] = fmaf(w.z, v[u][c + 2], s[q][u]);
          s[q][u] = fmaf(w.w, v[u][c + 3], s[q][u]);
        }
      }
      if (c0 + q < C) {
#pragma unroll
        for (int u = 0; u < kPw; ++u)
          if (in[u]) {
            const long long o = (b * C + co) * ng + r0 + u * kPwT;
            if (U) U[o] = s[q][u];
            Vn[o] = act ? gelu_f(s[q][u]) : s[q][u];
          }
      }
    }
  }
}

// dV[b][ci][r] = sum_co W[co][ci] dU[b][co][r] + dVspec[b][ci][r]; with Uprev (the pre-activation of the
// layer below) the result is multiplied by GELU'(Uprev), the gradient with respect to Uprev
template <int CP>
__global__ void __launch_bounds__(kPwT)
    k_fo_pointwise_back(const float *dU, const __nv_bfloat16 *W, const float *dVspec, const float *Uprev, float *dV, int C,
                        long long ng) {
  __shared__ __align__(16) float ws[CP * CP];
  pw_weights<CP, true>(W, ws, C);
  __syncthreads();
  const long long r0 = (long long)blockIdx.x * (kPwT * kPw) + threadIdx.x, b = blockIdx.y;
  float v[kPw][CP];
  bool in[kPw];
#pragma unroll
  for (int u = 0; u < kPw; ++u) {
    const long long r = r0 + u * kPwT;
    in[u] = r < ng;
#pragma unroll
    for (int c = 0; c < CP; ++c) v[u][c] = (in[u] && c < C) ? dU[(b * C + c) * ng + r] : 0.f;
  }
  for (int c0 = 0; c0 < C; c0 += 4) {  // groups of four, as above
    float s[4][kPw], up[4][kPw];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const long long o = (b * C + min(c0 + q, C - 1)) * ng + r0;
#pragma unroll
      for (int u = 0; u < kPw; ++u) {
        s[q][u] = in[u] ? dVspec[o + u * kPwT] : 0.f;
        up[q][u] = in[u] && Uprev ? Uprev[o + u * kPwT] : 0.f;
      }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int ci = min(c0 + q, C - 1);
#pragma unroll
      for (int c = 0; c < CP; c += 4) {
        const float4 w = *reinterpret_cast<const float4 *>(ws + ci * CP + c);
#pragma unroll
        for (int u = 0; u < kPw; ++u) {
          s[q][u] = fmaf(w.x, v[u][c], s[q][u]);
          s[q][u] = fmaf(w.y, v[u][c + 1], s[q][u]);
          s[q][u] = fmaf(w.z, v[u][c + 2], s[q][u]);
          s[q][u] = fmaf(w.w, v[u][c + 3], s[q][u]);
        }
      }
      if (c0 + q < C) {
#pragma unroll
        for (int u = 0; u < kPw; ++u)
          if (in[u]) dV[(b * C + ci) * ng + r0 + u * kPwT] = Uprev ? s[q][u] * gelu_grad_f(up[q][u]) : s[q][u];
      }
    }
  }
}

// ---- weight gradients -------------------------------------------------------------------------------
// part[chunk][i][j] = sum over a chunk of points of A[b][i][r] B[b][j][r], i < M, j < Nn, and for j = Nn
// the sum of A[b][i][r]: M, Nn <= 64 channels. 4 x 4 outputs per thread, the
// threads left over split the points of a tile and are summed at the end. Chunks are summed in FP32
// and stored in FP64 partials; the sums of A, which cancel most, as pairs of floats (Knuth's two-sum) for
// k_fo_wgrad_out. Bound by shared-memory reads (8 per 16 multiply-adds). 32 x 32 over
// 4 x 64^3 points: about 320 us (829 us, and 510 us for the bias alone, by the 64 x 64 tile GEMM).
// Three blocks per SM (80 registers): the gradients of the 64^3 network take 0.36 ms less than with two.
constexpr int kWgT = 256, kWgK = 64, kWgChunk = 1024;

inline size_t wg_smem(int M, int Nn) { return 2 * (size_t)(M + Nn) * (kWgK + 1) * sizeof(float); }

__device__ __forceinline__ void cp_async4(float *dst, const float *src, bool in) {
  // zero fill where the point does not exist
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src),
               "r"(in ? 4 : 0)
               : "memory");
}

__global__ void __launch_bounds__(kWgT, 3)
    k_fo_wgrad(const float *A, int M, const float *Bm, int Nn, long long ng, long long chunks_b, double *part) {
  extern __shared__ __align__(16) unsigned char fo_smem[];
  constexpr int ld = kWgK + 1;
  float *tile = reinterpret_cast<float *>(fo_smem);
  const int tile_n = (M + Nn) * ld;  // two tiles: the next one arrives while this one is summed
  const long long b = blockIdx.x / chunks_b, kbeg = (blockIdx.x - b * chunks_b) * kWgChunk;
  const long long kend = min(kbeg + kWgChunk, ng);
  const int n_tiles = (int)((kend - kbeg + kWgK - 1) / kWgK);
  const int N1 = Nn + 1, tm = (M + 3) / 4, tn = (N1 + 3) / 4, T = tm * tn;
  const int KS = T <= kWgT ? kWgT / T : 0;             // point slices; 0: more tiles than threads (64 x 65)
  const int passes = KS > 0 ? 1 : (T + kWgT - 1) / kWgT, step = KS > 0 ? KS : 1;
  double *o = part + (long long)blockIdx.x * M * N1;
  auto load = [&](int it) {
    const long long k0 = kbeg + (long long)it * kWgK;
    float *dst = tile + (it & 1) * tile_n;
    for (int l = threadIdx.x; l < (M + Nn) * kWgK; l += kWgT) {
      const int c = l / kWgK, k = l % kWgK;
      const bool in = k0 + k < kend;
      const float *src = c < M ? A + (b * M + c) * ng : Bm + (b * Nn + c - M) * ng;
      cp_async4(dst + c * ld + k, src + (in ? k0 + k : kbeg), in);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  for (int pass = 0; pass < passes; ++pass) {
    const int ks = KS > 0 ? threadIdx.x / T : 0, t = KS > 0 ? threadIdx.x - ks * T : threadIdx.x + pass * kWgT;
    const bool act = KS > 0 ? ks < KS : t < T;
    const int i0 = act ? (t % tm) * 4 : 0, j0 = act ? (t / tm) * 4 : 0;
    const int ones = Nn - j0;  // local index of the column of ones (>= 4: not in this tile)
    float acc[4][4], hi[4], lo[4];
    int ar[4], br[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      ar[i] = min(i0 + i, M - 1) * ld;
      br[i] = (M + min(j0 + i, Nn - 1)) * ld;
      hi[i] = lo[i] = 0.f;
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
    }
    load(0);
    for (int it = 0; it < n_tiles; ++it) {
      if (it + 1 < n_tiles) {
        load(it + 1);
        asm volatile("cp.async.wait_group 1;" ::: "memory");
      } else {
        asm volatile("cp.async.wait_group 0;" ::: "memory");
      }
      __syncthreads();
      const float *s = tile + (it & 1) * tile_n;
      if (act)
#pragma unroll 4
        for (int k = ks; k < kWgK; k += step) {
          float x[4], y[4];
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            x[i] = s[ar[i] + k];
            y[i] = s[br[i] + k];
          }
#pragma unroll
          for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(x[i], y[j], acc[i][j]);
          if (ones < 4)
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              const float t = hi[i] + x[i], z = t - hi[i];
              lo[i] += (hi[i] - (t - z)) + (x[i] - z);
              hi[i] = t;
            }
        }
      __syncthreads();
    }
    // the point slices of each tile, in slice order
    for (int q = 0; q < step; ++q) {
      __syncthreads();
      if (act && ks == q)
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int j = 0; j < 4; ++j)
            if (i0 + i < M && j0 + j < N1) {
              double *d = o + (long long)(i0 + i) * N1 + j0 + j;
              const double v = j == ones ? (double)hi[i] + (double)lo[i] : (double)acc[i][j];
              *d = q == 0 ? v : *d + v;
            }
    }
  }
}

// part[chunk][i] = sum over a chunk of the points k = b ng + r of A[b][i][r], one FP32 addition after the
// other. The order is part of the result: a bias gradient is a sum that cancels, so its last digits are those of the
// order of its additions. A lane of the last warp adds the points of a row, from a ring of tiles that the
// other warps keep three ahead. Bound by the chain of 4096 additions and the latency of the tiles: 43 us for 32
// rows over 4 x 64^3 points (24 us for one row).
constexpr int kBsLoad = 256, kBsT = kBsLoad + 32, kBsRows = 32, kBsP = 64, kBsStages = 4;
__global__ void __launch_bounds__(kBsT)
    k_fo_row_sums(const float *A, int M, long long ng, long long K, long long kchunk, double *part) {
  __shared__ float tile[kBsStages][kBsRows * (kBsP + 1)];
  const int m0 = blockIdx.y * kBsRows, rows = min(kBsRows, M - m0);
  const long long kbeg = (long long)blockIdx.x * kchunk, kend = min(kbeg + kchunk, K);
  const int n_tiles = (int)((kend - kbeg + kBsP - 1) / kBsP), m = (int)threadIdx.x - kBsLoad;
  const int p = threadIdx.x % kBsP;  // the same point of every row of a tile
  long long k = kbeg + p, b = k / ng, r = k - b * ng;
  auto load = [&](int it) {  // tiles in order; past the last one an empty group
    if (it < n_tiles) {
      const bool in = k < kend;
      const float *src = in ? A + (b * M + m0) * ng + r : A;
      for (int c = threadIdx.x / kBsP; c < rows; c += kBsLoad / kBsP)
        cp_async4(&tile[it % kBsStages][c * (kBsP + 1) + p], src + (in ? c * ng : 0), in);
      k += kBsP;
      for (r += kBsP; r >= ng; r -= ng) ++b;
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  float s = 0.f;
  if (m < 0)
    for (int it = 0; it < kBsStages - 1; ++it) load(it);
  for (int it = 0; it < n_tiles; ++it) {
    if (m < 0) asm volatile("cp.async.wait_group %0;" ::"n"(kBsStages - 2) : "memory");
    __syncthreads();  // tile `it` is there, and the one before it is summed: its place is free
    if (m < 0) {
      load(it + kBsStages - 1);
    } else if (m < rows) {
      const float *row = tile[it % kBsStages] + m * (kBsP + 1);
      float v[kBsP];
#pragma unroll
      for (int q = 0; q < kBsP; ++q) v[q] = row[q];
#pragma unroll
      for (int q = 0; q < kBsP; ++q) s += v[q];
    }
  }
  if (m >= 0 && m < rows) part[(long long)blockIdx.x * M + m0 + m] = (double)s;
}

// FP64 sums g[M][Nn + 1] (the last column as pairs of floats) and plain[M] (in order, k_fo_row_sums) -> weight
// gradient [M][Nn] and bias gradient [M]. The bias gradient is the plain sum, infinities included, unless
// cancellation leaves it less than ten right bits: then it is the sum of the pairs.
__global__ void k_fo_wgrad_out(const double *g, const double *plain, int M, int Nn, float *w, float *bias) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= M * (Nn + 1)) return;
  const int i = t / (Nn + 1), j = t - i * (Nn + 1);
  if (j < Nn)
    w[i * Nn + j] = (float)g[t];
  else if (bias)
    bias[i] = (float)(fabs(plain[i] - g[t]) > 0x1p-10 * fabs(g[t]) ? g[t] : plain[i]);
}

}  // namespace sbse
