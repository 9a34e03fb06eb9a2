// Lane-pair pencils: a pencil of N = 2H points is split over a lane pair (l, l ^ 16) of one warp, each lane
// holding H of them, so that the transforms of long pencils, or more warps of short ones, fit in the
// registers (fft_split.cu). Included by the translation units that use it, each with its own twiddles.
#pragma once

#include <math.h>

#include <type_traits>

#include "bounds.cuh"
#include "fft_reg.cuh"
#include "kernels.h"
#include "passes.cuh"
#include "tma.cuh"

namespace sbse {

namespace {

__constant__ float2 c_tws[kRegTotal];

struct TwS {
  __device__ __forceinline__ static float2 get(int i) { return c_tws[i]; }
};

constexpr unsigned kFull = 0xffffffffu;

// exp(SIGN 2 pi i k / N)
template <int N, int SIGN> __device__ __forceinline__ float2 tw_full(int k) {
  float2 w = TwS::get(reg_offset(N) + k);
  if (SIGN > 0) w.y = -w.y;
  return w;
}

__device__ __forceinline__ float2 shfl_pair(float2 v) {
  return make_float2(__shfl_xor_sync(kFull, v.x, 16), __shfl_xor_sync(kFull, v.y, 16));
}

// Decimation in time across the lane pair. On entry lane s of the pair holds x[2m + s], m < H;
// on return it holds X[s Q + j] in v[j] and X[H + s Q + j] in v[Q + j] (j < Q = H / 2), where
// X[k] = sum_n x[n] exp(SIGN 2 pi i n k / N): X[k] = E[k] + W^k O[k], X[k + H] = E[k] - W^k O[k]
// with E, O the H-point transforms of the even and odd samples.
template <int N, int SIGN> __device__ __forceinline__ void fft2_dit(float2 (&v)[N / 2], int s) {
  constexpr int H = N / 2, Q = H / 2;
  fft_reg<float, H, SIGN, TwS>(v);
#pragma unroll
  for (int j = 0; j < Q; ++j) {
    // lane 0 keeps E[j] and needs O[j]; lane 1 keeps O[Q + j] and needs E[Q + j]
    const float2 rcv = shfl_pair(s ? v[j] : v[Q + j]);
    const float2 e = s ? rcv : v[j];
    const float2 o = s ? v[Q + j] : rcv;
    float2 t = cmul(o, tw_full<N, SIGN>(j));
    if (s) t = cmul_si(t, SIGN);  // W^Q = exp(SIGN i pi / 2) = SIGN i
    v[j] = cadd(e, t);
    v[Q + j] = csub(e, t);
  }
}

// Decimation in frequency across the lane pair: the inverse of the layout change above. On entry
// lane s holds X[s Q + j] in v[j] and X[H + s Q + j] in v[Q + j]; on return it holds x[2m + s] in
// v[m], x[n] = sum_k X[k] exp(SIGN 2 pi i n k / N). The even outputs are the H-point transform of
// a_k = X[k] + X[k + H], the odd ones that of b_k = (X[k] - X[k + H]) W^k; lane 0 gathers every
// a_k and lane 1 every b_k.
template <int N, int SIGN> __device__ __forceinline__ void fft2_dif(float2 (&v)[N / 2], int s) {
  constexpr int H = N / 2, Q = H / 2;
#pragma unroll
  for (int j = 0; j < Q; ++j) {
    const float2 a = cadd(v[j], v[Q + j]);
    float2 b = cmul(csub(v[j], v[Q + j]), tw_full<N, SIGN>(j));
    if (s) b = cmul_si(b, SIGN);
    const float2 rcv = shfl_pair(s ? a : b);
    v[j] = s ? rcv : a;
    v[Q + j] = s ? b : rcv;
  }
  fft_reg<float, H, SIGN, TwS>(v);
}

// One-dimensional kinetic operator F^-1 diag(K / N) F on the pencil held by a lane pair, without
// leaving registers: on entry lane s holds x[2m + s], on return y[2m + s] (y = F^-1 K F x / N). Each
// lane takes the half-length transform of its samples (E for the even ones, O for the odd ones),
// receives the other lane's, forms E Kp + O M1 (lane 0: even outputs) or O Kp + E M2 (lane 1: odd
// outputs), and transforms back. tab = [Kp | M1 | M2], N/2 entries each (kin_tables.h).
template <int N>
__device__ __forceinline__ void kin_roundtrip(float2 (&v)[N / 2], int s, const float2 *tab) {
  constexpr int H = N / 2;
  fft_reg<float, H, -1, TwS>(v);
  const float2 *mt = tab + (s ? 2 * H : H);
#pragma unroll
  for (int k = 0; k < H; ++k) {
    const float2 o = shfl_pair(v[k]);
    const float2 kp = tab[k], mk = mt[k];
    v[k] = cmac2(v[k], kp, o, mk);
  }
  fft_reg<float, H, +1, TwS>(v);
}


// ------------------------------------------------------------------------------------------
// The pre-operation of a forward plane pass into the padded tile. Thread tid of the plane's 2N covers the
// points t + k 2N (k < N / 2) of the plane, i.e. row t / N + 2k, column t % N.
template <int N, bool PAIR>
__device__ __forceinline__ void preop_plane(const GView<float> &g, const XfwdArgs<float> &a, long long item,
                                            long long off, float2 *S, int tid) {
  using C = float2;
  constexpr int LD = N + 1, NT = 2 * N, KP = N / 2, UB = 8;
  const PreopItem<float> it = preop_item<float>(g, a, item);
  (void)SBSE_IDX(item, a.n_items);
  (void)SBSE_IDX(off + tid + (long long)(KP - 1) * NT, g.ng);  // the largest point this thread reads
  if constexpr (PAIR) (void)SBSE_IDX(item / a.L, a.n_items / a.L);     // the pair of E - 1
  const int y0 = tid / N;
  C *srow = S + y0 * LD + (tid - y0 * N);
  if constexpr (PAIR) {
    const C *dp = it.in + off + tid, *ap = it.a + off + tid, *pp = it.pv + off + tid;
    const C *ep = it.em1 ? it.em1 + off + tid : nullptr;
    // the deferred renormalisation is pending only in the step after a cleaning (cm1 != 0, the same
    // for the whole block): the other steps skip its arithmetic (d is then unchanged by it)
    auto sweep = [&](auto renorm) {
      constexpr bool RN = decltype(renorm)::value;
#pragma unroll 1
      for (int k0 = 0; k0 < KP; k0 += UB) {
        C dv[UB], av[UB], pv[UB], ev[UB];
#pragma unroll
        for (int k = 0; k < UB; ++k) {
          if (k0 + k < KP) {
            const int l = (k0 + k) * NT;
            dv[k] = dp[l];
            av[k] = ap[l];
            pv[k] = pp[l];
            ev[k] = ep ? ep[l] : C{0.f, 0.f};
          }
        }
#pragma unroll
        for (int k = 0; k < UB; ++k)
          if (k0 + k < KP)
            srow[2 * (k0 + k) * LD] =
                pair_phase<float>(pv[k], ev[k], av[k], RN ? renorm_value<float>(dv[k], av[k], it.cm1) : dv[k]);
      }
    };
    if (it.cm1 != 0.f)
      sweep(std::true_type{});
    else
      sweep(std::false_type{});
  } else {
    auto run = [&](auto f) {
#pragma unroll 1
      for (int k0 = 0; k0 < KP; k0 += UB) {
        C v[UB];
#pragma unroll
        for (int k = 0; k < UB; ++k)
          if (k0 + k < KP) v[k] = f(off + tid + (k0 + k) * NT);
#pragma unroll
        for (int k = 0; k < UB; ++k)
          if (k0 + k < KP) srow[2 * (k0 + k) * LD] = v[k];
      }
    };
    if (it.mode == XF_PHASE_A) {
      run([&](long long i) { return cmul(it.pv[i], it.in[i]); });
    } else if (it.mode == XF_PACK_DN) {
      if (it.r1)
        run([&](long long i) { return C{it.r0[i], it.r1[i]}; });
      else
        run([&](long long i) { return C{it.r0[i], 0.f}; });
    } else if (it.mode == XF_PACK_PROD) {
      if (it.r2)
        run([&](long long i) { return C{it.r0[i] * it.r1[i], it.r2[i] * it.r3[i]}; });
      else
        run([&](long long i) { return C{it.r0[i] * it.r1[i], 0.f}; });
    } else {
      run([&](long long i) { return preop_at<float>(g, it, i); });
    }
  }
}


// The potential phase and the x and y kinetic operators of one plane by its 2N threads (tid), stored to
// global; S is the plane's tile. Every thread of the block calls it (it synchronises).
template <int N, bool PAIR>
__device__ __forceinline__ void kin2_plane(const GView<float> &g, const XfwdArgs<float> &a, long long item, long long off,
                                           float2 *S, const float2 *tab, int tid) {
  using C = float2;
  constexpr int LD = N + 1, H = N / 2;
  preop_plane<N, PAIR>(g, a, item, off, S, tid);
  __syncthreads();
  const int lane = threadIdx.x & 31, s = lane >> 4, p = (tid >> 5) * 16 + (lane & 15);
  {  // x operator on row p, in place
    C v[H];
    C *row = S + p * LD;
#pragma unroll
    for (int m = 0; m < H; ++m) v[m] = row[2 * m + s];
    kin_roundtrip<N>(v, s, tab);
    __syncwarp();
#pragma unroll
    for (int m = 0; m < H; ++m) row[2 * m + s] = v[m];
  }
  __syncthreads();
  {  // y operator on column p, stored to global
    C v[H];
    const C *col = S + p;
#pragma unroll
    for (int m = 0; m < H; ++m) v[m] = col[(2 * m + s) * LD];
    kin_roundtrip<N>(v, s, tab);
    (void)SBSE_IDX(off + p + (long long)(N - 1) * N, g.ng);
    C *out = a.out + item * g.ng + off + p;
#pragma unroll
    for (int m = 0; m < H; ++m) out[(2 * m + s) * N] = v[m];
  }
}

int upload_pair_twiddles() {
  float2 hf[kRegTotal];
  for (int s = 0; s < kRegCount; ++s) {
    const int N = kRegSizes[s], off = reg_offset(N);
    for (int k = 0; k < N; ++k) {
      const double a = -2.0 * M_PI * (double)k / (double)N;
      hf[off + k] = make_float2((float)cos(a), (float)sin(a));
    }
  }
  return cudaMemcpyToSymbol(c_tws, hf, sizeof(hf)) == cudaSuccess ? 0 : -1;
}

}  // namespace

}  // namespace sbse
