// Multiplier tables of the one-dimensional kinetic operators F^-1 diag(K) F in FP32 (host only, no CUDA).
//
// A propagation applies the same operator thousands of times, so an error that is the same in every step adds up
// in proportion to the steps, while rounding errors of the data add up like their square root. Two errors are the
// same in every step: the transforms' constants are rounded, which gives each frequency a gain of 1 +- 4e-8, and so
// are the table's entries (1 +- 6e-8). The first is computed here and divided out of the table. The second depends
// on the table's scale: the x and y operators take K scaled by s, the z operator by 1 / (N^3 s^2), and s is
// searched for the pair of tables whose errors, weighted over the frequencies that orbitals hold, are least
// (about 0.5 ms, once per grid and time step). The sum over three axes stays near 3e-8 per step; with K / N rounded
// on every axis it was up to 2.4e-7, and on 20, 30 and 40 points W of 60 steps was 2 to 3 times as far from 64 bits as
// with 3D transforms. Error of W against 64 bits (200 steps; 3D transforms, or one table for the lane pairs of
// 80 and 96, against these): 20^3 2.3e-6, 6.1e-7; 30^3 8.1e-7, 7.9e-7; 40^3 1.8e-6, 8.1e-7; 48^3 9.4e-6, 1.1e-6;
// 60^3 2.3e-6, 2.1e-6; 64^3 4.5e-6, 3.3e-6; 96^3 1.1e-5, 6.8e-6.
#pragma once

#include <math.h>

#include <algorithm>
#include <complex>
#include <vector>

namespace sbse {

using Cd = std::complex<double>;

inline Cd round32(Cd z) { return Cd((double)(float)z.real(), (double)(float)z.imag()); }

// the register transform (fft_reg.cuh: radix 4, then 2, 3, 5, Stockham order) forward, with its FP32 constants
inline void transform_of_constants(std::vector<Cd> &x) {
  const int n = (int)x.size();
  std::vector<Cd> tw(n), w(n);
  for (int k = 0; k < n; ++k) {
    const double a = -2.0 * M_PI * (double)k / (double)n;
    tw[k] = round32(Cd(cos(a), sin(a)));
  }
  int m = n, ns = 1;
  for (int r : {4, 2, 3, 5})
    for (; m % r == 0; m /= r, ns *= r) {
      const int nb = n / r;
      for (int j = 0; j < nb; ++j) {
        const int jm = j % ns;
        Cd in[5];
        for (int q = 0; q < r; ++q) in[q] = x[j + q * nb] * (q * jm == 0 ? Cd(1.0) : tw[(q * jm * (n / (ns * r))) % n]);
        for (int p = 0; p < r; ++p) {
          Cd s = in[0];
          for (int q = 1; q < r; ++q) {
            const int e = p * q % r;  // exp(-2 pi i e / r) as the butterflies hold it
            Cd c = 1.0;
            if (r == 4) c = e == 0 ? Cd(1, 0) : e == 1 ? Cd(0, -1) : e == 2 ? Cd(-1, 0) : Cd(0, 1);
            else if (r == 2) c = e ? -1.0 : 1.0;
            else if (e) c = 2 * e < r ? tw[e * nb] : std::conj(tw[(r - e) * nb]);
            if (r == 3 && e) c = Cd(-0.5, c.imag());
            s += c * in[q];
          }
          w[(j / ns) * ns * r + jm + p * ns] = s;
        }
      }
      x.swap(w);
    }
}

// gain - 1 of each frequency in a forward and an inverse transform (over n); the inverse holds the conjugate of
// every constant
inline std::vector<Cd> transform_gains(int n) {
  std::vector<Cd> wave(n), fwd(n), back(n), col(n);
  for (int x = 0; x < n; ++x) wave[x] = Cd(cos(2.0 * M_PI * x / n), sin(2.0 * M_PI * x / n));
  for (int x = 0; x < n; ++x) {  // column x of the transform
    std::fill(col.begin(), col.end(), 0.0);
    col[x] = 1.0;
    transform_of_constants(col);
    for (int m = 0; m < n; ++m) {
      fwd[m] += col[m] * wave[(long long)m * x % n];
      back[x] += col[m] * wave[(long long)m * x % n];
    }
  }
  for (int m = 0; m < n; ++m) fwd[m] = fwd[m] / (double)n * std::conj(back[m] / (double)n) - 1.0;
  return fwd;
}

// The table of K for one thread per pencil (N entries) or for a lane pair (Kp, M1, M2 of N / 2 entries each: even
// outputs from E Kp + O M1, odd ones from O Kp + E M2, see fft_pair.cuh), with the gains of the N or N / 2 point
// transforms divided out; to be scaled and rounded
inline std::vector<Cd> kin_table(const std::vector<Cd> &K, const std::vector<Cd> &gain, bool pairs) {
  const int n = (int)K.size(), h = n / 2;
  std::vector<Cd> t(pairs ? 3 * h : n);
  for (int m = 0; !pairs && m < n; ++m) t[m] = K[m] / (1.0 + gain[m]);
  for (int k = 0; pairs && k < h; ++k) {
    const Cd w(cos(2.0 * M_PI * k / n), -sin(2.0 * M_PI * k / n)), d = (K[k] - K[k + h]) / (1.0 + gain[k]);
    t[k] = (K[k] + K[k + h]) / (1.0 + gain[k]);
    t[h + k] = w * d;
    t[2 * h + k] = std::conj(w) * d;
  }
  return t;
}

struct KinAxes {
  std::vector<Cd> xy, z;  // FP32 values
  double error;           // of the three axes' product, rms over the weights
};

// tables of the two sweeps for one-dimensional factors K (|K| = 1) with weights over the frequencies
inline KinAxes kin_axes(const std::vector<Cd> &K, const std::vector<double> &weight, bool pairs) {
  const int n = (int)K.size(), h = n / 2;
  const std::vector<Cd> gain = transform_gains(pairs ? h : n), table = kin_table(K, gain, pairs);
  double total = 0.0;
  for (double w : weight) total += w;
  // Error of the operator at a frequency: that of the entries it takes, times `to` (one thread per pencil: entry m;
  // lane pair: the mean of the even and the odd outputs). Frequencies below 1e-6 of the weights do not count.
  struct Term {
    double weight;
    int k;
    Cd to, wave;
  };
  std::vector<Term> terms;
  for (int m = 0; m < n; ++m)
    if (weight[m] > 1e-6 * total)
      terms.push_back({weight[m] / total, pairs ? m % h : m, (1.0 + gain[pairs ? m % h : m]) * std::conj(K[m]),
                       Cd(cos(2.0 * M_PI * m / n), sin(2.0 * M_PI * m / n))});
  auto off = [&](double s, int i) { return round32(s * table[i]) - s * table[i]; };
  // mean of the relative error over the weights, and its variance
  auto moments = [&](double s, Cd *mean) {
    Cd mu = 0.0;
    double sq = 0.0;
    for (const Term &t : terms) {
      Cd e = off(s, t.k);
      if (pairs) e = 0.5 * (e + 0.5 * (off(s, h + t.k) * t.wave + off(s, 2 * h + t.k) * std::conj(t.wave)));
      e *= t.to / s;
      mu += t.weight * e;
      sq += t.weight * std::norm(e);
    }
    *mean = mu;
    return sq - std::norm(mu);
  };
  double best = INFINITY, scale = 1.0 / n;
  for (int j = -512; j <= 512; ++j) {  // a quarter either way of 1 / N: the data between the sweeps keep their size
    const double s = (1.0 + j / 2048.0) / n;
    Cd mxy, mz;
    const double vxy = moments(s, &mxy), vz = moments(1.0 / ((double)n * n * n * s * s), &mz);
    const double err = std::max(0.0, 2.0 * vxy + vz) + std::norm(2.0 * mxy + mz);
    if (err < best) {
      best = err;
      scale = s;
    }
  }
  KinAxes r{table, table, sqrt(best)};
  for (Cd &e : r.xy) e = round32(scale * e);
  for (Cd &e : r.z) e = round32(1.0 / ((double)n * n * n * scale * scale) * e);
  return r;
}

}  // namespace sbse
