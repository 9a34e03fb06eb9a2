"""Tables of the kinetic operators (csrc/kin_tables.h) against an operator built here: the register
transform's structure with its FP32 constants, everything else in 64 bits, so that only the errors that every
step repeats are left."""
import os
import shutil
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2205_06690_gb300", "csrc")

PROGRAM = r"""
#include <stdio.h>
#include <stdlib.h>
#include "kin_tables.h"
int main(int argc, char **argv) {
  const int n = atoi(argv[1]), pairs = atoi(argv[2]);
  std::vector<sbse::Cd> K(n);
  std::vector<double> w(n);
  for (int m = 0; m < n; ++m) {
    double re, im;
    if (scanf("%lf %lf %lf", &re, &im, &w[m]) != 3) return 1;
    K[m] = sbse::Cd(re, im);
  }
  const sbse::KinAxes a = sbse::kin_axes(K, w, pairs != 0);
  for (const auto *t : {&a.xy, &a.z})
    for (const sbse::Cd &e : *t) printf("%.17g %.17g\n", e.real(), e.imag());
  printf("%.17g 0\n", a.error);
  return 0;
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("kin")
    (d / "t.cpp").write_text(PROGRAM)
    subprocess.run([cxx, "-O2", "-std=c++17", "-Wall", "-I", CSRC, str(d / "t.cpp"), "-o", str(d / "t")], check=True)
    return str(d / "t")


def _fp32(z):
    return z.real.astype(np.float32).astype(np.float64) + 1j * z.imag.astype(np.float32)


def _transform(x, sign):
    """Rows of x through the mixed-radix Stockham stages (4, then 2, 3, 5) with constants rounded to FP32."""
    n = x.shape[1]
    tw = _fp32(np.exp(-2j * np.pi * np.arange(n) / n))
    tw = np.conj(tw) if sign > 0 else tw
    ns, m = 1, n
    for r in (4, 2, 3, 5):
        while m % r == 0:
            i = 1j * (1 if sign > 0 else -1)
            if r == 4:
                w = np.array([[i ** (p * q % 4) for q in range(4)] for p in range(4)])
            elif r == 2:
                w = np.array([[1, 1], [1, -1]], dtype=complex)
            else:
                c = np.concatenate([[1.0], tw[n // r * np.arange(1, (r + 1) // 2)]])
                c = np.concatenate([c, np.conj(c[:0:-1])])
                if r == 3:
                    c = np.array([1.0, -0.5 + 1j * c[1].imag, -0.5 + 1j * c[2].imag])
                w = c[np.outer(np.arange(r), np.arange(r)) % r]
            y = np.empty_like(x)
            for j in range(n // r):
                jm = j % ns
                a = np.stack([x[:, j + q * (n // r)] * (tw[q * jm * (n // (ns * r)) % n] if q * jm else 1.0)
                              for q in range(r)])
                y[:, (j // ns) * ns * r + jm + ns * np.arange(r)] = (w @ a).T
            x, m, ns = y, m // r, ns * r
    return x


def _operator(x, table, pairs):
    """One kinetic operator on the rows of x: full pencils, or even and odd samples on the two lanes of a pair."""
    if not pairs:
        return _transform(_transform(x, -1) * table, +1)
    kp, m1, m2 = table.reshape(3, -1)
    e, o = _transform(x[:, 0::2], -1), _transform(x[:, 1::2], -1)
    y = np.empty_like(x)
    y[:, 0::2], y[:, 1::2] = _transform(e * kp + o * m1, +1), _transform(o * kp + e * m2, +1)
    return y


@pytest.mark.parametrize("n,pairs", [(8, 0), (10, 0), (16, 0), (18, 0), (20, 0), (24, 0), (25, 0), (27, 0), (30, 0), (36, 0),
                                     (40, 0), (45, 0), (48, 0), (50, 0), (54, 0), (60, 0), (32, 1), (48, 1), (64, 1), (80, 1),
                                     (96, 1)])
@pytest.mark.parametrize("spacing", [0.25, 1.0 / 3.0, 0.45])
def test_errors_of_every_step_stay_below_half_an_ulp(program, n, pairs, spacing):
    """x, y and z operator together, root mean square over orbitals' momenta: 2^-24, where a single rounding of
    each axis's table and the transforms' gains give up to 2.4e-7."""
    k = 2.0 * np.pi / (n * spacing) * np.fft.fftfreq(n) * n
    K, weight = np.exp(-0.025j * k * k), np.exp(-0.5 * k * k)
    lines = "\n".join("%.17g %.17g %.17g" % v for v in zip(K.real, K.imag, weight))
    out = subprocess.run([program, str(n), str(pairs)], input=lines, capture_output=True, text=True, check=True).stdout
    v = np.array([[float(t) for t in row.split()] for row in out.split("\n") if row])
    t = v[:, 0] + 1j * v[:, 1]
    xy, z, claimed = t[:(len(t) - 1) // 2], t[(len(t) - 1) // 2:-1], v[-1, 0]
    assert np.array_equal(xy, _fp32(xy)) and np.array_equal(z, _fp32(z))
    waves = np.exp(2j * np.pi * np.outer(np.arange(n), np.arange(n)) / n)
    f = [np.sum(np.conj(waves) * _operator(waves, a, pairs), axis=1) / n / K for a in (xy, z)]
    p = weight / weight.sum()
    scale = np.sum(p * f[0]).real  # the planes' operators carry a scale that the z operator takes back
    ex, ez = f[0] / scale - 1.0, f[1] * scale ** 2 - 1.0
    mx, mz = np.sum(p * ex), np.sum(p * ez)
    err = np.sqrt(2 * np.sum(p * abs(ex - mx) ** 2) + np.sum(p * abs(ez - mz) ** 2) + abs(2 * mx + mz) ** 2)
    assert err <= 2.0 ** -24
    assert abs(err - claimed) <= 1e-9 + 0.05 * claimed
    assert 0.74 < scale < 1.26
