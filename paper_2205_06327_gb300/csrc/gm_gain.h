// How much the rounded constants of a generic window's line transform scale
// each frequency (plain C++, so that it can be checked on the host).
#pragma once

#include <algorithm>
#include <cmath>
#include <complex>
#include <vector>

namespace ptycho {

namespace gain_detail {

using cd = std::complex<double>;

inline cd rounded(cd w) { return cd((float)w.real(), (float)w.imag()); }
inline cd root(int M, int e) {  // exp(-2 pi i e / M)
  const double ang = -6.283185307179586476925287 * (double)(e % M) / M;
  return cd(std::cos(ang), std::sin(ang));
}

// dft_r<R> (forward) with its FP32 constants, evaluated in FP64.
inline void dft_host(int R, cd* x) {
  if (R == 2) {
    const cd a = x[0];
    x[0] = a + x[1];
    x[1] = a - x[1];
  } else if (R == 3) {
    const cd a = x[0], t1 = x[1] + x[2], t2 = a - 0.5 * t1;
    const cd m = cd(0, -1) * ((double)(float)0.86602540378443864676 * (x[1] - x[2]));
    x[0] = a + t1;
    x[1] = t2 + m;
    x[2] = t2 - m;
  } else if (R == 4) {
    const cd t0 = x[0] + x[2], t1 = x[0] - x[2], t2 = x[1] + x[3], t3 = cd(0, -1) * (x[1] - x[3]);
    x[0] = t0 + t2;
    x[2] = t0 - t2;
    x[1] = t1 + t3;
    x[3] = t1 - t3;
  } else {  // one Cooley-Tukey step, R = R1 R2 (radix 8: even and odd samples)
    const int R1 = R == 6 ? 2 : R == 9 ? 3 : 4, R2 = R / R1;
    cd y[16], u[16];
    for (int n2 = 0; n2 < R2; ++n2) {
      for (int n1 = 0; n1 < R1; ++n1) u[n1] = x[R2 * n1 + n2];
      dft_host(R1, u);
      for (int k1 = 0; k1 < R1; ++k1) y[n2 * R1 + k1] = u[k1] * rounded(root(R, n2 * k1));
    }
    for (int k1 = 0; k1 < R1; ++k1) {
      for (int n2 = 0; n2 < R2; ++n2) u[n2] = y[n2 * R1 + k1];
      dft_host(R2, u);
      for (int k2 = 0; k2 < R2; ++k2) x[k1 + R1 * k2] = u[k2];
    }
  }
}

// D[k][n] of the radix-R transform, row by column.
inline std::vector<cd> dft_matrix(int R) {
  std::vector<cd> D((size_t)R * R), e(R);
  for (int n = 0; n < R; ++n) {
    std::fill(e.begin(), e.end(), cd(0));
    e[n] = 1;
    if (R > 1) dft_host(R, e.data());
    for (int k = 0; k < R; ++k) D[(size_t)k * R + n] = e[k];
  }
  return D;
}

}  // namespace gain_detail

// The rounded constants of a transform do not only scatter its result: the
// component that a forward and inverse pair should return unchanged comes
// back scaled, by a factor that depends on the frequency alone and repeats in
// every propagation, so that over a chain it outgrows the rounding of the
// arithmetic (14 propagations of 192 points, emulated: 9.5e-7 from the
// constants alone, 5.9e-7 from the arithmetic alone, 1.06e-6 together, 6.2e-7
// with the factor divided out).  gain[k] is that factor for the radices R1 R2
// R3 of an instance (R2 = 1: two); the propagator table is divided by it.
inline void gm_transform_gain(int R1, int R2, int R3, double* gain) {
  using namespace gain_detail;
  const int M = R1 * R2 * R3, MI = R2 * R3;
  const std::vector<cd> D1 = dft_matrix(R1), D2 = dft_matrix(R2), D3 = dft_matrix(R3);
  // forward (by output frequency) and inverse (by input frequency) gains of
  // the outer radix
  std::vector<cd> f1(R1), i1(R1);
  for (int k = 0; k < R1; ++k)
    for (int n = 0; n < R1; ++n) {
      const cd tone = std::conj(root(R1, k * n));
      f1[k] += D1[(size_t)k * R1 + n] * tone / (double)R1;
      i1[k] += std::conj(D1[(size_t)n * R1 + k] * tone) / (double)R1;
    }
  std::vector<cd> w(M), wr(M);  // exp(-2 pi i e / M), exact and rounded
  for (int e = 0; e < M; ++e) wr[e] = rounded(w[e] = root(M, e));
  for (int k = 0; k < M; ++k) {
    const int k1 = k % R1, kap = k / R1, k2 = kap % R2, k3 = kap / R2;
    cd f = 0, b = 0;
    for (int j = 0; j < MI; ++j) {
      const int j2 = j % R3, q2 = j / R3;
      // the tone, with the first split's twiddle as rounded / exact, and the
      // second split's twiddle
      cd u = std::conj(w[R1 * (kap * j % MI)]) * wr[k1 * j] * std::conj(w[k1 * j]);
      if (R2 > 1) u *= wr[R1 * k2 * j2];
      f += D2[(size_t)k2 * R2 + q2] * D3[(size_t)k3 * R3 + j2] * u;
      b += std::conj(D2[(size_t)q2 * R2 + k2] * D3[(size_t)j2 * R3 + k3] * u);
    }
    gain[k] = std::abs(f1[k1] * i1[k1] * f * b) / ((double)MI * MI);
  }
}

}  // namespace ptycho
