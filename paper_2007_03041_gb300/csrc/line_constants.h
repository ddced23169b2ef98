// Host-side constants of one sweep: the quadrature weights and decay factors
// a kernel reads, from the FP64 table of csrc/coeffs.cpp (Sec. 2.3-2.4).
#pragma once

#include <cmath>

#include "coeffs.h"
#include "sweep.cuh"

namespace molt {

// FP32 constants of the residual form of D_0.  With d_0 = delta^2 g(x),
// x = delta^2,
//   g(x) = f0 + f1 (2 + x) - kap (1+q) / ((1-q)^2 - q x),
// rounding q by delta shifts the relative symbol by delta (1 + 2q/(1-q)) between
// its low and its high end: 1.3e-7 at nu = 0.5, a change of the wave speed that
// a run accumulates.  kap, f0 and f1 are therefore fitted to the q the scans run
// (least squares of the relative error of g at wavelengths of 2, 4, .. 128
// points): first kap, rounded to FP32, then f0 and f1 against the rounded kap.
// Largest relative error of the symbol, nearest constants / fitted, 6-point
// rule: nu = 0.1 2.5e-7 / 1.3e-7, 0.3 1.5e-7 / 6.2e-8, 0.6 1.4e-7 / 2.5e-8, 1.0
// 6.5e-8 / 6.5e-9.  p = 1 - e^{-nu} in full precision; the 3-point rule keeps
// f1 = 0 (the kernels skip its taps).
inline void fit_residual_f32(SweepArgs& a, double q, double p, bool has_f1) {
  constexpr int K = 7;
  // x = -4 sin^2(pi / 2^(k+1)): a wavelength of 2^(k+1) points
  static constexpr double x[K] = {-4.0, -2.0, -5.8578643762690497e-1, -1.5224093497742647e-1, -3.8429439193539104e-2,
                                  -9.6305466556062275e-3, -2.4090875896552147e-3};
  const double q32 = double(float(q)), p32 = 1.0 - q32, m = has_f1 ? 1.0 : 0.0;
  // relative contributions of f0, f1 and kap to g, the first two orthonormalised
  double A[K], B[K], P[K], r00 = 0.0, r01 = 0.0, r11 = 0.0;
  for (int k = 0; k < K; ++k) {
    const double w = 1.0 / (a.f0 + a.f1 * (2.0 + x[k]) - a.kap * (1.0 + q) / (p * p - q * x[k]));
    A[k] = w;
    B[k] = m * (2.0 + x[k]) * w;
    P[k] = -w * (1.0 + q32) / (p32 * p32 - q32 * x[k]);
    r00 += A[k] * A[k];
  }
  r00 = std::sqrt(r00);
  for (int k = 0; k < K; ++k) r01 += (A[k] /= r00) * B[k];
  for (int k = 0; k < K; ++k) r11 += (B[k] -= r01 * A[k]) * B[k];
  r11 = has_f1 ? std::sqrt(r11) : 1.0;
  for (int k = 0; k < K; ++k) B[k] /= r11;
  // kap: the pole's part orthogonal to both, against 1
  double pa = 0.0, pb = 0.0, n = 0.0, z = 0.0;
  for (int k = 0; k < K; ++k) {
    pa += A[k] * P[k];
    pb += B[k] * P[k];
  }
  for (int k = 0; k < K; ++k) {
    const double o = P[k] - pa * A[k] - pb * B[k];
    n += o * o;
    z += o;
  }
  const float kap = float(z / n);
  // f0 and f1: what the rounded kap leaves
  double za = 0.0, zb = 0.0;
  for (int k = 0; k < K; ++k) {
    const double left = 1.0 - double(kap) * P[k];
    za += A[k] * left;
    zb += B[k] * left;
  }
  const double f1 = m * zb / r11, f0 = (za - r01 * f1) / r00;
  if (!std::isfinite(kap) || !std::isfinite(f0) || !std::isfinite(f1)) return;
  a.kapf = kap;
  a.f0f = float(f0);
  a.f1f = float(f1);
}

// Fills the weight and decay fields of `a` for lines of N intervals and E
// points per lane (a.g.n, a.bc and a.mode set).  FP32 sweeps run their scans
// with q rounded to FP32 (q32): the powers and boundary constants they meet
// are those of that ratio, so that the periodic image sum and the Dirichlet
// solve close the recurrences the kernel actually runs.  Every form takes
// differences of v, so D of a constant is exactly zero at any rounding.
//   b[]     K_R(x_i) = sum_m b_m d_{i+m}, m = -2..2 (the weights of J sum to
//     1 - q, the taps on its differences to (1 - q) / nu)
//   f0, f1, kap   the residual form of D_0: with N(z) = (1-q/z)(1-qz) -
//     [J(z)(1-qz) + J(1/z)(1-q/z)]/2 = delta^2 (a0 + a1 (z+1/z) + a2 (z^2+1/z^2))
//     and x = delta^2 = z - 2 + 1/z, M(x) = M0 + M1 x + M2 x^2 is divided by
//     (1-q)^2 - q x: M = (Q0 + Q1 x)((1-q)^2 - q x) + rho, and
//     U + V = -(1+q) delta^2 v / ((1-q)^2 - q x) gives kap = -rho/(1+q),
//     f0 = Q0 - 2 Q1, f1 = Q1.  Q0 and Q1 are below 0.03 up to nu = 1.2; those of
//     the 5- and 6-point rules grow like e^{3 nu}, and past kResidualMax (nu = 1.66
//     and 2.08), where their cancellation against kap (U + V) would show in the
//     last digits, the K filters run.  The 3-point rule's stay below 0.04.
constexpr double kResidualMax = 0.125;
// linear: the sweep reads the FP32 residual form (not with WENO-Z weights).
inline void set_line_constants(SweepArgs& a, const QuadTable& qt, int N, int E, bool f32_sweeps, bool linear = true) {
  const double nu = qt.nu, qx = qt.q;
  const double* c = qt.c;
  // difference taps
  const double b[5] = {c[0], c[0] + c[1], c[0] + c[1] + c[2] + qx, -(c[4] + c[5]), -c[5]};
  for (int i = 0; i < 5; ++i) a.b[i] = b[i];
  // residual form of D_0
  auto cc = [c](int m) { return m >= -3 && m <= 2 ? c[m + 3] : 0.0; };
  double h[4];
  for (int m = 0; m < 4; ++m) h[m] = 0.5 * (cc(m) - qx * cc(m - 1) + cc(-m) - qx * cc(-m - 1));
  const double n1 = -qx - h[1], n2 = -h[2], n3 = -h[3];
  const double a0 = n1 + 2.0 * n2 + 3.0 * n3, a1 = n2 + 2.0 * n3, a2 = n3;
  const double M0 = a0 + 2.0 * a1 + 2.0 * a2, M1 = a1 + 4.0 * a2, M2 = a2;
  const double p = -std::expm1(-nu), xs = p * p / qx;
  const double Q1 = -M2 / qx, Q0 = (Q1 * p * p - M1) / qx;
  a.f0 = Q0 - 2.0 * Q1;
  a.f1 = Q1;
  a.kap = -(M0 + xs * (M1 + xs * M2)) / (1.0 + qx);
  a.d0 = std::fabs(Q0) + std::fabs(Q1) <= kResidualMax ? 1 : 0;   // NaN: the K filters
  if (!a.d0) {
    a.f0 = a.f1 = 0.0;
    a.kap = 0.5;
  }
  // WENO-Z substencil rules on the differences (csrc/sweep.cuh, wenoz_defect)
  a.wk[0] = qt.sub[0][0] + qt.sub[0][1];
  a.wk[1] = qt.sub[0][0];
  a.wk[2] = 1.0 - qt.sub[1][2];
  a.wk[3] = qt.sub[1][0];
  a.wk[4] = qt.sub[2][0] + qx;
  a.wk[5] = -qt.sub[2][2];
  for (int r = 0; r < 3; ++r) a.d[r] = qt.d[r];
  // decays
  // (clamped where q vanishes beside 1 in the arithmetic: 1/q stays finite)
  double lq = std::fmax(f32_sweeps ? std::log(double(float(qx))) : -nu, f32_sweeps ? -40.0 : -300.0);
  double pw = 1.0;
  for (int k = 0; k < 13; ++k, pw *= 2.0) a.qp[k] = std::exp(lq * pw);
  const int n = a.g.n, span = 32 * E;
  a.qlast = std::exp(lq * double((n - 1) % E + 1));
  a.qlw = std::exp(lq * double((n - 1) % span + 1));
  // boundary constants (Sec. 2.3, 3.3), of scans whose first position adds
  // its decay: periodic C = T/(1 - mu); D_0 between Dirichlet walls from the
  // 2x2 system with determinant 1 - mu^2; one-sided Dirichlet D start from 0
  a.kA = a.kB = 0.0;
  a.close = 0;
  if (a.bc == 0) {
    a.kA = 1.0 / (-std::expm1(lq * double(N)));
    a.close = 1;
  } else if (a.mode == MODE_0) {
    const double k = std::exp(-lq) / (-std::expm1(2.0 * lq * double(N)));
    a.kA = std::exp(lq * double(N)) * k;
    a.kB = -k;
    a.close = 2;
  }
  a.kAh = float(a.kA);
  a.kAl = float(a.kA - double(a.kAh));
  a.kBh = float(a.kB);
  a.kBl = float(a.kB - double(a.kBh));
  // one-sided derivatives alpha D: D carries the factor (1-q)/(1-q32); the
  // two-sided linear kernels of a Hamilton-Jacobi pass take it in their taps
  const double al = f32_sweeps ? a.alpha * std::expm1(lq) / std::expm1(-nu) : a.alpha;
  a.alphaf = float(al);
  if (a.mode == MODE_RL)
    for (int i = 0; i < 5; ++i) a.b[i] *= al;
  // FP32 copies
  for (int i = 0; i < 5; ++i) a.bf[i] = float(a.b[i]);
  a.f0f = float(a.f0);
  a.f1f = float(a.f1);
  a.kapf = float(a.kap);
  if (f32_sweeps && linear && a.d0 && a.mode == MODE_0) fit_residual_f32(a, qx, p, a.f1 != 0.0);
  for (int i = 0; i < 6; ++i) a.wkf[i] = float(a.wk[i]);
  for (int r = 0; r < 3; ++r) a.df[r] = float(a.d[r]);
  for (int k = 0; k < 13; ++k) a.qpf[k] = float(a.qp[k]);
  a.qlastf = float(a.qlast);
  a.qlwf = float(a.qlw);
}

}  // namespace molt
