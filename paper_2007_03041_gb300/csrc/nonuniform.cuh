// Fast summation on non-uniform lines (the point-local quadrature that
// Sec. 2.4 describes for non-uniform meshes): per point i the J_R / J_L
// weights of its own stencil nodes and the cell decay q_i = e^{-alpha (x_i -
// x_{i-1})}; the recurrences I_R(x_i) = q_i I_R(x_{i-1}) + J_R(x_i),
// I_L(x_i) = q_{i+1} I_L(x_{i+1}) + J_L(x_i) close over the period with
// mu = prod q_i = e^{-alpha L} (Sec. 2.3), or on a Dirichlet line start at
// the ends with the boundary constants fixed by the boundary values.
//
// Host side: build_nonuniform_tables() integrates the Lagrange basis of each
// point's stencil against the exponential by 16-point Gauss-Legendre
// quadrature (FP64); pack_nonuniform() brings them into difference form and
// into the order the kernel's lanes read them.  Device side: the scan of
// csrc/sweep.cuh (E consecutive points per lane, both directions at once, one
// CTA barrier per application of D) with a multiplier per point.
#pragma once

#include <cmath>
#include <vector>

#include "sweep.cuh"

namespace molt {

struct NuArgs {
  LineGeom g;
  int mode, P;
  int bc;               // 0 periodic, 1 Dirichlet (nodes x_0 = a .. x_{n-1} = b)
  int nw, LS;           // warps per line, shared line stride (elements)
  int close;            // boundary constants C = kA T_same + kB T_other: 0 none, 1 kA, 2 both
  double kA, kB;
  float kAh, kAl, kBh, kBl;   // kA, kB as FP32 pairs
  const void* tab;      // device tables (pack_nonuniform) in the compute type
  const void* in;
  void* out;
};

// Roots and weights of the n-point Gauss-Legendre rule on [-1, 1] (Newton on
// the three-term recurrence of the Legendre polynomials).
inline void gauss_legendre(int n, double* x, double* w) {
  for (int i = 0; i < n; ++i) {
    double z = std::cos(M_PI * (i + 0.75) / (n + 0.5));
    for (int it = 0; it < 100; ++it) {
      double p0 = 1.0, p1 = z;
      for (int k = 2; k <= n; ++k) {
        const double p2 = ((2.0 * k - 1.0) * z * p1 - (k - 1.0) * p0) / k;
        p0 = p1;
        p1 = p2;
      }
      const double dp = n * (z * p1 - p0) / (z * z - 1.0);
      const double dz = p1 / dp;
      z -= dz;
      if (std::fabs(dz) < 1e-16) {
        x[i] = z;
        w[i] = 2.0 / ((1.0 - z * z) * dp * dp);
        break;
      }
      x[i] = z;
      w[i] = 2.0 / ((1.0 - z * z) * dp * dp);
    }
  }
}

// x_j for any j: periodic images (L > 0, x the nodes of one period), or for a
// Dirichlet line (L == 0, nodes x_0 = a .. x_{n-1} = b, n >= 4) the ghost
// nodes mirrored about the ends, x_{-j} = 2a - x_j, x_{N+j} = 2b - x_{N-j}
// (Sec. 2.3: the stencils reach odd-reflected data there).
inline double nu_node(const std::vector<double>& x, double L, long long j) {
  const long long n = static_cast<long long>(x.size());
  if (L > 0) {
    long long r = j % n;
    if (r < 0) r += n;
    return x[size_t(r)] + double((j - r) / n) * L;
  }
  const long long N = n - 1;
  if (j < 0) return 2.0 * x[0] - x[size_t(-j)];
  if (j > N) return 2.0 * x[size_t(N)] - x[size_t(2 * N - j)];
  return x[size_t(j)];
}

// cR, cL: 6*n (slot-major), q: n.  x: the n nodes of one period [x_0, x_0 + L),
// or (L == 0) of a Dirichlet line.  Dirichlet lines start their recurrences
// at the ends, I_R(x_0) = 0 and I_L(x_N) = 0: J_R(x_0) and J_L(x_N) are zero
// and q_0 = 0, so a scan over the whole line gives exactly those values.
inline void build_nonuniform_tables(const std::vector<double>& x, double L, double alpha, int npts,
                                    std::vector<double>* cR, std::vector<double>* cL, std::vector<double>* q) {
  const int n = int(x.size());
  int lo = -3, hi = 2;                 // J_R stencil offsets (6 points)
  if (npts == 5) hi = 1;
  if (npts == 3) { lo = -1; hi = 1; }
  const int k = hi - lo + 1;
  cR->assign(6 * size_t(n), 0.0);
  cL->assign(6 * size_t(n), 0.0);
  q->assign(n, 0.0);
  constexpr int kG = 16;
  double gx[kG], gw[kG];
  gauss_legendre(kG, gx, gw);
  auto node = [&](long long j) { return nu_node(x, L, j); };
  for (int i = 0; i < n; ++i) {
    const double xi = x[size_t(i)];
    for (int side = 0; side < 2; ++side) {
      // J_R: cell [x_{i-1}, x_i], nodes x_{i+l}; J_L: cell [x_i, x_{i+1}], nodes x_{i-l}
      const double a = side == 0 ? node(i - 1) : xi, b = side == 0 ? xi : node(i + 1);
      double t[6];
      for (int m = 0; m < k; ++m) t[m] = node(side == 0 ? i + lo + m : i - (lo + m)) - xi;
      for (int m = 0; m < k; ++m) {
        double sum = 0.0;
        for (int gq = 0; gq < kG; ++gq) {
          const double s = 0.5 * (b - a) * gx[gq] + 0.5 * (b + a);
          double ell = 1.0;
          for (int r = 0; r < k; ++r)
            if (r != m) ell *= ((s - xi) - t[r]) / (t[m] - t[r]);
          const double kern = side == 0 ? std::exp(-alpha * (xi - s)) : std::exp(-alpha * (s - xi));
          sum += 0.5 * (b - a) * gw[gq] * alpha * kern * ell;
        }
        (side == 0 ? *cR : *cL)[size_t(lo + m + 3) * n + i] = sum;
      }
    }
    (*q)[size_t(i)] = std::exp(-alpha * (xi - node(i - 1)));
  }
  if (!(L > 0)) {
    for (int m = 0; m < 6; ++m) {
      (*cR)[size_t(m) * n] = 0.0;
      (*cL)[size_t(m) * n + n - 1] = 0.0;
    }
    (*q)[0] = 0.0;
  }
}

// WENO-Z tables of the 5-point rule (quadratic substencils S_r = offsets
// {r-3, r-2, r-1}, Sec. 2.4), per point and direction, slot-major [kNuWeno][n]
// (periodic lines, or Dirichlet lines with L == 0 as above):
//   slots 3r+j       c^{(r)}_j: J^{(r)} = sum_j c^{(r)}_j v(node j of S_r)
//   slots 9+r        d_r, the linear weights with sum_r d_r c^{(r)} = c
//   slots 12+3r+j    A_{rj} = l_j'(0), slots 21+3r+j  B_{rj} = l_j''
// in the cell variable t in [-1, 0] (t = (s - x_i)/dx for J_R on
// [x_{i-1}, x_i], t = (x_i - s)/dx for J_L on [x_i, x_{i+1}]), l_j the
// Lagrange basis of S_r.  With a = sum A v and b = sum B v the interpolant has
// p_t = a + b t, so its smoothness indicator int_{-1}^0 p_t^2 + p_tt^2 dt is
// a^2 - a b + 4/3 b^2.  The node of slot j of S_r is x_{i + (r + j - 3)} for
// J_R and x_{i - (r + j - 3)} for J_L.  Since every rule integrates the
// constant exactly (weights summing to 1 - q), d_1 = 1 - d_0 - d_2 once the
// two outer nodes, each in one substencil only, fix d_0 and d_2.
constexpr int kNuWeno = 30;

inline void build_nonuniform_weno_tables(const std::vector<double>& x, double L, double alpha,
                                         std::vector<double>* wR, std::vector<double>* wL) {
  const int n = int(x.size());
  wR->assign(size_t(kNuWeno) * n, 0.0);
  wL->assign(size_t(kNuWeno) * n, 0.0);
  constexpr int kG = 16;
  double gx[kG], gw[kG];
  gauss_legendre(kG, gx, gw);
  auto node = [&](long long j) { return nu_node(x, L, j); };
  // nu int_{-1}^0 e^{nu t} l_m(t) dt for the Lagrange basis on nodes t[0..k)
  auto rule = [&](const double* t, int k, int m, double nu) {
    double sum = 0.0;
    for (int g = 0; g < kG; ++g) {
      const double tt = 0.5 * (gx[g] - 1.0);
      double ell = 1.0;
      for (int r = 0; r < k; ++r)
        if (r != m) ell *= (tt - t[r]) / (t[m] - t[r]);
      sum += 0.5 * gw[g] * nu * std::exp(nu * tt) * ell;
    }
    return sum;
  };
  for (int i = 0; i < n; ++i) {
    const double xi = x[size_t(i)];
    for (int side = 0; side < 2; ++side) {
      const double dx = side == 0 ? xi - node(i - 1) : node(i + 1) - xi;
      const double nu = alpha * dx;
      double t5[5];
      for (int k = 0; k < 5; ++k) {
        const int off = k - 3;
        t5[k] = side == 0 ? (node(i + off) - xi) / dx : (xi - node(i - off)) / dx;
      }
      std::vector<double>& w = side == 0 ? *wR : *wL;
      auto at = [&](int slot) -> double& { return w[size_t(slot) * n + i]; };
      for (int r = 0; r < 3; ++r) {
        const double* t = t5 + r;
        for (int j = 0; j < 3; ++j) {
          const double ta = t[(j + 1) % 3], tb = t[(j + 2) % 3];
          const double den = (t[j] - ta) * (t[j] - tb);
          at(3 * r + j) = rule(t, 3, j, nu);
          at(12 + 3 * r + j) = -(ta + tb) / den;
          at(21 + 3 * r + j) = 2.0 / den;
        }
      }
      const double d0 = rule(t5, 5, 0, nu) / at(0);
      const double d2 = rule(t5, 5, 4, nu) / at(8);
      at(9) = d0;
      at(10) = 1.0 - d0 - d2;
      at(11) = d2;
    }
  }
  if (!(L > 0)) {
    // Dirichlet ends: J_R(x_0) = J_L(x_N) = 0 (zero rules, equal weights)
    for (int side = 0; side < 2; ++side) {
      std::vector<double>& w = side == 0 ? *wR : *wL;
      const size_t i = side == 0 ? 0 : size_t(n - 1);
      for (int slot = 0; slot < kNuWeno; ++slot) w[size_t(slot) * n + i] = 0.0;
      for (int r = 0; r < 3; ++r) w[size_t(9 + r) * n + i] = 1.0 / 3.0;
    }
  }
}

// Slots of the device tables: decays qR, qL, then per direction the forcing's
// filter.  Linear rule: b_m, m = -2..2, K_R(x_i) = sum_m b_m d_{i+m}, K_L(x_i)
// = -sum_m b_m d_{i+1-m} (d_i = v_i - v_{i-1}).  WENO-Z: per direction 21
// values, in the differences e0 = v_i - v_{i-1}, e1, e2 (further back), f =
// v_{i+1} - v_i (mirrored for L): the substencil rules K_0 = e0 + k0 e1 + k1
// e2, K_1 = k2 e0 + k3 e1, K_2 = k4 e0 + k5 f (sum_j c^{(r)}_j = 1 - q makes
// K_r = v_i - q v_{i-1} - J^{(r)} a filter of the differences), d_r, and per r
// the two weights each of a = p_t(0) and b = p_tt on the substencil's two
// differences (their rows sum to zero).
constexpr int kNuLinSlots = 5, kNuWenoSlots = 21;
constexpr int kNuMaxWarps = 16;
inline int nu_slots(bool weno) { return 2 + 2 * (weno ? kNuWenoSlots : kNuLinSlots); }

// Points per lane: the fewest that let 16 warps cover the line (FP32 from 8
// on: two lines share a CTA's table reads).
inline int nu_points_per_lane(int n, bool f64) {
  if (f64 && n <= 4 * 32 * kNuMaxWarps) return 4;
  return n <= 8 * 32 * kNuMaxWarps ? 8 : 16;
}

// Index of slot s of point e (lane e / E of the line) in the device tables:
// groups of V points (nu_group), those of a line's lanes side by side, so that a
// warp's reads are contiguous.
inline size_t nu_index(int s, int e, int E, int V, int lanes) {
  const int lane = e / E, k = e % E;
  return (size_t(s) * (E / V) + k / V) * lanes * V + size_t(lane) * V + k % V;
}

// Device tables from the point rules (linear: cR, cL of
// build_nonuniform_tables; WENO-Z: wR, wL of build_nonuniform_weno_tables),
// padded with pass-through points (decay 1, no forcing).  Dirichlet lines
// (L == 0): the scans' start nodes have decay 1, so the start value passes on
// unchanged (the kernel sets no forcing there).
inline std::vector<double> pack_nonuniform(const std::vector<double>& cR, const std::vector<double>& cL,
                                           const std::vector<double>& q, bool weno, bool dirichlet, int E, int V,
                                           int nw) {
  const int n = int(q.size()), lanes = 32 * nw, cap = lanes * E, ns = nu_slots(weno);
  std::vector<double> t(size_t(ns) * cap, 0.0);
  auto put = [&](int s, int i, double v) { t[nu_index(s, i, E, V, lanes)] = v; };
  for (int i = 0; i < cap; ++i) {
    put(0, i, 1.0);
    put(1, i, 1.0);
  }
  for (int i = 0; i < n; ++i) {
    const double qr = q[size_t(i)], ql = q[size_t(i + 1 < n ? i + 1 : 0)];
    put(0, i, dirichlet && i == 0 ? 1.0 : qr);
    put(1, i, dirichlet && i == n - 1 ? 1.0 : ql);
    for (int side = 0; side < 2; ++side) {
      const std::vector<double>& c = side == 0 ? cR : cL;
      const double qd = side == 0 ? qr : ql;
      auto at = [&](int slot) { return c[size_t(slot) * n + i]; };
      if (!weno) {
        const int s0 = 2 + side * kNuLinSlots;
        put(s0 + 0, i, at(0));
        put(s0 + 1, i, at(0) + at(1));
        put(s0 + 2, i, at(0) + at(1) + at(2) + qd);
        put(s0 + 3, i, -(at(4) + at(5)));
        put(s0 + 4, i, -at(5));
      } else {
        const int s0 = 2 + side * kNuWenoSlots;
        put(s0 + 0, i, at(0) + at(1));
        put(s0 + 1, i, at(0));
        put(s0 + 2, i, 1.0 - at(5));
        put(s0 + 3, i, at(3));
        put(s0 + 4, i, at(6) + qd);
        put(s0 + 5, i, -at(8));
        for (int r = 0; r < 3; ++r) {
          put(s0 + 6 + r, i, at(9 + r));
          put(s0 + 9 + 4 * r, i, -at(12 + 3 * r));
          put(s0 + 10 + 4 * r, i, at(14 + 3 * r));
          put(s0 + 11 + 4 * r, i, -at(21 + 3 * r));
          put(s0 + 12 + 4 * r, i, at(23 + 3 * r));
        }
      }
    }
  }
  return t;
}

// One group of V values of a table.  ORDERED loads are volatile: left free,
// the compiler gathers a whole chunk's WENO-Z tables ahead of the arithmetic
// and spills them (2 KB a thread); the linear rule's it may move.
template <typename T, int V> struct NuVec { T v[V]; };
#define MOLT_NU_LOAD(TYPE, V, TEXT, ...)                                          \
  template <bool ORDERED>                                                          \
  __device__ __forceinline__ void nu_load(NuVec<TYPE, V>& x, const TYPE* p) {      \
    if constexpr (ORDERED) asm volatile(TEXT : __VA_ARGS__ : "l"(p));              \
    else asm(TEXT : __VA_ARGS__ : "l"(p));                                         \
  }
MOLT_NU_LOAD(float, 4, "ld.global.nc.v4.f32 {%0,%1,%2,%3}, [%4];", "=f"(x.v[0]), "=f"(x.v[1]), "=f"(x.v[2]), "=f"(x.v[3]))
MOLT_NU_LOAD(float, 2, "ld.global.nc.v2.f32 {%0,%1}, [%2];", "=f"(x.v[0]), "=f"(x.v[1]))
MOLT_NU_LOAD(double, 2, "ld.global.nc.v2.f64 {%0,%1}, [%2];", "=d"(x.v[0]), "=d"(x.v[1]))
MOLT_NU_LOAD(double, 1, "ld.global.nc.f64 %0, [%1];", "=d"(x.v[0]))
#undef MOLT_NU_LOAD
// Values per group: 16 bytes, with WENO-Z weights (44 values a point) 8.
template <typename T, bool WENO>
__host__ __device__ constexpr int nu_group() { return (WENO ? 8 : 16) / int(sizeof(T)); }

// WENO-Z forcing from the point's 21 table values w (kNuWenoSlots) and its
// differences in the orientation of the direction: beta_r = a^2 - a b +
// 4/3 b^2, w~_r = d_r (1 + tau/(eps + beta_r)), tau = |beta_0 - beta_2|,
// eps = 1e-6 (Sec. 2.4).  The mean of the K_r is K_1 plus the weighted
// differences from it: three roundings of the result's size, where the
// weighted sum took six (FP32, 10% noise: one application of D_R errs by
// 6.7e-8 of the result against 1.04e-7, of D_0 by 6.0e-8 against 8.7e-8).
template <typename T>
__device__ __forceinline__ T nu_wenoz_defect(const T (&w)[kNuWenoSlots], T e0, T e1, T e2, T f) {
  const T K[3] = {fma(w[0], e1, w[1] * e2) + e0, fma(w[2], e0, w[3] * e1), fma(w[4], e0, w[5] * f)};
  const T lo[3] = {e2, e1, e0}, hi[3] = {e1, e0, f};
  T beta[3];
#pragma unroll
  for (int r = 0; r < 3; ++r) {
    const T a = fma(w[9 + 4 * r], lo[r], w[10 + 4 * r] * hi[r]);
    const T b = fma(w[11 + 4 * r], lo[r], w[12 + 4 * r] * hi[r]);
    beta[r] = fma(a, a - b, T(4.0 / 3.0) * b * b);
  }
  const T tau = fabs(beta[0] - beta[2]);
  const T eps = T(1e-6);
  T wt[3];
#pragma unroll
  for (int r = 0; r < 3; ++r) wt[r] = fma(w[6 + r] * tau, weight_rcp(eps + beta[r]), w[6 + r]);
  const T mix = fma(wt[2], K[2] - K[1], wt[0] * (K[0] - K[1]));
  return fma(mix, weight_rcp(wt[0] + wt[1] + wt[2]), K[1]);
}

// S_P along non-uniform lines, periodic or Dirichlet, G lines per CTA of `nw`
// warps: lane tl owns points E tl .. E tl + E - 1 of every line, staged in
// the padded layout of csrc/sweep.cuh.  W_R = v - L_R^{-1}[v] and W_L obey
// the recurrences of I with forcings K that are filters of the differences
// (no value of the size of v is subtracted from another; D of a constant is
// zero).  The decays' products -- inside the lane, over the lanes of a warp,
// over the warps of a line -- depend on the tables alone and are formed once
// per CTA; an application of D then scans one value per lane and direction.
// Boundary constants (Sec. 2.3, the 2x2 algebra of Sec. 3.3): line_constant.
// Bound by instructions and by the table reads, 12 values a point (WENO-Z 44)
// per application and CTA, from L2: G lines share them.
template <typename T, typename TIO, bool WENO, int E, int G>
__global__ void __launch_bounds__(512) nonuniform_kernel(const NuArgs a) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  constexpr unsigned FULL = 0xffffffffu;
  constexpr int V = nu_group<T, WENO>(), NS = WENO ? kNuWenoSlots : kNuLinSlots;
  const int n = a.g.n, nw = a.nw, LS = a.LS;
  const int lane = threadIdx.x & 31, part = threadIdx.x >> 5, tl = threadIdx.x;
  const int e0 = tl * E;
  T* totals = reinterpret_cast<T*>(smem_raw);        // [G + 1][nw][2]; the last row: the warps' decays
  T* lines = totals + (G + 1) * kNuMaxWarps * 2;
  const T* tab = static_cast<const T*>(a.tab);
  const int tstride = 32 * nw * V;                    // elements of one group of all lanes
  const long long line0 = (long long)blockIdx.x * G;
  const TIO* in = static_cast<const TIO*>(a.in);
  TIO* out = static_cast<TIO*>(a.out);
  const bool dir = a.bc == 1;
  long long base[G];
#pragma unroll
  for (int g = 0; g < G; ++g) {
    base[g] = line_base(a.g, line0 + g < a.g.nlines ? line0 + g : a.g.nlines - 1);
    T* v = lines + g * LS;
#pragma unroll 4
    for (int i = threadIdx.x; i < n; i += blockDim.x) v[phys<E>(i)] = T(in[base[g] + i * a.g.stride]);
  }
  // decays and their products
  T qR[E], qL[E];
  auto load_q = [&](int slot, T (&q)[E]) {
#pragma unroll
    for (int j = 0; j < E / V; ++j) {
      NuVec<T, V> x;
      nu_load<WENO>(x, tab + (size_t(slot) * (E / V) + j) * tstride + tl * V);
#pragma unroll
      for (int k = 0; k < V; ++k) q[j * V + k] = x.v[k];
    }
  };
  load_q(0, qR);
  load_q(1, qL);
  T mR[5], mL[5], pwR, pwL;     // multipliers of the warp scan's steps; decay inside the warp before the lane
  T mX[4], qwR, qwL;            // the same over the warps of the line
  {
    T pr = T(1), pl = T(1);
#pragma unroll
    for (int k = 0; k < E; ++k) {
      pr *= qR[k];
      pl *= qL[k];
    }
#pragma unroll
    for (int k = 0; k < 5; ++k) {
      const int o = 1 << k;
      mR[k] = pr;
      mL[k] = pl;
      const T xr = shfl_up(pr, o), xl = shfl_down(pl, o);
      if (lane >= o) pr *= xr;
      if (lane + o < 32) pl *= xl;
    }
    pwR = shfl_up(pr, 1);
    pwL = shfl_down(pl, 1);
    if (lane == 0) pwR = T(1);
    if (lane == 31) pwL = T(1);
    T* wd = totals + G * kNuMaxWarps * 2;
    if (lane == 31) wd[2 * part] = pr;
    if (lane == 0) wd[2 * part + 1] = pl;
    __syncthreads();
    const int j = lane & 15;
    T x = T(1);
    if (j < nw) x = lane >= 16 ? wd[2 * (nw - 1 - j) + 1] : wd[2 * j];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      mX[k] = x;
      const T xp = __shfl_up_sync(FULL, x, 1 << k, 16);
      if (j >= (1 << k)) x *= xp;
    }
    T ex = __shfl_up_sync(FULL, x, 1, 16);
    if (j == 0) ex = T(1);
    qwR = __shfl_sync(FULL, ex, part);
    qwL = __shfl_sync(FULL, ex, 15 + nw - part);
  }
  T S[G][E];
  for (int p = 0; p < a.P; ++p) {
    // ghosts (periodic images, or odd reflection about the end values)
    if (threadIdx.x < 6 * G) {
      const int g = threadIdx.x / 6, k = threadIdx.x - 6 * g;
      T* v = lines + g * LS;
      if (k < 3) {
        const int j = k + 1;
        v[phys<E>(-j)] = dir ? T(2) * v[phys<E>(0)] - v[phys<E>(j)] : v[phys<E>(((n - j) % n + n) % n)];
      } else {
        const int j = k - 2;
        v[phys<E>(n - 1 + j)] =
            dir ? T(2) * v[phys<E>(n - 1)] - v[phys<E>(n - 1 - j)] : v[phys<E>((j - 1) % n)];
      }
    }
    __syncthreads();
    // differences of the lane's window: dd[j] = v_{e0-2+j} - v_{e0-3+j}
    T dd[G][E + 5];
#pragma unroll
    for (int g = 0; g < G; ++g) {
      const T* c = lines + g * LS + (E + 1) * tl;
      T w[E + 6];
#pragma unroll
      for (int j = 0; j < E + 6; ++j) w[j] = c[chunk_off<E>(j - 3)];
#pragma unroll
      for (int j = 0; j < E + 5; ++j) dd[g][j] = w[j + 1] - w[j];
    }
    // forcings
    T KR[G][E], KL[G][E];
#pragma unroll
    for (int j = 0; j < E / V; ++j) {
#pragma unroll
      for (int side = 0; side < 2; ++side) {
        NuVec<T, V> t[NS];
#pragma unroll
        for (int s = 0; s < NS; ++s)
          nu_load<WENO>(t[s], tab + (size_t(2 + side * NS + s) * (E / V) + j) * tstride + tl * V);
#pragma unroll
        for (int kk = 0; kk < V; ++kk) {
          const int k = j * V + kk;
#pragma unroll
          for (int g = 0; g < G; ++g) {
            const T* d = dd[g];
            T K;
            if constexpr (WENO) {
              T w[NS];
#pragma unroll
              for (int s = 0; s < NS; ++s) w[s] = t[s].v[kk];
              K = side == 0 ? nu_wenoz_defect<T>(w, d[k + 2], d[k + 1], d[k], d[k + 3])
                            : nu_wenoz_defect<T>(w, -d[k + 3], -d[k + 4], -d[k + 5], -d[k + 2]);
            } else {
              K = T(0);
#pragma unroll
              for (int j = 0; j < 5; ++j) {
                const int s = j < 2 ? j : (j < 4 ? j + 1 : 2);   // the large tap last: one rounding at its size
                K = fma(t[s].v[kk], side == 0 ? d[k + s] : -d[k + 5 - s], K);
              }
            }
            // points past the end, and Dirichlet nodes where a scan starts
            const int e = e0 + k;
            if (e >= n || (dir && e == (side == 0 ? 0 : n - 1))) K = T(0);
            (side == 0 ? KR : KL)[g][k] = K;
          }
        }
      }
    }
    // scans from zero
    T bR[G], bL[G], cR[G], cL[G];
#pragma unroll
    for (int g = 0; g < G; ++g) {
      bR[g] = bL[g] = T(0);
#pragma unroll
      for (int k = 0; k < E; ++k) {
        bR[g] = fma(qR[k], bR[g], KR[g][k]);
        bL[g] = fma(qL[E - 1 - k], bL[g], KL[g][E - 1 - k]);
      }
#pragma unroll
      for (int k = 0; k < 5; ++k) {
        const int o = 1 << k;
        const T xr = shfl_up(bR[g], o), xl = shfl_down(bL[g], o);
        const T nr = fma(mR[k], xr, bR[g]), nl = fma(mL[k], xl, bL[g]);
        bR[g] = lane >= o ? nr : bR[g];
        bL[g] = lane + o < 32 ? nl : bL[g];
      }
      cR[g] = shfl_up(bR[g], 1);
      cL[g] = shfl_down(bL[g], 1);
      if (lane == 0) cR[g] = T(0);
      if (lane == 31) cL[g] = T(0);
      T* tot = totals + g * kNuMaxWarps * 2;
      if (lane == 31) tot[2 * part] = bR[g];
      if (lane == 0) tot[2 * part + 1] = bL[g];
    }
    __syncthreads();
#pragma unroll
    for (int g = 0; g < G; ++g) {
      const T* tot = totals + g * kNuMaxWarps * 2;
      const int j = lane & 15;
      T x = T(0);
      if (j < nw) x = lane >= 16 ? tot[2 * (nw - 1 - j) + 1] : tot[2 * j];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        if ((1 << k) < nw) {
          const T xp = __shfl_up_sync(FULL, x, 1 << k, 16);
          const T nx = fma(mX[k], xp, x);
          x = j >= (1 << k) ? nx : x;
        }
      }
      T ex = __shfl_up_sync(FULL, x, 1, 16);
      if (j == 0) ex = T(0);
      T inR = __shfl_sync(FULL, ex, part), inL = __shfl_sync(FULL, ex, 15 + nw - part);
      if (a.close) {
        const T tR = __shfl_sync(FULL, x, nw - 1), tL = __shfl_sync(FULL, x, 15 + nw);
        inR = fma(qwR, line_constant<T>(a, tR, tL), inR);
        inL = fma(qwL, line_constant<T>(a, tL, tR), inL);
      }
      T yR = fma(pwR, inR, cR[g]), yL = fma(pwL, inL, cL[g]);
#pragma unroll
      for (int k = 0; k < E; ++k) {
        yR = fma(qR[k], yR, KR[g][k]);
        KR[g][k] = yR;
        yL = fma(qL[E - 1 - k], yL, KL[g][E - 1 - k]);
        KL[g][E - 1 - k] = yL;
      }
      T* c = lines + g * LS + (E + 1) * tl;
#pragma unroll
      for (int k = 0; k < E; ++k) {
        const T D = a.mode == MODE_0 ? T(0.5) * (KR[g][k] + KL[g][k]) : (a.mode == MODE_R ? KR[g][k] : KL[g][k]);
        S[g][k] = p == 0 ? D : S[g][k] + D;
        // (every lane read its window before the totals' barrier)
        if (e0 + k < n) c[chunk_off<E>(k)] = p + 1 < a.P ? D : S[g][k];
      }
    }
    __syncthreads();
  }
#pragma unroll
  for (int g = 0; g < G; ++g) {
    if (line0 + g >= a.g.nlines) break;
    const T* v = lines + g * LS;
#pragma unroll 4
    for (int i = threadIdx.x; i < n; i += blockDim.x) out[base[g] + i * a.g.stride] = TIO(v[phys<E>(i)]);
  }
}

}  // namespace molt
