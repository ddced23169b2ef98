// Line-sweep kernel: the O(N) fast summation of L^{-1} and the successive-
// convolution partial sums S_P = sum_{p=1}^P D^p along one axis of a grid
// (arXiv 2007.03041, Sec. 2.1-2.4), with a fused epilogue that consumes S_P
// (store, accumulate, or the time-integrator update).
//
// Mapping.  A CTA owns W lines of one axis.  The lines are staged in shared
// memory (converted to the compute type T) with ghost cells on both ends;
// each line is processed by `nwl` warps and every lane owns E consecutive
// points of it in registers.  Per application of D:
//   1. forcings of the recurrences from a register window of the lane's points
//      plus 3 neighbours per side, as filters of the differences d_i = v_i -
//      v_{i-1} (Sec. 2.4 / App. C; linear, WENO-Z or learned weights);
//   2. the recurrences of v - L_R^{-1}[v] and v - L_L^{-1}[v] as scans: a serial
//      fold per lane, a shuffle scan across the warp, a scan of the warps'
//      totals (the exact block split of the convolution sums, Sec. 3, without
//      any truncation);
//   3. the boundary constants from the line totals (Sec. 2.3: periodic
//      C = T/(1-mu); Dirichlet: the 2x2 system with determinant 1-mu^2,
//      Sec. 3.3), folded into the scans as their initial values;
//   4. the scans again from their carries, which give D.
// D is written back to shared memory for the next power.  The epilogue runs
// in the coalesced load mapping.  compute_lines() has the algebra.
//
// Precision plumbing.  GB300 executes FP64 arithmetic and FP64<->FP32
// conversions at a small fraction of the FP32 rate (two FP64 FMAs per clock
// and SM, 64 cycles of a scheduler's pipe per warp instruction), so FP32
// sweeps keep FP64 to the update itself: they read an FP32 copy of the state
// (written by the previous update), conversions are done with integer bit
// operations, and only the state update uses FP64 fused multiply-adds.  FP64
// sweeps are bound by that pipe: their form is the one with the fewest
// operations a point.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "mlp.cuh"

namespace molt {

constexpr int kE = 16;   // points per lane
constexpr int kG = 16;   // ghost slots per side in shared memory (3 used)
#ifndef MOLT_MAX_THREADS
#define MOLT_MAX_THREADS 512
#endif
constexpr int kMaxThreads = MOLT_MAX_THREADS;
static_assert(kMaxThreads <= 512,
              "16 warps a line at most: their totals are scanned by half a warp, q^(points before a warp) has four bits, "
              "and lines of several warps have at most eight barriers");
// Shared memory per CTA (the GPU allows 227 KB): a sweep tile's budget, and the
// dynamic size the sweep kernels opt into (a TMA tile plus its staging buffer
// must fit it).
constexpr size_t kSmemTileBudget = 200 * 1024;
constexpr size_t kSmemOptIn = 210 * 1024;

enum Epi {
  EPI_STORE = 0,       // out = S
  EPI_ACC_SET = 1,     // acc = S
  EPI_ACC_ADD = 2,     // acc += S
  EPI_HEAT_FINAL = 3,  // dst = a0*un + a1*(us + coefS*(acc + S))
  EPI_WAVE_FINAL = 4,  // dst = 2u - uprev + coefS*(acc+S)  (or from rest)
  EPI_HJ_X = 5,        // hx = H^_x(D_R, D_L); speed max
  EPI_HJ_Y = 6,        // u -= dt*H^; speed max
  EPI_HJ_XG = 7,       // EPI_HJ_X for every Hamiltonian (HamKind)
  EPI_HJ_YG = 8,       // EPI_HJ_Y for every Hamiltonian, a source F(x, t), speed-only passes
  EPI_ACC_AXPY = 9,    // acc += coefS * S (advection-diffusion terms)
  EPI_ADV_FINAL = 10   // dst = a0*un + a1*(us + (acc + S)) (advection-diffusion, fused axis kernel)
};
// The general Hamilton-Jacobi kernels (XG/YG) carry more operands per point;
// the |grad u|^2/2 kernels without a source keep their own instantiations.
__host__ __device__ constexpr bool epi_hj_x(int e) { return e == EPI_HJ_X || e == EPI_HJ_XG; }
__host__ __device__ constexpr bool epi_hj_y(int e) { return e == EPI_HJ_Y || e == EPI_HJ_YG; }
__host__ __device__ constexpr bool epi_hj_gen(int e) { return e == EPI_HJ_XG || e == EPI_HJ_YG; }
// Hamiltonian of the Hamilton-Jacobi step (values of molt_hamiltonian).
//   HALF_SQ:   H = |grad u|^2/2, separable: each pass adds its axis's part of
//              the local Lax-Friedrichs Hamiltonian
//   LINEAR:    H = sum_d a_d u_d, separable (upwind: H^_d = a_d v^-_d for
//              a_d > 0, a_d v^+_d for a_d < 0)
//   AFFINE_SQ: H = (h0 + sum_d a_d u_d)^2/2, not separable: the x pass leaves
//              sigma_x = a_x mean_x and delta_x = |a_x| (v^+_x - v^-_x)/2, the
//              last pass forms H^ from all axes
enum HamKind { HAM_HALF_SQ = 0, HAM_LINEAR = 1, HAM_AFFINE_SQ = 2 };
enum Mode { MODE_L = 0, MODE_R = 1, MODE_0 = 2, MODE_RL = 3 };
enum StatusBits { ST_NONFINITE = 1, ST_TIMEOUT = 2 };

struct LineGeom {
  int n;              // stored points per line
  long long nlines;   // lines in this pass
  long long nlo;      // line l = hi*nlo + lo
  long long s_lo, s_hi;
  long long stride;   // element stride along the line
};

// Constants of the scans along a line (csrc/line_constants.h); the FP32 copies
// are rounded on the host (converting on the device would use the FP64 pipe).
struct LineConst {
  int d0;             // JQ_D0: 1 residual form, 0 K filters
  int close;          // boundary constants: 0 none, 1 kA, 2 kA and kB
  double b[5];        // K_R taps on the differences d_{i-2} .. d_{i+2}
  double f0, f1, kap; // residual form of D_0 (K form: kap = 1/2)
  double wk[6];       // WENO-Z substencil rules in difference form
  double d[3];        // WENO linear weights
  double qp[13];      // q^(2^k), q = e^{-nu}
  double qlast, qlw;  // q^(valid points of the last lane / of the last warp)
  double kA, kB;      // boundary constants C = kA T_same + kB T_other
  float bf[5], f0f, f1f, kapf, wkf[6], df[3], qpf[13], qlastf, qlwf;
  float kAh, kAl, kBh, kBl;   // kA, kB as FP32 pairs
};

struct SweepArgs : LineConst {
  LineGeom g;
  int W, nwl, LS;     // lines per CTA, warps per line, shared line stride (elements)
  int E;              // points per lane of the plain kernel (16, 8 or 4; others mean 16)
  int bc;             // 0 periodic, 1 Dirichlet
  int mode;           // Mode
  int P;
  int contiguous;     // stride == 1
  double alpha;
  float alphaf;
  // epilogue operands
  const void* in;     // sweep input (TIN)
  void* out;          // EPI_STORE destination / HJ: H^_x buffer (state type)
  void* acc;          // accumulator (compute type)
  const void* un;     // heat: u^n; wave: u^n; HJ: u (state type)
  const void* us;     // heat: stage state; wave: u^{n-1}
  void* dst;          // final destination (state type)
  void* dst2;         // wave: receives u^n (old state) when non-null
  float* shadow;      // FP32 copy of dst written by final epilogues (or null)
  double a0, a1, coefS;
  int from_rest;      // wave Taylor start
  // Hamilton-Jacobi
  const unsigned long long* lag;  // lagged speed (double bits)
  unsigned long long* speed;      // this pass's speed slot (double bits)
  // adaptive step (Eq. "adaptive time rule"): dt = cfl min_d h_d / c_d =
  // cfl / max_d (c_d / h_d); the passes publish c_d / h_d
  double cfl, dt_max, inv_h;   // inv_h = 1 / h of this pass's axis
  double* t_dev;            // time accumulator (HJ_Y, block 0)
  int ham;                  // HamKind
  int two_out;              // MODE_RL with AFFINE_SQ: a second line buffer (delta)
  double vel, h0, vmax;     // a_d of this axis, h0, max_d |a_d| / h_d
  float velf;
  void* out2;               // AFFINE_SQ: delta_x (state type; written by the x pass, read by the last)
  const void* src;          // source coefficients F_k, k = 0..src_deg (state type) or null
  int src_deg;
  long long src_stride;     // elements between F_k and F_{k+1}
  const double* t_now;      // time of the state being advanced (read with a source)
  int* status;
  // learned weights (JQ_LEARNED kernels)
  const MlpBlob* mlp;               // BF16 network
  unsigned long long* mlp_stats;    // [stencils evaluated, WENO-Z fallbacks]
};

// Kind of a sweep kernel (template parameter JQ): the local quadrature, and
// whether both scans run (LINEAR, WENOZ, LEARNED: D_R and D_L, or their mean),
// D_0 with linear weights (D0), or one side alone (LINEAR1, WENOZ1).
enum JQuad { JQ_LINEAR = 0, JQ_WENOZ = 1, JQ_LEARNED = 2, JQ_D0 = 3, JQ_LINEAR1 = 4, JQ_WENOZ1 = 5 };

// Registers per thread of the scan kernels: 128 (512 threads per SM), and
// fewer for the D_0 and one-sided linear sweeps, whose other warps cover what
// a spilled value costs.  FP64 (bound by the FP64 pipe: a second or third
// resident CTA keeps it busy while another loads or stores) 80: 5277^2
// diffusion, 2 steps, 128 / 80 / 64 registers 5.11 / 3.87 / 3.97 ms (the
// two-sided Hamilton-Jacobi sweeps of a 1759^2 FP64 run 2.05 / 2.29 / 2.36 ms).
// FP32 tiles of 8 and 4 points a lane 64 and 48: 201x151x101 wave, 5 steps,
// 128 and 128 / 80 and 64 / 64 and 48 registers 0.80 / 0.70 / 0.68 ms; of 16
// points 128 (96 and 80 measured the same).
template <typename T, int JQ, int E = kE>
__host__ __device__ constexpr int sweep_regs() {
  if (JQ != JQ_D0 && JQ != JQ_LINEAR1) return 128;
  return sizeof(T) == 8 ? 80 : (E == 4 ? 48 : (E == 8 ? 64 : 128));
}

// Shared-memory index of point e of a line whose lanes own E points each: one
// pad word after every E words (kG is a multiple of E), so lane chunks start
// (E+1) words apart -- an odd stride, hence bank-conflict free.
template <int E>
__host__ __device__ constexpr int log2i() { return E == 16 ? 4 : (E == 8 ? 3 : (E == 4 ? 2 : -1)); }

template <int E = kE>
__host__ __device__ constexpr int phys(int e) {
  static_assert(log2i<E>() > 0, "points per lane must be 4, 8 or 16");
  return (e + kG) + ((e + kG) >> log2i<E>());
}

// For a lane chunk starting at e0 = E*t: phys(e0 + j) = (E+1)*t +
// chunk_off<E>(j), a compile-time constant for unrolled j.
template <int E = kE>
__host__ __device__ constexpr int chunk_off(int j) { return (j + kG) + ((j + kG) >> log2i<E>()); }

// Base offset of line l (32-bit division: the host keeps nlines < 2^31; a
// 64-bit division would run on the FP64 pipe).
__device__ __forceinline__ long long line_base(const LineGeom& g, long long l) {
  const unsigned int lu = unsigned(l), nlo = unsigned(g.nlo);
  const unsigned int hi = lu / nlo, lo = lu - hi * nlo;
  return (long long)hi * g.s_hi + (long long)lo * g.s_lo;
}

// ------------------------------------------------------------ conversions
// The hardware conversions between FP32 and FP64 run on the FP64 pipe, which
// is narrow on this part; the common operands are converted by integer
// operations on the bit patterns instead.  The rare operands leave through a
// call to the hardware conversion (a plain branch to it would be if-converted,
// executing it for every operand).  A translation unit whose kernels have no
// registers to spare for a call defines MOLT_CONV_SELECT 1: the rare operands
// then take integer operations in place too (same results; measured: the
// batched heat step 6.8 ms with calls against 5.1; the 512^3 wave step 1.77 ms
// with calls against 1.85 in place).
#ifndef MOLT_CONV_SELECT
#define MOLT_CONV_SELECT 0
#endif
static __device__ __noinline__ float d2f_rare(double x) { return __double2float_rn(x); }
static __device__ __noinline__ double f2d_rare(float x) { return double(x); }

// The rare operands by integer operations: subnormal results (the 24-bit
// significand moves right by 1..24 bits), overflow, infinities, NaN.
__device__ __forceinline__ float d2f_slow(double x) {
  const unsigned int hi = __double2hiint(x), lo = __double2loint(x);
  const unsigned int sign = hi & 0x80000000u, e11 = (hi >> 20) & 0x7FFu;
  if (e11 > 1150u) {
    const bool nan = e11 == 0x7FFu && ((hi & 0xFFFFFu) | lo) != 0u;
    return __uint_as_float(sign | (nan ? 0x7FFFFFFFu : 0x7F800000u));
  }
  const unsigned int sh = 897u - e11, full = ((hi & 0xFFFFFu) << 3) | (lo >> 29) | 0x800000u;
  const unsigned int out = full & ((1u << sh) - 1u), mant = full >> sh;
  const unsigned int half = 1u << (sh - 1u), below = (out & (half - 1u)) | (lo & 0x1FFFFFFFu);
  const unsigned int up = (out & half) && (below || (mant & 1u));
  return __uint_as_float(sign | (mant + up));
}
__device__ __forceinline__ double f2d_slow(float x) {
  unsigned int u = __float_as_uint(x), off = 1792u;
  if (((u >> 23) & 0xFFu) == 255u) {
    if (u & 0x7FFFFFu) u |= 0x400000u;              // infinities, NaN
  } else {
    u = __float_as_uint(x * 4294967296.f);          // 2^32 x is normal
    off = 864u;
  }
  const unsigned int hi = (u & 0x80000000u) | ((((u >> 23) & 0xFFu) + off) << 20) | ((u & 0x7FFFFFu) >> 3);
  return __hiloint2double(int(hi), int(u << 29));
}

// double -> float, round to nearest even: normal results by integer
// operations; results that round to zero (|x| < 2^-150) give the signed
// zero; subnormal results, overflow, inf and NaN take the hardware conversion.
__device__ __forceinline__ float d2f(double x) {
  const unsigned int hi = __double2hiint(x);
  const unsigned int lo = __double2loint(x);
  const unsigned int e11 = (hi >> 20) & 0x7FFu;
  if (e11 < 897u || e11 > 1150u) {
    if (e11 < 873u) return __uint_as_float(hi & 0x80000000u);
    if constexpr (MOLT_CONV_SELECT) return d2f_slow(x);
    else return d2f_rare(x);
  }
  const unsigned int mant = ((hi & 0xFFFFFu) << 3) | (lo >> 29);
  const unsigned int rest = lo & 0x1FFFFFFFu;           // 29 dropped bits
  const unsigned int half = 0x10000000u;
  const unsigned int up = (rest > half) | ((rest == half) & (mant & 1u));
  const unsigned int bits = (hi & 0x80000000u) | (((e11 - 896u) << 23) + mant + up);
  return __uint_as_float(bits);
}

// float -> double (exact): normal numbers and zeros by integer operations;
// subnormals, inf and NaN take the hardware conversion.
__device__ __forceinline__ double f2d(float x) {
  const unsigned int u = __float_as_uint(x);
  const unsigned int e8 = (u >> 23) & 0xFFu;
  if (e8 == 0u || e8 == 255u) {
    if ((u << 1) == 0u) return __hiloint2double(int(u & 0x80000000u), 0);
    if constexpr (MOLT_CONV_SELECT) return f2d_slow(x);
    else return f2d_rare(x);
  }
  const unsigned int hi = (u & 0x80000000u) | ((e8 + 896u) << 20) | ((u & 0x7FFFFFu) >> 3);
  const unsigned int lo = u << 29;
  return __hiloint2double(int(hi), int(lo));
}

template <typename T>
__device__ __forceinline__ T pick(double d, float f) {
  if constexpr (sizeof(T) == 4) return f; else return d;
}

// Non-finite test on the exponent bits (no floating-point instruction).
__device__ __forceinline__ bool nonfinite(double x) { return (__double2hiint(x) & 0x7FF00000) == 0x7FF00000; }
__device__ __forceinline__ bool nonfinite(float x) { return (__float_as_uint(x) & 0x7F800000u) == 0x7F800000u; }

// Global load; CG = true reads through L2 only (data written earlier in the
// same kernel by other CTAs must not come from a stale L1 line).
template <bool CG, typename V>
__device__ __forceinline__ V gload(const V* p) {
  if constexpr (CG) return __ldcg(p); else return *p;
}

template <typename TO, typename FROM>
__device__ __forceinline__ TO cvt(FROM x) {
  if constexpr (sizeof(TO) == 4 && sizeof(FROM) == 8) return d2f(x);
  else if constexpr (sizeof(TO) == 8 && sizeof(FROM) == 4) return f2d(x);
  else return TO(x);
}

template <typename T>
__device__ __forceinline__ T shfl_up(T v, int d) { return __shfl_up_sync(0xffffffffu, v, d); }
template <typename T>
__device__ __forceinline__ T shfl_down(T v, int d) { return __shfl_down_sync(0xffffffffu, v, d); }

// Reciprocal for the nonlinear weights: FP32 takes the hardware
// approximation (at most 1 ulp; the arguments eps + beta_r and sum_r w~_r are
// at least 1e-6 and about 1), FP64 the division.
__device__ __forceinline__ float weight_rcp(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ double weight_rcp(double x) { return 1.0 / x; }

// WENO-Z forcing K(x_i) = v_i - q v_{i-1} - J(x_i) in the orientation of J_R
// (J_L passes the mirrored differences): e0 = v_i - v_{i-1}, e1 = v_{i-1} -
// v_{i-2}, e2 = v_{i-2} - v_{i-3}, f = v_{i+1} - v_i.  Every substencil rule
// integrates the constant to 1 - q and the weights sum to one, so
// K = sum_r w_r K_r with K_r = q e0 + sum_j c^{(r)}_j (v_i - v_j) a filter of
// the differences (wk, csrc/line_constants.h; the e0 weight of K_0 is 1).
// WENO-Z (Sec. 2.4): w~_r = d_r (1 + tau/(eps+beta_r)), tau = |beta_0-beta_2|.
// The indicators arrive with eps added.
template <typename T>
__device__ __forceinline__ T wenoz_defect(T e0, T e1, T e2, T f, T b0, T b1, T b2, const T (&wk)[6], const T (&d)[3]) {
  const T K[3] = {fma(wk[1], e2, fma(wk[0], e1, e0)), fma(wk[3], e1, wk[2] * e0), fma(wk[5], f, wk[4] * e0)};
  const T b[3] = {b0, b1, b2};
  const T tau = fabs(b0 - b2);
  T wt[3], sum = T(0);
#pragma unroll
  for (int r = 0; r < 3; ++r) {
    wt[r] = fma(d[r] * tau, weight_rcp(b[r]), d[r]);   // d_r (1 + tau/(eps+beta_r))
    sum += wt[r];
  }
  return (wt[0] * K[0] + wt[1] * K[1] + wt[2] * K[2]) * weight_rcp(sum);
}

// Smoothness indicators: beta_r = int_{-1}^0 (p_r')^2 + (p_r'')^2 dt for the
// quadratic through the node triple (a, b, c) of substencil r; with s1 =
// (c - a)/2 and s2 = a - 2b + c, beta_r = s1^2 + k_r s1 s2 + m_r s2^2 (k = 3,
// 1, -1; m = 10/3, 4/3, 4/3).  A triple serves three points' J_R and,
// mirrored (s1 -> -s1), three points' J_L, with four different values: as
// substencil 0 of J_R, 0 of J_L, 1 of J_R (2 of J_L) and 2 of J_R (1 of J_L).
// They are formed once per triple, with eps = 1e-6 added, from its differences
// da = b - a, db = c - b (the compiler shares them among the points).
template <typename T>
struct Indicators {
  T outer, outer_mir, plus, minus;
  __device__ __forceinline__ Indicators(T da, T db) {
    const T s1 = T(0.5) * (da + db), s2 = db - da;
    const T p12 = s1 * s2, p22 = s2 * s2, p11 = fma(s1, s1, T(1e-6));
    const T A = fma(T(4.0 / 3.0), p22, p11), B = fma(T(10.0 / 3.0), p22, p11);
    outer = fma(T(3), p12, B);
    outer_mir = fma(T(-3), p12, B);
    plus = A + p12;
    minus = A - p12;
  }
};

// -------------------------------------------------------------- tile staging
// Barrier of the warps that share line lw of a tile.  A barrier number held in
// a register reserves all 16 barriers for the CTA, and an SM, with 64, then
// takes no more than four CTAs of any size: the y lines of a 512^2 FP32 wave,
// 512 CTAs of one warp, took 28.8 us a sweep, some SMs busy for 51 thousand
// cycles and some for 30.  The sweep kernels therefore take the CTA's own
// barrier (5 such steps 224 -> 191 us; 201 x 151 x 101 mixed wave, 5 steps, 685 ->
// 653 us; 4096^2 WENO-Z, 4 steps, 1293 -> 1277 us), FP64 tiles of 16 points a
// lane constant numbers 1 to 4, more than four lines of several warps sharing
// one with their neighbours (5277^2 diffusion, 2 steps, register / CTA / constant
// numbers 3890 / 3919 / 3824 us; the FP32 wave above 685 / 653 / 706 us).
// Translation units that measured faster with a barrier a line define
// MOLT_LINE_BARRIERS 1 and keep the register: the batched kernel (two CTAs of
// 512 threads per SM in any case; 10.4 ms against 11.1 with the CTA's barrier)
// and the advection-diffusion axis kernel (1500^2 FP32 WENO-Z, 2 steps, 194 us
// against 203).
#ifndef MOLT_LINE_BARRIERS
#define MOLT_LINE_BARRIERS 0
#endif
template <typename T, int E>
__device__ __forceinline__ void line_sync(int nwl, int lw) {
  if (nwl == 1) {
    __syncwarp();
  } else if constexpr (MOLT_LINE_BARRIERS) {
    asm volatile("bar.sync %0, %1;" ::"r"(1 + lw), "r"(32 * nwl) : "memory");
  } else if constexpr (sizeof(T) == 8 && E == 16) {
    const int share = blockDim.x > 128 * nwl ? 1 : 0, count = (32 * nwl) << share;
    switch (lw >> share) {
      case 0: asm volatile("bar.sync 1, %0;" ::"r"(count) : "memory"); break;
      case 1: asm volatile("bar.sync 2, %0;" ::"r"(count) : "memory"); break;
      case 2: asm volatile("bar.sync 3, %0;" ::"r"(count) : "memory"); break;
      default: asm volatile("bar.sync 4, %0;" ::"r"(count) : "memory"); break;
    }
  } else {
    __syncthreads();
  }
}

// Contiguous lines: the nwl warps of line lw read it with consecutive lanes.
// Strided lines: thread (p, w) with w fastest, so a warp reads whole rows of
// W neighbouring lines.
// put(shared destination, global source) moves one value.
template <typename T, typename TIN, int E, typename Put>
__device__ __forceinline__ void load_tile(const SweepArgs& a, const TIN* in, T* lines, long long line0, int lw, int tl,
                                          Put put) {
  const int W = a.W, n = a.g.n;
  if (a.contiguous) {
    const long long gl = line0 + lw;
    if (gl >= a.g.nlines) return;
    const TIN* src = in + line_base(a.g, gl);
    T* dstl = lines + lw * a.LS;
    const int step = a.nwl * 32;
#pragma unroll 4
    for (int p = tl; p < n; p += step) put(dstl + phys<E>(p), src + p);
  } else {
    // prow = blockDim/W is a multiple of 16, so phys<E>() advances by a constant
    const int w = threadIdx.x % W;
    const int prow = blockDim.x / W;
    const long long gl = line0 + w;
    if (gl >= a.g.nlines) return;
    const long long st = a.g.stride;
    int p = threadIdx.x / W;
    const TIN* src = in + line_base(a.g, gl) + p * st;
    const long long sstep = prow * st;
    T* dst = lines + w * a.LS + phys<E>(p);
    const int dstep = prow + prow / E;
#pragma unroll 8
    for (; p < n; p += prow) {
      put(dst, src);
      src += sstep;
      dst += dstep;
    }
  }
}

// ------------------------------------------------------------------- kernels
// T: compute type; TIN: sweep input element type; TST: state type of the
// epilogue operands.

struct TileSmem {
  void* totals;      // [W][nwl][2] of T: end values of the warps' scans from zero (R, L)
  void* lines;       // [W][LS] of T
  void* lines2;      // two_out: [W][LS] of T (delta of AFFINE_SQ)
  float* jloc;       // JQ_LEARNED: [W][2][LS] forcings K_R, K_L
  MlpNet* net;       // JQ_LEARNED: the network
  unsigned char* mlp_scratch;   // JQ_LEARNED: kMlpScratchBytes per warp
};

// Shared bytes of a tile beyond the lines for learned weights (the host
// planner adds the same amount).
__host__ __device__ constexpr size_t learned_extra_bytes(int W, int LS, int nwl) {
  return 32 + size_t(2) * W * LS * sizeof(float) + sizeof(MlpNet) + size_t(W) * nwl * kMlpScratchBytes;
}

// Shared bytes before the lines: the warps' totals.
__host__ __device__ constexpr size_t tile_head_bytes(int W, int nwl, size_t elem) {
  return (size_t(W) * nwl * 2 * elem + 15) & ~size_t(15);
}

template <typename T, int JQ = JQ_LINEAR>
__device__ __forceinline__ TileSmem carve(unsigned char* smem, const SweepArgs& a, size_t* used) {
  TileSmem t;
  t.totals = smem;
  const size_t off = tile_head_bytes(a.W, a.nwl, sizeof(T));
  t.lines = smem + off;
  *used = off + size_t(a.W) * a.LS * sizeof(T);
  t.lines2 = nullptr;
  if (a.two_out) {
    const size_t l2 = (*used + 15) & ~size_t(15);
    t.lines2 = smem + l2;
    *used = l2 + size_t(a.W) * a.LS * sizeof(T);
  }
  t.jloc = nullptr;
  t.net = nullptr;
  t.mlp_scratch = nullptr;
  if constexpr (JQ == JQ_LEARNED) {
    const size_t j0 = (*used + 15) & ~size_t(15);
    t.jloc = reinterpret_cast<float*>(smem + j0);
    const size_t n0 = j0 + size_t(2) * a.W * a.LS * sizeof(float);
    t.net = reinterpret_cast<MlpNet*>(smem + n0);
    const size_t c0 = (n0 + sizeof(MlpNet) + 15) & ~size_t(15);
    t.mlp_scratch = smem + c0;
    *used = c0 + size_t(a.W) * a.nwl * kMlpScratchBytes;
  }
  return t;
}

// ------------------------------------------------------------- line constants
template <typename T>
__device__ __forceinline__ T qpow_bit(const LineConst& a, int k) { return pick<T>(a.qp[k], a.qpf[k]); }

// q^e for 0 <= e < 2^COUNT, times 2^LO: the product of the stored powers
// q^(2^(LO + k)) over the bits of e.
template <typename T, int LO, int COUNT>
__device__ __forceinline__ T qpow(const LineConst& a, int e) {
  T r = T(1);
#pragma unroll
  for (int k = 0; k < COUNT; ++k)
    if ((e >> k) & 1) r *= qpow_bit<T>(a, LO + k);
  return r;
}

// Line boundary constants (Sec. 2.3, Sec. 3.3): the value C = kA T_same +
// kB T_other that enters the line before its first scan position, from the
// end values T of the scans started from zero.  FP64 sweeps compute it in
// FP64.  FP32 sweeps compute it in pairs of FP32 numbers (kA, kB as hi + lo;
// exact product errors by FMA, TwoSum for the addition: 48 bits, rounded once
// to the FP32 that enters the scan), so that every warp solves its own line:
// the FP64 pipe, two FMAs per clock and SM here, held a barrier of the whole
// CTA per application of D.
template <typename T, typename Args>
__device__ __forceinline__ T line_constant(const Args& a, T same, T other) {
  if constexpr (sizeof(T) == 8) {
    const T c = a.kA * same;
    return a.close == 2 ? fma(a.kB, other, c) : c;
  } else {
    T p = a.kAh * same;
    T e = fmaf(a.kAl, same, fmaf(a.kAh, same, -p));
    if (a.close == 2) {
      const T p2 = a.kBh * other;
      e += fmaf(a.kBl, other, fmaf(a.kBh, other, -p2));
      const T s = p + p2, bb = s - p;
      e += (p - (s - bb)) + (p2 - bb);
      p = s;
    }
    return p + e;
  }
}

// Ghost cells of one line by the lanes of the warp that owns it.
template <typename T, int E = kE>
__device__ __forceinline__ void warp_fill_ghosts(const SweepArgs& a, T* b, int lane) {
  const int n = a.g.n;
  if (lane < 3) {
    const int j = lane + 1;  // ghost e = -j
    T val;
    if (a.bc == 0) {
      int s = (-j) % n;
      if (s < 0) s += n;
      val = b[phys<E>(s)];
    } else {
      const int m = j < n - 1 ? j : n - 1;
      val = T(2) * b[phys<E>(0)] - b[phys<E>(m)];
    }
    b[phys<E>(-j)] = val;
  } else if (lane < 6) {
    const int j = lane - 2;  // ghost e = n-1+j
    T val;
    if (a.bc == 0) {
      val = b[phys<E>((n - 1 + j) % n)];
    } else {
      const int m = n - 1 - j > 0 ? n - 1 - j : 0;
      val = T(2) * b[phys<E>(n - 1)] - b[phys<E>(m)];
    }
    b[phys<E>(n - 1 + j)] = val;
  }
}

// Learned local integrals of the points a warp owns (32*E consecutive points
// of its line from `first`): 16 points at a time, lanes 0-15 take their J_R
// stencils (v_{e-3..e+1}), lanes 16-31 the J_L ones (mirrored: v_{e+3..e-1}),
// the warp evaluates the network on the tensor cores, and every lane finishes
// its stencil: WENO-Z fallback check, then K = v - q v_prev - sum_r w_r
// J^{(r)} into jr / jl (shared, line layout).
template <int E>
__device__ __forceinline__ void learned_local_integrals(const SweepArgs& a, const MlpNet& net, const float* buf,
                                                        float* jr, float* jl, unsigned char* scratch, int first,
                                                        int n, int lane) {
  MlpRegs R;
  mlp_load_regs(net, lane, R);
  float wk[6], d[3];
#pragma unroll
  for (int r = 0; r < 3; ++r) d[r] = a.df[r];
#pragma unroll
  for (int i = 0; i < 6; ++i) wk[i] = a.wkf[i];
  unsigned evaluated = 0, fallbacks = 0;
  const bool left = lane >= 16;
  float* jk = left ? jl : jr;
  for (int b = 0; b < 32 * E; b += 16) {
    if (first + b >= n) break;   // warp-uniform
    const int e = first + b + (lane & 15), ec = e < n ? e : n - 1;
    float v[5], p[3];
#pragma unroll
    for (int j = 0; j < 5; ++j) v[j] = buf[phys<E>(ec + (left ? 3 - j : j - 3))];
    mlp_eval32(R, scratch, lane, v, p);
    if (e < n) {
      float w[3];
      fallbacks += mlp_final_weights(v, p, d, w) ? 1u : 0u;
      ++evaluated;
      // K = sum_r w_r K_r in difference form (wenoz_defect)
      const float f0 = v[3] - v[2], f1 = v[2] - v[1], f2 = v[1] - v[0], f = v[4] - v[3];
      const float K0 = fmaf(wk[1], f2, fmaf(wk[0], f1, f0));
      const float K1 = fmaf(wk[3], f1, wk[2] * f0), K2 = fmaf(wk[5], f, wk[4] * f0);
      jk[phys<E>(e)] = fmaf(w[0], K0, fmaf(w[1], K1, w[2] * K2));
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    evaluated += __shfl_xor_sync(0xffffffffu, evaluated, o);
    fallbacks += __shfl_xor_sync(0xffffffffu, fallbacks, o);
  }
  if (lane == 0 && a.mlp_stats) {
    atomicAdd(a.mlp_stats, (unsigned long long)evaluated);
    if (fallbacks) atomicAdd(a.mlp_stats + 1, (unsigned long long)fallbacks);
  }
}

// Value of ghost point e (-3 <= e < 0 or n <= e < n + 3) of an exact-fit
// line (n >= 128): the periodic image, or the odd reflection about the end
// value (Sec. 2.3).
template <typename T, int E>
__device__ __forceinline__ T ghost_value(const T* b, int e, int n, int bc) {
  if (bc == 0) return b[phys<E>(e < 0 ? e + n : e - n)];
  if (e < 0) return T(2) * b[phys<E>(0)] - b[phys<E>(-e)];
  return T(2) * b[phys<E>(n - 1)] - b[phys<E>(2 * (n - 1) - e)];
}

// A lane's place in its line, for the scans below.
template <typename T, bool ONE, bool RAGGED, int E>
struct LineLane {
  T* totals;
  T* buf;              // the line
  T* cbase;            // the lane's chunk: phys<E>(e0 + j) = (E+1)*ch + chunk_off<E>(j)
  int n, nwl, lw, part, lane, e0, ch;
  bool mir;            // one-sided L scans run the line mirrored
  bool dir, own;
  bool end0, endN;     // the chunk holds a Dirichlet end node (x_0, x_{n-1})
  int lastR;           // the lane whose last point closes the R scan of its warp

  __device__ __forceinline__ LineLane(const SweepArgs& a, const TileSmem& sm) {
    static_assert(phys<E>(E * 3 + 2) == (E + 1) * 3 + chunk_off<E>(2), "lane base / chunk offset mismatch");
    nwl = a.nwl;
    n = a.g.n;
    totals = static_cast<T*>(sm.totals);
    const int warp = threadIdx.x >> 5;
    lane = threadIdx.x & 31;
    lw = warp / nwl;
    part = warp - lw * nwl;
    buf = static_cast<T*>(sm.lines) + lw * a.LS;
    mir = ONE && a.mode == MODE_L;
    const int tl = part * 32 + lane;
    ch = mir ? nwl * 32 - 1 - tl : tl;
    e0 = ch * E;
    cbase = buf + (E + 1) * ch;
    dir = a.bc == 1;
    own = nwl == 1;
    lastR = (RAGGED && !mir && part == nwl - 1) ? ((n - 1) / E) & 31 : 31;
    end0 = dir && e0 == 0;
    endN = dir && n - 1 >= e0 && n - 1 < e0 + E;
  }
  // point k of the chunk in scan order lies on the line
  __device__ __forceinline__ bool valid(int k) const { return !RAGGED || (mir ? e0 + E - 1 - k : e0 + k) < n; }
  // writes the chunk's values (scan order) back to the line
  __device__ __forceinline__ void store(const T (&x)[E]) const {
    if (!mir) {
#pragma unroll
      for (int k = 0; k < E; ++k)
        if (valid(k)) cbase[chunk_off<E>(k)] = x[k];
    } else {
#pragma unroll
      for (int k = 0; k < E; ++k)
        if (valid(k)) cbase[chunk_off<E>(E - 1 - k)] = x[k];
    }
  }
};

// Powers of q: up to this lane inside its warp, up to this warp (R: from the
// left end, L: from the right end; one-sided: in scan order), and the decay
// of the lane that closes the warp's R scan.
template <typename T>
struct LinePowers {
  T pwR, pwL, qwR, qwL, mulR;
};
template <typename T, bool ONE, bool RAGGED, int E>
__device__ __forceinline__ LinePowers<T> line_powers(const LineConst& L, const LineLane<T, ONE, RAGGED, E>& ln) {
  constexpr int LE = log2i<E>();
  LinePowers<T> p{T(1), T(1), T(1), T(1), T(1)};
  const bool ragged_first = RAGGED && (ONE ? ln.mir && ln.part == 0 : ln.part == ln.nwl - 1);
  p.pwR = qpow<T, LE, 5>(L, ln.lane);
  if (!ONE || ln.mir) {
    T pl = ONE ? p.pwR : __shfl_sync(0xffffffffu, p.pwR, 31 - ln.lane);
    if (ragged_first) {
      const int before = ln.n - ln.e0 - E;
      pl = before > 0 ? qpow<T, 0, LE + 5>(L, before) : T(1);
    }
    if (ONE) p.pwR = pl; else p.pwL = pl;
  }
  if (!ln.own) {
    const T qlw = pick<T>(L.qlw, L.qlwf);
    if (!ln.mir) p.qwR = qpow<T, LE + 5, 4>(L, ln.part);
    else if (ln.part > 0) p.qwR = qlw * qpow<T, LE + 5, 4>(L, ln.part - 1);
    if (!ONE && ln.part < ln.nwl - 1) p.qwL = qlw * qpow<T, LE + 5, 4>(L, ln.nwl - 2 - ln.part);
  }
  p.mulR = (RAGGED && !ln.mir && ln.part == ln.nwl - 1) ? pick<T>(L.qlast, L.qlastf) : qpow_bit<T>(L, LE);
  return p;
}

// The chunk's window with three points on either side (ragged lines: their
// ghost cells are in place).
template <typename T, bool ONE, bool RAGGED, int E>
__device__ __forceinline__ void load_window(const LineLane<T, ONE, RAGGED, E>& ln, T (&win)[E + 6]) {
  // window of the chunk in scan orientation: win[j] = v at offset j - 3
  // from the chunk's first point
  if (!ln.mir) {
#pragma unroll
    for (int j = 0; j < E + 6; ++j) win[j] = ln.cbase[chunk_off<E>(j - 3)];
  } else {
#pragma unroll
    for (int j = 0; j < E + 6; ++j) win[j] = ln.cbase[chunk_off<E>(E + 2 - j)];
  }
  if constexpr (!RAGGED) {
    // ghosts of an exact-fit line: only the end lanes need them
    if (ln.e0 == 0 || ln.e0 + E == ln.n) {
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        const int el = ln.mir ? ln.e0 + E + 2 - j : ln.e0 + j - 3;
        const int er = ln.mir ? ln.e0 - 1 - j : ln.e0 + E + j;
        if (el < 0 || el >= ln.n) win[j] = ghost_value<T, E>(ln.buf, el, ln.n, (ln.dir ? 1 : 0));
        if (er < 0 || er >= ln.n) win[E + 3 + j] = ghost_value<T, E>(ln.buf, er, ln.n, (ln.dir ? 1 : 0));
      }
    }
  }
}

// K_R into X and K_L into F of the linear rule (ONE: X alone, in scan order)
// from the window's differences dd[j] = win[j+1] - win[j].
template <typename T, bool ONE, int E>
__device__ __forceinline__ void linear_forcings(const LineConst& a, const T (&dd)[E + 5], T (&X)[E + 1], T (&F)[E]) {
#pragma unroll
  for (int k = 0; k < E; ++k) {
    T r = T(0), l = T(0);
#pragma unroll
    for (int j = 0; j < 5; ++j) {
      const int i = j < 2 ? j : (j < 4 ? j + 1 : 2);   // the large tap last: one rounding at its size
      r = fma(pick<T>(a.b[i], a.bf[i]), dd[k + i], r);
      if constexpr (!ONE) l = fma(-pick<T>(a.b[i], a.bf[i]), dd[k + 5 - i], l);
    }
    X[k] = r;
    if (!ONE) F[k] = l;
  }
}

// The same with WENO-Z weights: dR the differences of the values J_R
// integrates, dL those of J_L (the same ones but for split fluxes).
template <typename T, bool ONE, int E>
__device__ __forceinline__ void wenoz_forcings(const LineConst& a, const T (&dR)[E + 5], const T (&dL)[E + 5],
                                               T (&X)[E + 1], T (&F)[E]) {
  T wc[6], dw[3];
#pragma unroll
  for (int i = 0; i < 6; ++i) wc[i] = pick<T>(a.wk[i], a.wkf[i]);
#pragma unroll
  for (int r = 0; r < 3; ++r) dw[r] = pick<T>(a.d[r], a.df[r]);
  // J_R of point k uses the triples k, k+1, k+2, J_L the triples k+4, k+3,
  // k+2 mirrored
#pragma unroll
  for (int k = 0; k < E; ++k) {
    const Indicators<T> i0(dR[k], dR[k + 1]), i1(dR[k + 1], dR[k + 2]), i2(dR[k + 2], dR[k + 3]);
    X[k] = wenoz_defect<T>(dR[k + 2], dR[k + 1], dR[k], dR[k + 3], i0.outer, i1.plus, i2.minus, wc, dw);
    if constexpr (!ONE) {
      const Indicators<T> l2(dL[k + 2], dL[k + 3]), l1(dL[k + 3], dL[k + 4]), l0(dL[k + 4], dL[k + 5]);
      F[k] = wenoz_defect<T>(-dL[k + 3], -dL[k + 4], -dL[k + 5], -dL[k + 2], l0.outer_mir, l1.minus, l2.plus, wc, dw);
    }
  }
}

// Forcings of D_0 with linear weights: the residual form (X the differences
// d_k, k = 0..E, F the FIR part), or the K filters.
template <typename T, int E>
__device__ __forceinline__ void d0_forcings(const LineConst& a, const T (&dd)[E + 5], T (&X)[E + 1], T (&F)[E]) {
  if (a.d0) {
    const T f0 = pick<T>(a.f0, a.f0f), f1 = pick<T>(a.f1, a.f1f);
    if (f1 != T(0)) {
#pragma unroll
      for (int k = 0; k < E; ++k) {
        const T s0 = dd[k + 2] - dd[k + 1], s1 = dd[k + 3] - dd[k + 2], s2 = dd[k + 4] - dd[k + 3];
        F[k] = fma(f1, s0 + s2, f0 * s1);
      }
    } else {
#pragma unroll
      for (int k = 0; k < E; ++k) F[k] = f0 * (dd[k + 3] - dd[k + 2]);
    }
#pragma unroll
    for (int k = 0; k <= E; ++k) X[k] = dd[k + 2];
  } else {
    linear_forcings<T, false, E>(a, dd, X, F);
  }
}

// Scans of the forcings, R in X and L in F (ONE: X alone; D_0's residual
// form, L.d0: X the differences, F the FIR part): scans from zero (lane
// folds, warp scan, warps of the line), boundary constants, and the scans
// again from their carries.  Leaves W_R in X and W_L in F; ONE, D0: D in F.
template <typename T, bool D0, bool ONE, bool RAGGED, int E>
__device__ __forceinline__ void line_scans(const LineConst& L, const LineLane<T, ONE, RAGGED, E>& ln,
                                           const LinePowers<T>& pw, T (&X)[E + 1], T (&F)[E]) {
  constexpr unsigned FULL = 0xffffffffu;
  constexpr int LE = log2i<E>();
  const T q = qpow_bit<T>(L, 0);
  // Dirichlet ends: no forcing at the node where a scan starts
  const bool resid = D0 && L.d0;
  if (ONE) {
    if (ln.dir) {
#pragma unroll
      for (int k = 0; k < E; ++k) {
        const int e = ln.mir ? ln.e0 + E - 1 - k : ln.e0 + k;
        if (e == (ln.mir ? ln.n - 1 : 0)) X[k] = T(0);
      }
    }
  } else {
    if (ln.end0) X[0] = T(0);
    if (ln.endN) {
#pragma unroll
      for (int k = 0; k < E; ++k)
        if (RAGGED ? ln.e0 + k == ln.n - 1 : k == E - 1) {
          if (resid) X[k + 1] = T(0); else F[k] = T(0);
        }
    }
  }

  // scans from zero: lane folds, warp scan, warps of the line
  T bR = T(0), bL = T(0);
#pragma unroll
  for (int k = 0; k < E; ++k)
    if (ln.valid(k)) bR = fma(q, bR, X[k]);
  if constexpr (!ONE) {
    if (resid) {
#pragma unroll
      for (int k = E - 1; k >= 0; --k)
        if (ln.valid(k)) bL = fma(q, bL, -X[k + 1]);
    } else {
#pragma unroll
      for (int k = E - 1; k >= 0; --k)
        if (ln.valid(k)) bL = fma(q, bL, F[k]);
    }
  }
  const T ownR = bR;
#pragma unroll
  for (int k = 0; k < 5; ++k) {
    const int o = 1 << k;
    const T m = qpow_bit<T>(L, LE + k);
    const T bp = shfl_up(bR, o);
    const T sR = fma(m, bp, bR);
    bR = ln.lane >= o ? sR : bR;
    if constexpr (!ONE) {
      const T bn = shfl_down(bL, o);
      const T sL = fma(m, bn, bL);
      bL = ln.lane + o < 32 ? sL : bL;
    }
  }
  T cR = shfl_up(bR, 1), cL = T(0);     // value entering the lane from zero before the warp
  if (ln.lane == 0) cR = T(0);
  if constexpr (!ONE) {
    cL = shfl_down(bL, 1);
    if (ln.lane == 31) cL = T(0);
  }
  const T endR = fma(pw.mulR, cR, ownR);   // at lane lastR: the warp's R end value
  T inR = T(0), inL = T(0), tR, tL = T(0);
  if (ln.own) {
    tR = __shfl_sync(FULL, endR, ln.lastR);
    if constexpr (!ONE) tL = __shfl_sync(FULL, bL, 0);
  } else {
    T* tot = ln.totals + ln.lw * ln.nwl * 2;
    if (ln.lane == ln.lastR) tot[2 * ln.part] = endR;
    if (!ONE && ln.lane == 0) tot[2 * ln.part + 1] = bL;
    line_sync<T, E>(ln.nwl, ln.lw);
    const int j = ln.lane & 15;
    const bool left = ln.lane >= 16;
    T x = T(0);
    if (j < ln.nwl && !(ONE && left)) x = left ? tot[2 * (ln.nwl - 1 - j) + 1] : tot[2 * j];
    const T x0 = x;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if ((1 << k) < ln.nwl) {
        const T xp = __shfl_up_sync(FULL, x, 1 << k, 16);
        const T sx = fma(qpow_bit<T>(L, LE + 5 + k), xp, x);
        x = j >= (1 << k) ? sx : x;
      }
    }
    T ex = __shfl_up_sync(FULL, x, 1, 16);   // value entering warp j
    if (j == 0) ex = T(0);
    const T lastw = (left || ln.mir) ? qpow_bit<T>(L, LE + 5) : pick<T>(L.qlw, L.qlwf);
    const T te = fma(lastw, ex, x0);
    tR = __shfl_sync(FULL, te, ln.nwl - 1);
    inR = __shfl_sync(FULL, ex, ln.part);
    if constexpr (!ONE) {
      tL = __shfl_sync(FULL, te, 15 + ln.nwl);
      inL = __shfl_sync(FULL, ex, 15 + ln.nwl - ln.part);
    }
  }
  // boundary constants, carried to the lane
  if (L.close) {
    inR = fma(pw.qwR, line_constant<T>(L, tR, tL), inR);
    if constexpr (!ONE) inL = fma(pw.qwL, line_constant<T>(L, tL, tR), inL);
  }
  if (L.close || !ln.own) {
    cR = fma(pw.pwR, inR, cR);
    if constexpr (!ONE) cL = fma(pw.pwL, inL, cL);
  }
  // the scans from their carries -> D of the power (in F; two-sided
  // forms keep W_R, W_L)
  T y = cR;
  if (resid) {
#pragma unroll
    for (int k = 0; k < E; ++k) {
      if (ln.valid(k)) y = fma(q, y, X[k]);
      F[k] = fma(pick<T>(L.kap, L.kapf), y, F[k]);
    }
    y = cL;
#pragma unroll
    for (int k = E - 1; k >= 0; --k) {
      if (ln.valid(k)) y = fma(q, y, -X[k + 1]);
      F[k] = fma(pick<T>(L.kap, L.kapf), y, F[k]);
    }
  } else {
#pragma unroll
    for (int k = 0; k < E; ++k) {
      if (ln.valid(k)) y = fma(q, y, X[k]);
      X[k] = y;
    }
    if constexpr (ONE) {
#pragma unroll
      for (int k = 0; k < E; ++k) F[k] = X[k];
    } else {
      y = cL;
#pragma unroll
      for (int k = E - 1; k >= 0; --k) {
        if (ln.valid(k)) y = fma(q, y, F[k]);
        F[k] = D0 ? T(0.5) * (X[k] + y) : y;
      }
    }
  }
  if constexpr (D0) {
    // D_0 vanishes at Dirichlet ends
    if (ln.end0) F[0] = T(0);
    if (ln.endN) {
#pragma unroll
      for (int k = 0; k < E; ++k)
        if (RAGGED ? ln.e0 + k == ln.n - 1 : k == E - 1) F[k] = T(0);
    }
  }
}

// Applies D P times to the staged lines and leaves S_P (or, for MODE_RL, the
// per-axis Lax-Friedrichs Hamiltonian) in the line buffers.  Returns the
// thread's largest one-sided derivative magnitude (MODE_RL).  Ends
// synchronised (contiguous lines: the line's warps, strided: the CTA).
//
// All scans run in difference form: with W_R = v - L_R^{-1}[v], W_L = v -
// L_L^{-1}[v] and d_i = v_i - v_{i-1} the recurrences of Sec. 2.4 give
//   W_R(x_i) = q W_R(x_{i-1}) + K_R(x_i),  K_R(x_i) = v_i - q v_{i-1} - J_R(x_i),
//   W_L(x_i) = q W_L(x_{i+1}) + K_L(x_i),  K_L(x_i) = v_i - q v_{i+1} - J_L(x_i),
// with K a 5-tap filter of the differences d (the weights of J sum to 1 - q,
// App. C): no value of the size of v is subtracted from another, so FP32
// needs no compensated arithmetic and D of a constant is exactly zero.
//
// D_0 with linear weights (JQ_D0).  D_0 = (W_R + W_L)/2 is a symmetric filter
// delta^2 M(delta^2) / ((1-q)^2 - q delta^2) of v (delta^2 the second
// difference, M a quadratic from the weights).  Dividing M by the denominator
// leaves
//   D_0 v_i = kap (U_i + V_i) + f0 s_i + f1 (s_{i-1} + s_{i+1}),
//   U_i = q U_{i-1} + d_i,  V_i = q V_{i+1} - d_{i+1},  s = delta^2 v:
// the scans take the bare differences, and the whole quadrature enters as
// three constants (the 3-point rule has f1 = 0).  Per point: 11 operations
// (9 with the 3-point rule) where the two 6-tap integrals, folds, fix-ups and
// D = v - (I_R + I_L)/2 took 20.  f0, f1 of the 5- and 6-point rules grow like
// e^{3 nu}: a.d0 chooses this form while they stay small (set_line_constants),
// else the K filters.
//
// JQ_LINEAR1 / JQ_WENOZ1 (MODE_R or MODE_L alone): the one side that is
// asked for, the L side as the R scan of the mirrored line.
//
// Constants of the scans come from the host as powers q^(2^k): the lane maps
// all have the multiplier q^E, so a warp scan moves one value per lane, and a
// line of several warps scans its warps' totals 16 lanes at a time (R in
// lanes 0-15, L in lanes 16-31), each warp for itself: one line_sync per
// application of D and one per write-back, no barrier for a line owned by one
// warp.
// GEN: MODE_RL supports every HamKind (else |grad u|^2/2 only).
template <typename T, int JQ, bool RAGGED, int E = kE, bool GEN = false>
__device__ __forceinline__ double compute_lines(const SweepArgs& a, const TileSmem& sm, bool line_ok) {
  static_assert(JQ != JQ_LEARNED || sizeof(T) == 4, "learned weights run in FP32");
  constexpr bool ONE = JQ == JQ_LINEAR1 || JQ == JQ_WENOZ1;
  constexpr bool WENO = JQ == JQ_WENOZ || JQ == JQ_WENOZ1;
  const LineLane<T, ONE, RAGGED, E> ln(a, sm);
  LinePowers<T> pw;
  if constexpr (JQ != JQ_LEARNED) pw = line_powers<T, ONE, RAGGED, E>(a, ln);   // (not live across the network)
  T S[E];
  T rmax = T(0);

  for (int p = 0; p < a.P; ++p) {
    // ---- 1. forcings of the scans
    // JQ_D0: X the differences d, F the FIR part; else (and in D_0's K form)
    // X = K_R, F = K_L.  Scalar arithmetic: in packed FP32x2 form (R ascending
    // with L descending) the moves that build the pairs cost more than the
    // halved FMA count saved (64 heat problems 11.4 against 12.4 ms a pass).
    T X[E + 1], F[E];
    if constexpr (JQ == JQ_LEARNED || RAGGED) {
      if (ln.part == 0) warp_fill_ghosts<T, E>(a, ln.buf, ln.lane);
      line_sync<T, E>(ln.nwl, ln.lw);
    }
    if constexpr (JQ == JQ_LEARNED) {
      float* jrl = sm.jloc + ln.lw * 2 * a.LS;
      if (line_ok)
        learned_local_integrals<E>(a, *sm.net, ln.buf, jrl, jrl + a.LS,
                                   sm.mlp_scratch + (threadIdx.x >> 5) * kMlpScratchBytes, ln.part * 32 * E, ln.n,
                                   ln.lane);
      __syncwarp();
      pw = line_powers<T, ONE, RAGGED, E>(a, ln);
#pragma unroll
      for (int k = 0; k < E; ++k) {
        X[k] = jrl[(E + 1) * ln.ch + chunk_off<E>(k)];
        F[k] = jrl[a.LS + (E + 1) * ln.ch + chunk_off<E>(k)];
      }
    } else {
      T win[E + 6], dd[E + 5];
      load_window<T, ONE, RAGGED, E>(ln, win);
#pragma unroll
      for (int j = 0; j < E + 5; ++j) dd[j] = win[j + 1] - win[j];
      if constexpr (WENO) wenoz_forcings<T, ONE, E>(a, dd, dd, X, F);
      else if constexpr (JQ == JQ_D0) d0_forcings<T, E>(a, dd, X, F);
      else linear_forcings<T, ONE, E>(a, dd, X, F);
    }
    // ---- 2. scans and boundary constants
    line_scans<T, JQ == JQ_D0, ONE, RAGGED, E>(a, ln, pw, X, F);
    // ---- 3. sum over the powers, write back for the next one
    if constexpr (JQ != JQ_D0 && !ONE) {
      if (a.mode == MODE_RL) {
        // one-sided derivatives v^- = alpha D_R, v^+ = -alpha D_L and the
        // per-axis part of the Lax-Friedrichs Hamiltonian (Sec. 2.5); the
        // linear rule's taps carry the factor alpha
        const T al = JQ == JQ_LINEAR ? T(1) : pick<T>(a.alpha, a.alphaf);
        if (!GEN || a.ham == HAM_HALF_SQ) {
#pragma unroll
          for (int k = 0; k < E; ++k) {
            const T vm = al * X[k];
            const T vp = -al * F[k];
            const T r = fmax(fabs(vm), fabs(vp));
            const T mean = T(0.5) * (vm + vp);
            S[k] = T(0.5) * mean * mean + r * T(0.5) * (vm - vp);
            if (line_ok && (!RAGGED || ln.e0 + k < ln.n)) rmax = fmax(rmax, r);
          }
        } else if constexpr (GEN) {
          // H_d' = a_d (LINEAR) has |H_d'| = |a_d| everywhere; AFFINE_SQ
          // leaves (sigma, delta) and the last pass takes the box maximum
          const T ah = T(0.5) * al * pick<T>(a.vel, a.velf), aa = fabs(ah);
          T* cbase2 = static_cast<T*>(sm.lines2) + (ln.cbase - static_cast<T*>(sm.lines));
#pragma unroll
          for (int k = 0; k < E; ++k) {
            const T mean2 = X[k] - F[k], diff = X[k] + F[k];   // v^- + v^+, v^- - v^+ (over al)
            if (a.ham == HAM_LINEAR) {
              S[k] = fma(ah, mean2, aa * diff);
            } else {
              S[k] = ah * mean2;
              if (ln.valid(k)) cbase2[chunk_off<E>(k)] = -aa * diff;
            }
          }
          if (a.ham == HAM_LINEAR && line_ok) rmax = fabs(pick<T>(a.vel, a.velf));
        }
      } else {
#pragma unroll
        for (int k = 0; k < E; ++k) {
          T D;
          if (a.mode == MODE_0) D = T(0.5) * (X[k] + F[k]);
          else if (a.mode == MODE_R) D = X[k];
          else D = F[k];
          F[k] = D;
        }
      }
    }
    if (JQ == JQ_D0 || ONE || a.mode != MODE_RL) {
#pragma unroll
      for (int k = 0; k < E; ++k) S[k] = p == 0 ? F[k] : S[k] + F[k];
      if (p + 1 < a.P) {
        // every lane of the line has read its window: of a line of several
        // warps, before the totals' barrier
        if (ln.own) __syncwarp();
        ln.store(F);
        line_sync<T, E>(ln.nwl, ln.lw);
      }
    }
  }

  if (ln.own) __syncwarp();
  ln.store(S);
  // the epilogue reads contiguous lines by their ln.own warps, strided ones by rows
  if (a.contiguous) line_sync<T, E>(ln.nwl, ln.lw); else __syncthreads();
  return cvt<double>(rmax);
}

// Epilogue operands of one point, loaded ahead of the stores so that the
// loads of a batch of points are in flight together (the compiler cannot
// move a load past a store to a possibly aliasing array).
template <typename T, typename TST>
struct EpiOps {
  T acc;
  TST x, y;
};

template <typename T, typename TST, int EPI, bool CG = false>
struct Epilogue {
  const SweepArgs& a;
  double dt;
  double tn;   // general HJ_Y with a source: time of the state being advanced

  __device__ __forceinline__ EpiOps<T, TST> load(long long gidx) const {
    EpiOps<T, TST> o{T(0), TST(0), TST(0)};
    if constexpr (EPI == EPI_ACC_ADD || EPI == EPI_ACC_AXPY) {
      o.acc = gload<CG>(static_cast<const T*>(a.acc) + gidx);
    } else if constexpr (EPI == EPI_HEAT_FINAL || EPI == EPI_WAVE_FINAL || EPI == EPI_ADV_FINAL) {
      if (a.acc) o.acc = gload<CG>(static_cast<const T*>(a.acc) + gidx);
      o.x = gload<CG>(static_cast<const TST*>(a.un) + gidx);
      if (EPI != EPI_WAVE_FINAL || !a.from_rest) o.y = gload<CG>(static_cast<const TST*>(a.us) + gidx);
    } else if constexpr (epi_hj_y(EPI)) {
      o.x = gload<CG>(static_cast<const TST*>(a.un) + gidx);
      if (a.out) o.y = gload<CG>(static_cast<const TST*>(a.out) + gidx);
    }
    return o;
  }

  __device__ __forceinline__ void store(long long gidx, T s, const EpiOps<T, TST>& o) const {
    if constexpr (EPI == EPI_STORE) {
      static_cast<TST*>(a.out)[gidx] = cvt<TST>(s);
    } else if constexpr (EPI == EPI_ACC_SET) {
      static_cast<T*>(a.acc)[gidx] = s;
    } else if constexpr (EPI == EPI_ACC_ADD) {
      static_cast<T*>(a.acc)[gidx] = o.acc + s;
    } else if constexpr (EPI == EPI_ACC_AXPY) {
      static_cast<T*>(a.acc)[gidx] = fma(T(a.coefS), s, o.acc);
    } else if constexpr (EPI == EPI_HEAT_FINAL) {
      // u_s = a0 u^n + a1 (u_{s-1} + dt F), dt F = coefS (acc + S)
      const TST r = fma(TST(a.a0), o.x, TST(a.a1) * fma(TST(a.coefS), cvt<TST>(o.acc + s), o.y));
      static_cast<TST*>(a.dst)[gidx] = r;
      if (a.shadow) a.shadow[gidx] = cvt<float>(r);
      if (nonfinite(r)) atomicOr(a.status, ST_NONFINITE);
    } else if constexpr (EPI == EPI_ADV_FINAL) {
      const TST r = fma(TST(a.a0), o.x, TST(a.a1) * (o.y + cvt<TST>(o.acc + s)));
      static_cast<TST*>(a.dst)[gidx] = r;
      if (nonfinite(r)) atomicOr(a.status, ST_NONFINITE);
    } else if constexpr (EPI == EPI_WAVE_FINAL) {
      // u^{n+1} = 2u^n - u^{n-1} + coefS (acc + S)   (from rest: u^n + coefS/2 (acc + S))
      const TST tot = cvt<TST>(o.acc + s);
      const TST r = a.from_rest ? fma(TST(0.5 * a.coefS), tot, o.x) : fma(TST(a.coefS), tot, fma(TST(2), o.x, -o.y));
      if (a.dst2) static_cast<TST*>(a.dst2)[gidx] = o.x;
      static_cast<TST*>(a.dst)[gidx] = r;
      if (a.shadow) a.shadow[gidx] = cvt<float>(r);
      if (nonfinite(r)) atomicOr(a.status, ST_NONFINITE);
    } else if constexpr (epi_hj_x(EPI)) {
      if (a.out) static_cast<TST*>(a.out)[gidx] = TST(s);
    } else if constexpr (epi_hj_y(EPI)) {
      const TST r = o.x - TST(dt) * (o.y + TST(s));
      static_cast<TST*>(a.dst)[gidx] = r;
      if (nonfinite(r)) atomicOr(a.status, ST_NONFINITE);
    }
  }

  // ---- general Hamilton-Jacobi passes (EPI_HJ_XG / EPI_HJ_YG)
  // z: delta_x of AFFINE_SQ from the x pass (last pass), 0 otherwise
  __device__ __forceinline__ TST load_z(long long gidx) const {
    if constexpr (EPI == EPI_HJ_YG)
      if (a.out2) return gload<CG>(static_cast<const TST*>(a.out2) + gidx);
    return TST(0);
  }

  // F(x, t_n) = sum_k t_n^k F_k(x) (Horner)
  __device__ __forceinline__ TST source(long long gidx) const {
    const TST* f = static_cast<const TST*>(a.src) + gidx;
    const TST t = TST(tn);
    TST F = f[a.src_deg * a.src_stride];
    for (int k = a.src_deg - 1; k >= 0; --k) F = fma(F, t, f[k * a.src_stride]);
    return F;
  }

  // s2: the second line buffer's value (two_out).  Returns the point's wave
  // speed over vmax where the last pass determines it (AFFINE_SQ), else 0.
  __device__ __forceinline__ T store_general(long long gidx, T s, const EpiOps<T, TST>& o, TST z, T s2) const {
    if constexpr (EPI == EPI_HJ_XG) {
      if (a.out) static_cast<TST*>(a.out)[gidx] = TST(s);
      if (a.out2) static_cast<TST*>(a.out2)[gidx] = TST(s2);
      return T(0);
    } else {
      TST H;
      T speed = T(0);
      if (a.ham == HAM_AFFINE_SQ) {
        // local Lax-Friedrichs over the box of one-sided derivatives:
        // |dH/dp_d| = |a_d| |h0 + a.p| is largest at a corner, where
        // |h0 + a.p| reaches m = |sbar| + sum_d |delta_d|; then
        // H^ = H(means) - sum_d |a_d| m (v^+_d - v^-_d)/2 = sbar^2/2 - m sum_d delta_d;
        // the speeds c_d = |a_d| m enter as max_d c_d / h_d = m vmax
        const TST sbar = TST(a.h0) + o.y + TST(s);
        const TST m = fabs(sbar) + fabs(z) + fabs(TST(s2));
        H = TST(0.5) * sbar * sbar - m * (z + TST(s2));
        speed = T(m);   // times vmax, once a thread
      } else {
        H = o.y + TST(s);
      }
      if (a.src) H -= source(gidx);
      if (a.dst) {
        const TST r = o.x - TST(dt) * H;
        static_cast<TST*>(a.dst)[gidx] = r;
        if (nonfinite(r)) atomicOr(a.status, ST_NONFINITE);
      }
      return speed;
    }
  }
};

// Applies the epilogue to the tile's W lines in the coalesced mapping, in
// batches of kEpiBatch points per thread: all operand loads of a batch are
// issued before its stores.
#ifndef MOLT_EPI_BATCH
#define MOLT_EPI_BATCH 8
#endif
constexpr int kEpiBatch = MOLT_EPI_BATCH;

// The epilogue of the general Hamilton-Jacobi passes over one thread's points
// p0, p0 + pstep, ... of a line: shared values sp[k*pdelta] and sp2[k*pdelta]
// (second line buffer, or null), global index g + k*gstep, B points per
// batch with all loads of a batch issued before its stores.  Returns the
// largest wave speed it determined, over vmax.
template <typename T, typename TST, int EPI, bool CG, int B>
__device__ __forceinline__ double epilogue_general(const Epilogue<T, TST, EPI, CG>& ep, const T* sp, const T* sp2,
                                                   long long g, int p0, int n, int pstep, long long gstep,
                                                   int pdelta) {
  T rmax = T(0);
  for (int pb = p0; pb < n; pb += B * pstep) {
    EpiOps<T, TST> ops[B];
    T sv[B], sv2[B];
    TST oz[B];
#pragma unroll
    for (int k = 0; k < B; ++k) {
      if (pb + k * pstep < n) {
        ops[k] = ep.load(g + k * gstep);
        oz[k] = ep.load_z(g + k * gstep);
        sv[k] = sp[k * pdelta];
        sv2[k] = sp2 ? sp2[k * pdelta] : T(0);
      }
    }
#pragma unroll
    for (int k = 0; k < B; ++k)
      if (pb + k * pstep < n) rmax = fmax(rmax, ep.store_general(g + k * gstep, sv[k], ops[k], oz[k], sv2[k]));
    g += B * gstep;
    sp += B * pdelta;
    if (sp2) sp2 += B * pdelta;
  }
  return cvt<double>(rmax);
}

// Returns the largest wave speed the epilogue determined (HJ_Y with
// AFFINE_SQ), else 0.  lines2: the second line buffer (two_out) or null.
template <typename T, typename TST, int EPI, int E = kE, bool CG = false>
__device__ __forceinline__ double epilogue_tile(const SweepArgs& a, const T* lines, long long line0, double dt,
                                                const T* lines2 = nullptr) {
  const Epilogue<T, TST, EPI, CG> ep{a, dt, (epi_hj_y(EPI) && epi_hj_gen(EPI) && a.src) ? *a.t_now : 0.0};
  const int W = a.W, n = a.g.n, nwl = a.nwl;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  long long g0;
  const T* src0;
  int p0, pstep, sstep;
  long long gstep;
  if (a.contiguous) {
    const int lw = warp / nwl, tl = (warp - lw * nwl) * 32 + lane;
    if (line0 + lw >= a.g.nlines) return 0.0;
    p0 = tl;
    pstep = nwl * 32;
    g0 = line_base(a.g, line0 + lw) + p0;
    gstep = pstep;
    src0 = lines + lw * a.LS;
    sstep = 0;
  } else {
    const int w = tid % W;
    const long long gl = line0 + w;
    if (gl >= a.g.nlines) return 0.0;
    p0 = tid / W;
    pstep = blockDim.x / W;
    g0 = line_base(a.g, gl) + p0 * a.g.stride;
    gstep = pstep * a.g.stride;
    src0 = lines + w * a.LS;
    sstep = 1;
  }
  // shared index of point p: contiguous lines step p by a multiple of 32,
  // strided lines by blockDim/W (a multiple of 16), so phys<E>() advances by a
  // constant in both cases
  const int pdelta = pstep + pstep / E;
  const T* sp = src0 + phys<E>(p0);
  (void)sstep;
  if constexpr (epi_hj_gen(EPI)) {
    // more operands per point: a smaller batch
    return a.vmax * epilogue_general<T, TST, EPI, CG, 4>(ep, sp, lines2 ? lines2 + (sp - lines) : nullptr, g0, p0, n,
                                                          pstep, gstep, pdelta);
  } else {
    long long g = g0;
    for (int pb = p0; pb < n; pb += kEpiBatch * pstep) {
      EpiOps<T, TST> ops[kEpiBatch];
      T sv[kEpiBatch];
#pragma unroll
      for (int k = 0; k < kEpiBatch; ++k) {
        if (pb + k * pstep < n) {
          ops[k] = ep.load(g + k * gstep);
          sv[k] = sp[k * pdelta];
        }
      }
#pragma unroll
      for (int k = 0; k < kEpiBatch; ++k)
        if (pb + k * pstep < n) ep.store(g + k * gstep, sv[k], ops[k]);
      g += kEpiBatch * gstep;
      sp += kEpiBatch * pdelta;
    }
    return 0.0;
  }
}

template <int EPI>
__device__ __forceinline__ double hj_dt(const SweepArgs& a) {
  double dt = 0.0;
  if constexpr (epi_hj_y(EPI)) {
    if (!a.lag) return 0.0;   // a pass that only measures speeds
    const double cl = __longlong_as_double((long long)a.lag[0]);
    dt = a.dt_max;
    if (cl > 0.0 && a.cfl / cl < dt) dt = a.cfl / cl;
  }
  return dt;
}

template <int EPI>
__device__ __forceinline__ void publish_speed(const SweepArgs& a, double rmax) {
  if constexpr (epi_hj_x(EPI) || epi_hj_y(EPI)) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) rmax = fmax(rmax, __shfl_xor_sync(0xffffffffu, rmax, o));
    if ((threadIdx.x & 31) == 0 && rmax > 0.0 && a.speed)
      atomicMax(a.speed, (unsigned long long)__double_as_longlong(rmax));
  }
}

// One tile per CTA, plain coalesced loads (any size / alignment).
template <typename T, typename TIN, typename TST, int JQ, int EPI, bool RAGGED, int E = kE>
__global__ void __maxnreg__((sweep_regs<T, JQ, E>())) sweep_kernel(const SweepArgs a) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  size_t used;
  const TileSmem sm = carve<T, JQ>(smem_raw, a, &used);
  if constexpr (JQ == JQ_LEARNED) mlp_load_net_half(*sm.net, a.mlp);
  T* lines = static_cast<T*>(sm.lines);
  const long long line0 = (long long)blockIdx.x * a.W;
  const int warp = threadIdx.x >> 5, lw = warp / a.nwl;
  const int tl = (warp - lw * a.nwl) * 32 + (threadIdx.x & 31);
  load_tile<T, TIN, E>(a, static_cast<const TIN*>(a.in), lines, line0, lw, tl,
                       [](T* d, const TIN* g) { *d = cvt<T>(*g); });
  if (a.contiguous && JQ != JQ_LEARNED) line_sync<T, E>(a.nwl, lw); else __syncthreads();
  if constexpr (epi_hj_x(EPI) || epi_hj_y(EPI)) {
    const double rmax =
        compute_lines<T, JQ, RAGGED, E, epi_hj_gen(EPI)>(a, sm, line0 + lw < a.g.nlines) * a.inv_h;
    // the general last pass finds its speeds in the epilogue
    if constexpr (!epi_hj_gen(EPI)) publish_speed<EPI>(a, rmax);
    const double dt = hj_dt<EPI>(a);
    if (epi_hj_y(EPI) && blockIdx.x == 0 && threadIdx.x == 0 && a.t_dev) *a.t_dev += dt;
    const double re = epilogue_tile<T, TST, EPI, E>(a, lines, line0, dt, static_cast<const T*>(sm.lines2));
    if constexpr (epi_hj_gen(EPI)) publish_speed<EPI>(a, fmax(rmax, re));
  } else {
    compute_lines<T, JQ, RAGGED, E>(a, sm, line0 + lw < a.g.nlines);
    epilogue_tile<T, TST, EPI, E>(a, lines, line0, 0.0);
  }
}

}  // namespace molt
