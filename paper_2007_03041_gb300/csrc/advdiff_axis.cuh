// One axis of an advection-diffusion stage in one pass over the state (FP32
// and FP64 states, periodic axes, one term per sum): per line
//   S = cR D_R[f^+] + cL D_L[f^-] + cD D_0[u],  f^{+-} = (g(u) +- c u)/2
// (arXiv 2007.03041, Sec. 2.5), the split fluxes formed from the staged
// state, both one-sided scans side by side, then the diffusive pair.  The
// terms as passes of their own (fluxes to memory, one accumulating sweep
// each) moved 15 values a point and axis where this moves 2 or 3, and staged
// the line three times.  Bound by instructions with WENO-Z weights (three
// weighted integrals a point).
#pragma once

#include "sweep.cuh"

namespace molt {

struct AdvArgs {
  SweepArgs a;        // geometry, epilogue operands, constants of the hyperbolic terms
  LineConst dif;      // constants of the diffusive term
  int burgers, diffusive;
  double c, vel;      // splitting speed, g(u) = vel u (not Burgers)
  double cR, cL, cD;
};

template <typename T, bool WENO, int EPI, bool RAGGED, int E>
__global__ void __maxnreg__(128) advdiff_axis_kernel(const AdvArgs A) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  const SweepArgs& a = A.a;
  size_t used;
  const TileSmem sm = carve<T>(smem_raw, a, &used);
  const long long line0 = (long long)blockIdx.x * a.W;
  const LineLane<T, false, RAGGED, E> ln(a, sm);
  load_tile<T, T, E>(a, static_cast<const T*>(a.in), static_cast<T*>(sm.lines), line0, ln.lw,
                     ln.part * 32 + ln.lane, [](T* d, const T* g) { *d = *g; });
  if (a.contiguous) line_sync<T, E>(ln.nwl, ln.lw); else __syncthreads();
  if constexpr (RAGGED) {
    if (ln.part == 0) warp_fill_ghosts<T, E>(a, ln.buf, ln.lane);
    line_sync<T, E>(ln.nwl, ln.lw);
  }
  T S[E], X[E + 1], F[E];
  {
    T win[E + 6], dR[E + 5], dL[E + 5];
    load_window<T, false, RAGGED, E>(ln, win);
    auto flux = [&](T v, T* p, T* m) {
      const T g = A.burgers ? T(0.5) * v * v : T(A.vel) * v, cu = T(A.c) * v;
      *p = T(0.5) * (g + cu);
      *m = T(0.5) * (g - cu);
    };
    T p0, m0;
    flux(win[0], &p0, &m0);
#pragma unroll
    for (int j = 0; j < E + 5; ++j) {
      T p1, m1;
      flux(win[j + 1], &p1, &m1);
      dR[j] = p1 - p0;
      dL[j] = m1 - m0;
      p0 = p1;
      m0 = m1;
    }
    if constexpr (WENO) {
      wenoz_forcings<T, false, E>(a, dR, dL, X, F);
    } else {
      T unused[E], X2[E + 1];
      linear_forcings<T, false, E>(a, dR, X, unused);
      linear_forcings<T, false, E>(a, dL, X2, F);
    }
    line_scans<T, false, false, RAGGED, E>(a, ln, line_powers<T, false, RAGGED, E>(a, ln), X, F);
#pragma unroll
    for (int k = 0; k < E; ++k) S[k] = fma(T(A.cL), F[k], T(A.cR) * X[k]);
  }
  if (A.diffusive) {
    line_sync<T, E>(ln.nwl, ln.lw);   // the totals are reused
    T win[E + 6], dd[E + 5];
    load_window<T, false, RAGGED, E>(ln, win);
#pragma unroll
    for (int j = 0; j < E + 5; ++j) dd[j] = win[j + 1] - win[j];
    if constexpr (WENO) wenoz_forcings<T, false, E>(A.dif, dd, dd, X, F);
    else d0_forcings<T, E>(A.dif, dd, X, F);
    line_scans<T, !WENO, false, RAGGED, E>(A.dif, ln, line_powers<T, false, RAGGED, E>(A.dif, ln), X, F);
#pragma unroll
    for (int k = 0; k < E; ++k) S[k] = fma(T(A.cD), WENO ? T(0.5) * (X[k] + F[k]) : F[k], S[k]);
  }
  // (every lane of the line read its window before the last scan's barrier)
  if (ln.own) __syncwarp();
  ln.store(S);
  if (a.contiguous) line_sync<T, E>(ln.nwl, ln.lw); else __syncthreads();
  epilogue_tile<T, T, EPI, E>(a, static_cast<const T*>(sm.lines), line0, 0.0);
}

// epi: EPI_ACC_SET, EPI_ACC_ADD or EPI_ADV_FINAL (defined for float and double).
template <typename T>
cudaError_t launch_advdiff_axis_t(bool weno, int epi, const AdvArgs& A, int grid, int block, size_t smem,
                                  cudaStream_t s);

}  // namespace molt
