// Launch of the fused advection-diffusion axis kernel for one state type (a
// translation unit each).
#pragma once

#include "advdiff_axis.cuh"

namespace molt {

template <typename T, bool WENO, int EPI, bool RAGGED, int E>
cudaError_t launch_advdiff_kernel(const AdvArgs& A, int grid, int block, size_t smem, cudaStream_t s) {
  static bool configured = false;
  if (!configured) {
    const cudaError_t e = cudaFuncSetAttribute(&advdiff_axis_kernel<T, WENO, EPI, RAGGED, E>,
                                               cudaFuncAttributeMaxDynamicSharedMemorySize, int(kSmemTileBudget));
    if (e != cudaSuccess) return e;
    configured = true;
  }
  advdiff_axis_kernel<T, WENO, EPI, RAGGED, E><<<grid, block, smem, s>>>(A);
  return cudaGetLastError();
}

// Exact-fit lines of 16 points a lane run unmasked, all others masked.
template <typename T, bool WENO, int EPI>
cudaError_t launch_advdiff_shape(const AdvArgs& A, int grid, int block, size_t smem, cudaStream_t s) {
  if (A.a.E == 8) return launch_advdiff_kernel<T, WENO, EPI, true, 8>(A, grid, block, smem, s);
  if (A.a.E == 4) return launch_advdiff_kernel<T, WENO, EPI, true, 4>(A, grid, block, smem, s);
  if (A.a.g.n == A.a.nwl * 32 * 16) return launch_advdiff_kernel<T, WENO, EPI, false, 16>(A, grid, block, smem, s);
  return launch_advdiff_kernel<T, WENO, EPI, true, 16>(A, grid, block, smem, s);
}

template <typename T>
cudaError_t launch_advdiff_axis_t(bool weno, int epi, const AdvArgs& A, int grid, int block, size_t smem,
                                  cudaStream_t s) {
  if (epi == EPI_ACC_SET)
    return weno ? launch_advdiff_shape<T, true, EPI_ACC_SET>(A, grid, block, smem, s)
                : launch_advdiff_shape<T, false, EPI_ACC_SET>(A, grid, block, smem, s);
  if (epi == EPI_ACC_ADD)
    return weno ? launch_advdiff_shape<T, true, EPI_ACC_ADD>(A, grid, block, smem, s)
                : launch_advdiff_shape<T, false, EPI_ACC_ADD>(A, grid, block, smem, s);
  if (epi == EPI_ADV_FINAL)
    return weno ? launch_advdiff_shape<T, true, EPI_ADV_FINAL>(A, grid, block, smem, s)
                : launch_advdiff_shape<T, false, EPI_ADV_FINAL>(A, grid, block, smem, s);
  return cudaErrorNotSupported;
}

}  // namespace molt
