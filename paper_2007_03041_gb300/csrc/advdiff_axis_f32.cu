// The fused advection-diffusion axis kernel (csrc/advdiff_axis.cuh), FP32.
#define MOLT_LINE_BARRIERS 1
#include "advdiff_axis_launch.h"

namespace molt {
template cudaError_t launch_advdiff_axis_t<float>(bool, int, const AdvArgs&, int, int, size_t, cudaStream_t);
}  // namespace molt
