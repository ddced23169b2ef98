// FP32 sweeps on FP64 state: the sweeps read the FP32 copy of the state, the
// state update runs in FP64, the boundary constants in pairs of FP32 numbers.
#include "sweep_launch.h"

namespace molt {
MOLT_DEFINE_LAUNCH
MOLT_INST(float, float, double, JQ_D0, EPI_STORE)
MOLT_INST(float, float, double, JQ_D0, EPI_ACC_SET)
MOLT_INST(float, float, double, JQ_D0, EPI_ACC_ADD)
MOLT_INST(float, float, double, JQ_D0, EPI_HEAT_FINAL)
MOLT_INST(float, float, double, JQ_D0, EPI_WAVE_FINAL)
MOLT_INST(float, double, double, JQ_D0, EPI_STORE)
MOLT_INST(float, double, double, JQ_LINEAR1, EPI_STORE)
MOLT_INST(float, double, double, JQ_WENOZ, EPI_STORE)
MOLT_INST(float, double, double, JQ_WENOZ1, EPI_STORE)
}  // namespace molt
