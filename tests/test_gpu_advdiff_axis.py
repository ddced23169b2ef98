"""The fused advection-diffusion axis kernel against the oracle at the edges
of its shapes: lines around lane, warp and tile ends (exact-fit lines of 512,
1024 points; masked ones of 4, 8 and 16 points a lane), one to three axes,
no diffusion, both integrators, and y lines long enough to run on the
transposed state (rows of a tile under 32 bytes)."""
import pytest

from paper_2007_03041_gb300 import molt as M
from tests.test_gpu_advdiff import test_advdiff_steps_match_oracle as run_case

pytestmark = pytest.mark.gpu

L, B = M.FLUX_LINEAR, M.FLUX_BURGERS
F32, F64 = M.PREC_F32, M.PREC_F64
LIN, WZ = M.W_LINEAR, M.W_WENOZ

# numpy shape, flux, rk3, P, prec, weights, npts, kappa, beta, c
CASES = [
    ((33, 127), B, False, 1, F32, WZ, 5, 0.01, 0.6, 1.6),
    ((128, 129), B, False, 1, F32, LIN, 3, 0.01, 0.6, 1.6),
    ((512, 513), L, False, 1, F32, WZ, 5, 0.01, 0.5, 1.0),
    ((37, 512), B, True, 1, F64, LIN, 5, 0.0, 0.4, 1.6),
    ((1024, 21), B, False, 1, F64, WZ, 5, 0.01, 0.6, 1.6),
    ((511,), L, True, 1, F32, LIN, 6, 0.02, 0.5, 1.0),
    ((1024,), B, False, 1, F64, WZ, 5, 0.0, 0.6, 1.6),
    ((9, 17, 33), L, True, 1, F32, LIN, 6, 0.03, 0.3, 1.0),
    ((2053, 70), B, False, 1, F32, WZ, 5, 0.01, 0.6, 1.6),
    ((4096, 65), B, False, 1, F32, LIN, 6, 0.01, 0.6, 1.6),
    ((2049, 33), L, True, 1, F64, WZ, 5, 0.01, 0.5, 1.0),
]


@pytest.mark.parametrize("case", CASES, ids=["x".join(map(str, c[0])) for c in CASES])
def test_fused_axis_edges(case):
    run_case(case)
