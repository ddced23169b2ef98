"""The fused advection-diffusion axis kernel against the oracle at the edges
of its shapes: lines around lane, warp and tile ends, one to three axes, no
diffusion, both integrators.  In 2-D the y axis runs on column tiles in place,
that of larger grids whose tiles have narrow rows on the transposed state:
ROUTES has both sides of that rule, and the unmasked kernel of 16 points a lane
in both precisions."""
import numpy as np
import pytest

from oracle import schemes
from paper_2007_03041_gb300 import molt as M
from tests.gpu_util import assert_grid_parity, need_gpu, state_dtype, to_dev, tol_for
from tests.test_gpu_advdiff import _field
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


# numpy shape, prec, weights, npts, whether y runs on the transposed state
ROUTES = [
    ((70, 2600), F32, WZ, 5, False),       # column tiles, 4 points a lane, masked
    ((300, 2600), F32, LIN, 6, False),     # 16 points a lane, masked
    ((512, 2600), F32, WZ, 5, False),      # 16 points a lane, exact
    ((512, 2600), F32, LIN, 6, False),
    ((1024, 2440), F32, WZ, 5, False),     # two warps a line
    ((64, 1300), F64, WZ, 5, False),
    ((1024, 1300), F64, WZ, 5, False),     # exact, two warps a line
    ((1024, 1300), F64, LIN, 6, False),
    ((1300, 1024), F64, WZ, 5, False),     # x exact
    ((128, 128), F32, WZ, 5, False),       # rows of 4 bytes, small
    ((512, 512), F32, WZ, 5, False),       # rows of 4 bytes, 2^18 points
    ((512, 515), F32, WZ, 5, True),        # just over
    ((1024, 700), F32, LIN, 6, True),      # rows of 8 bytes; the transposed lines exact
    ((1024, 1500), F32, WZ, 5, False),     # rows of 16 bytes
    ((2048, 1500), F32, LIN, 6, True),     # the same, long lines
    ((8192, 129), F32, WZ, 5, True),       # the longest lines
    ((2048, 150), F64, LIN, 6, True),      # FP64: long lines only
    ((2047, 150), F64, WZ, 5, False),
    ((11, 20, 35), F32, WZ, 5, None),      # 3-D: column tiles along y and z
    ((10, 33, 18), F64, WZ, 5, None),
    ((9, 64, 128), F64, LIN, 6, None),
]


@pytest.mark.parametrize("case", ROUTES, ids=["x".join(map(str, c[0])) + "-%d-%d" % c[1:3] for c in ROUTES])
def test_fused_axis_routes(case):
    need_gpu()
    shape, prec, weights, npts, transposed = case
    nd = len(shape)
    vel = (0.7, -0.4, 0.25)[:nd]
    hs = [2 * np.pi / n for n in shape]
    c, kappa, beta = 1.6, 0.01, 0.6
    dt = 0.5 * min(hs) / c
    u0 = _field(shape, 60 + nd)
    if prec == F32:
        u0 = u0.astype(np.float32).astype(np.float64)
    d = M.make_desc(tuple(reversed(shape)), lo=[0.0] * nd, hi=[2 * np.pi] * nd, P=1, quad_points=npts, weights=weights,
                    beta=beta, pde=M.PDE_ADVDIFF, c=c, diffusivity=kappa, dt=dt, prec=prec, velocity=vel, flux=B,
                    integrator=M.INT_EULER)
    ctx = M.molt_create(d)
    try:
        M.molt_set_option(ctx, M.OPT_PROFILE, 1)
        u = to_dev(u0, state_dtype(prec))
        M.molt_step(ctx, u, None, nsteps=2, t=[0.0])
        got = u.double().cpu().numpy()
        axes = M.molt_profile_read(ctx, M.KERNEL_ACC_ADD)[1]
        turns = M.molt_profile_read(ctx, M.KERNEL_TRANSPOSE)[1]
        flux = M.molt_profile_read(ctx, M.KERNEL_FLUX)[1]
    finally:
        M.molt_destroy(ctx)
    assert (axes, turns, flux) == (2 * nd, 2 if transposed else 0, 0)
    want = u0
    for _ in range(2):
        want = schemes.advdiff_step(want, hs, dt, schemes.FLUX_BURGERS, vel[::-1], c, kappa, beta, npts, 1, False,
                                    "wenoz" if weights == WZ else "linear")
    assert_grid_parity(got, want, tol_for(prec), what=str(case))
