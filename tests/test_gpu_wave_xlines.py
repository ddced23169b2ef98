"""The wave step's fused update and x sweep (xline_wave_kernel) against the
FP64 oracle: every multi-step call of a mixed problem whose x lines are 16 S
points, from rest and continued, in the forms whose code differs: lines of 512
points and shorter ones (several to a warp, one to a warp with idle lanes),
periodic and Dirichlet, line counts that leave the last warp's group partly
empty, 2-D and 3-D, P = 1 and 2, the K filters of a large nu, two problems in
one context.  The launch counts say which route ran."""
import numpy as np
import pytest

from oracle import schemes
from paper_2007_03041_gb300 import molt as M
from paper_2007_03041_gb300 import workloads
from tests.gpu_util import assert_grid_parity, need_gpu, to_dev

pytestmark = pytest.mark.gpu

BCS = {M.BC_PERIODIC: "periodic", M.BC_DIRICHLET: "dirichlet"}
BETA = 0.8


class Wave:
    """One mixed wave problem, its state on the GPU and the oracle's."""

    def __init__(self, shape, bc, P, npts, step, seed):
        import torch
        g = workloads.rng(seed)
        self.bc, self.P, self.npts = bc, P, npts
        per = bc == M.BC_PERIODIC
        self.hs = [1.0 / (n if per else n - 1) for n in shape]
        self.dt = step * self.hs[-1]                # numpy's last axis is x
        u = np.zeros(shape)
        for _ in range(3):
            f = 1.0
            for k, (n, h) in enumerate(zip(shape, self.hs)):
                x = (np.arange(n) * h).reshape([-1 if j == k else 1 for j in range(len(shape))])
                m = int(g.integers(1, 4))
                f = f * (np.sin(2 * np.pi * m * x + g.uniform(0, 6)) if per else np.sin(np.pi * m * x))
            u = u + g.uniform(0.3, 1.0) * f
        self.cur, self.prev = u, None
        self.u, self.up = to_dev(u, torch.float64), torch.full(u.shape, float("nan"), device="cuda", dtype=torch.float64)
        self.desc = M.make_desc(tuple(reversed(shape)), bc=[bc] * len(shape), P=P, quad_points=npts, beta=BETA,
                                pde=M.PDE_WAVE, c=1.0, dt=self.dt, prec=M.PREC_F32_F64UPDATE)

    def oracle(self, nsteps):
        for _ in range(nsteps):
            nxt = schemes.wave_step(self.cur, self.prev, self.hs, self.dt, 1.0, BETA, [BCS[self.bc]] * self.cur.ndim,
                                    self.npts, self.P, from_rest=self.prev is None)
            self.prev, self.cur = self.cur, nxt

    def check(self, what):
        assert_grid_parity(self.u.cpu().numpy(), self.cur, 1e-5, what="u " + what)
        assert_grid_parity(self.up.cpu().numpy(), self.prev, 1e-5, what="u_prev " + what)


def run_calls(waves, calls=(3, 1, 2)):
    need_gpu()
    ctx = M.molt_create([w.desc for w in waves])
    try:
        M.molt_set_option(ctx, M.OPT_PROFILE, 1)
        t = [0.0] * len(waves)
        for nsteps in calls:
            t = M.molt_step(ctx, [w.u for w in waves], [w.up for w in waves], nsteps=nsteps, t=t)
            count = {k: M.molt_profile_read(ctx, k)[1] for k in (M.KERNEL_XLINES_WAVE, M.KERNEL_XLINES_ACC_SET,
                                                                M.KERNEL_UPDATE)}
            # the copy with the first x sweep, updates with the next one, the last update alone
            assert count == {M.KERNEL_XLINES_WAVE: (nsteps - 1) * len(waves), M.KERNEL_XLINES_ACC_SET: len(waves),
                             M.KERNEL_UPDATE: len(waves)}, (nsteps, count)
            for w in waves:
                w.oracle(nsteps)
                w.check("%s after a call of %d steps" % (w.cur.shape, nsteps))
    finally:
        M.molt_destroy(ctx)


# numpy shape, P, rule, dt / h_x (nu = BETA h / dt)
CASES = [
    ((5, 7, 512), 2, 6, 2.0),      # one 512-point line a warp
    ((19, 512), 1, 5, 2.0),        # 2-D, P = 1
    ((7, 9, 64), 2, 6, 2.0),       # 8 lines a warp, 63 of them
    ((3, 11, 16), 2, 6, 2.0),      # 32 lines a warp, 33
    ((37, 96), 2, 6, 1.0),         # 6 segments: one line a warp, 26 idle lanes
    ((6, 5, 128), 2, 3, 2.0),      # the 3-point rule (f1 = 0)
    ((6, 5, 128), 2, 6, 0.3),      # nu = 2.7: K filters
]


@pytest.mark.parametrize("bc", [M.BC_PERIODIC, M.BC_DIRICHLET])
@pytest.mark.parametrize("case", CASES, ids=["x".join(map(str, c[0])) + "-P%d-r%d-%g" % c[1:] for c in CASES])
def test_update_with_the_next_x_sweep(case, bc):
    need_gpu()
    run_calls([Wave(case[0], bc, case[1], case[2], case[3], seed=len(case[0]) + case[0][-1])])


def test_two_wave_problems_in_one_context():
    need_gpu()
    run_calls([Wave((9, 10, 64), M.BC_DIRICHLET, 2, 6, 2.0, seed=1), Wave((21, 512), M.BC_PERIODIC, 2, 6, 2.0, seed=2)])
