"""The scan kernel's forms of D against the oracle, where they can go wrong:
D_0 with linear weights on both sides of the rule that picks the residual
form or the K filters (nu = 1.66 for the 5-point rule, 2.08 for the 6-point
one; the 3-point rule stays with the residual form), one-sided sweeps
(the L side runs the line mirrored), and lines around the edges of lanes,
warps and tiles, where the scans' carries change hands."""
import numpy as np
import pytest

from oracle import sweep
from paper_2007_03041_gb300 import molt as M
from tests.gpu_util import need_gpu, to_dev
from tests.test_gpu_apply_D import check, run_apply

pytestmark = pytest.mark.gpu

LENGTHS = (5, 15, 16, 17, 127, 128, 129, 256, 511, 512, 513, 528, 1024, 1025, 1536, 3000, 8191, 8192)


@pytest.mark.parametrize("prec", [M.PREC_F64, M.PREC_F32_F64UPDATE, M.PREC_F32])
@pytest.mark.parametrize("bc", [M.BC_PERIODIC, M.BC_DIRICHLET])
@pytest.mark.parametrize("op", [M.OP_L, M.OP_R, M.OP_0])
def test_line_edges(prec, bc, op):
    for k, n in enumerate(LENGTHS):
        got, want = run_apply((3, n), 0, op, 1 + k % 3, 0.3, bc, (3, 5, 6)[k % 3], prec, seed=n)
        check(got, want, prec, 2, 0, (n, "rows"))
    for n in (100, 513, 2048):
        got, want = run_apply((n, 21), 1, op, 2, 0.3, bc, 6, prec, seed=n)
        check(got, want, prec, 2, 1, (n, "columns"))


@pytest.mark.parametrize("prec", [M.PREC_F64, M.PREC_F32])
@pytest.mark.parametrize("bc", [M.BC_PERIODIC, M.BC_DIRICHLET])
@pytest.mark.parametrize("npts", [3, 5, 6])
def test_both_forms_of_D0(prec, bc, npts):
    for nu in (1.2, 1.6, 1.8, 2.0, 2.3, 2.6, 4.0, 9.0):
        for n in (300, 512, 2048):
            got, want = run_apply((2, n), 0, M.OP_0, 2, nu, bc, npts, prec, seed=n)
            check(got, want, prec, 2, 0, (n, nu))


@pytest.mark.parametrize("prec", [M.PREC_F64, M.PREC_F32])
@pytest.mark.parametrize("bc", [M.BC_PERIODIC, M.BC_DIRICHLET])
@pytest.mark.parametrize("op", [M.OP_L, M.OP_R, M.OP_0])
def test_wenoz_line_edges(prec, bc, op):
    for n in (100, 128, 513, 1024, 2048):
        got, want = run_apply((3, n), 0, op, 1, 2.0 / 3.0, bc, 5, prec, weights=M.W_WENOZ, seed=n)
        check(got, want, prec, 2, 0, n)


@pytest.mark.parametrize("prec", [M.PREC_F64, M.PREC_F32])
@pytest.mark.parametrize("n,W", [(1000, 4), (1024, 4), (1100, 2), (1536, 2), (2048, 2)])
def test_tiles_of_several_lines_of_several_warps(prec, n, W):
    """Enough lines that a CTA holds 2 or 4 lines of 2 to 4 warps, whose
    barriers it shares or keeps apart; the last tile is partly empty."""
    lines = 1301
    plan = M.molt_plan_sweep(M.make_desc((n, lines), prec=prec), 0, M.OP_0, 2, 0.3 * n)
    assert (plan["points_per_lane"], plan["lines_per_cta"]) == (16, W) and plan["warps_per_line"] > 1
    for k, bc in enumerate((M.BC_PERIODIC, M.BC_DIRICHLET)):
        got, want = run_apply((lines, n), 0, M.OP_0, 2, 0.3, bc, 6, prec, seed=n + k)
        check(got, want, prec, 2, 0, (n, "rows"))
        got, want = run_apply((n, lines), 1, (M.OP_R, M.OP_L)[k], 2, 0.3, bc, 6, prec, seed=n + k)
        check(got, want, prec, 2, 1, (n, "columns"))
    if prec == M.PREC_F32:
        got, want = run_apply((lines, n), 0, M.OP_0, 1, 2.0 / 3.0, M.BC_PERIODIC, 5, prec, weights=M.W_WENOZ, seed=n)
        check(got, want, prec, 2, 0, (n, "WENO-Z rows"))


@pytest.mark.parametrize("npts", [3, 5, 6])
@pytest.mark.parametrize("n", [500, 512])
def test_symbol_of_D0_in_fp32(n, npts):
    """The gain of D_0 on Fourier modes, by projection over many lines of
    random phase (rounding noise averages out: 5e-9), is that of the exact
    rule to 2^-25 / (1 - q).  Rounding q to FP32 moves the relative symbol by
    up to 2^-25 (1 + 2q/(1-q)) between its ends; the other constants, fitted to
    the rounded q, leave at most half of that and half an ulp of kap.  The
    nearest FP32 constants leave the whole of it."""
    need_gpu()
    import torch
    lines = 2048
    phase = np.random.default_rng(n).uniform(0.0, 2 * np.pi, (lines, 1))
    for nu in (0.2, 0.3, 0.6):
        bound = 2.0 ** -25 / (-np.expm1(-nu)) + 5e-9
        for k in (4, 25, 100):
            u = np.cos(2 * np.pi * k * np.arange(n) / n + phase).astype(np.float32)
            ctx = M.molt_create(M.make_desc((n, lines), P=1, quad_points=npts, prec=M.PREC_F32))
            try:
                uin = to_dev(u, torch.float32)
                out = torch.empty_like(uin)
                M.molt_apply_D(ctx, 0, 0, M.OP_0, 1, nu * n, uin, out)
                got = out.double().cpu().numpy()
            finally:
                M.molt_destroy(ctx)
            want = sweep.partial_sum(u.astype(np.float64), 1, nu * n, 1.0 / n, "0", "periodic", npts, 1, "linear")
            gain = np.vdot(got, want) / np.vdot(want, want) - 1.0
            assert abs(gain) <= bound, (nu, k, gain, bound)
