"""The scan kernel's forms of D against the oracle, where they can go wrong:
D_0 with linear weights on both sides of the rule that picks the residual
form or the K filters (nu about 1.7 for the 6-point rule), one-sided sweeps
(the L side runs the line mirrored), and lines around the edges of lanes,
warps and tiles, where the scans' carries change hands."""
import pytest

from paper_2007_03041_gb300 import molt as M
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
