"""Barriers that the sweep kernels reserve, as ptxas reports them (compiled
here, no GPU): an SM has 64, so a kernel that reserves 16 a CTA runs at most
four CTAs per SM, and the one-warp CTAs of a grid with few lines leave it idle."""
import re
import subprocess

import pytest

from paper_2007_03041_gb300 import build


def barriers(tmp_path, kernel):
    try:
        nvcc = build.nvcc()
    except RuntimeError:
        pytest.skip("needs nvcc")
    src = tmp_path / "k.cu"
    src.write_text('#include "sweep.cuh"\nnamespace molt {\ntemplate __global__ void %s(const SweepArgs);\n}\n' % kernel)
    r = subprocess.run([nvcc] + build.ARCH + build.FLAGS + ["-Xptxas", "-v", "-cubin", "-o", str(tmp_path / "k.cubin"),
                                                            str(src)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return int(re.search(r"used (\d+) barriers", r.stderr).group(1))


@pytest.mark.parametrize("kernel,most", [
    ("sweep_kernel<float, float, float, JQ_D0, EPI_STORE, true, 4>", 1),
    ("sweep_kernel<float, float, float, JQ_D0, EPI_STORE, false, 16>", 1),
    ("sweep_kernel<double, double, double, JQ_D0, EPI_STORE, true, 8>", 1),
    ("sweep_kernel<double, double, double, JQ_D0, EPI_STORE, true, 16>", 5),   # 12 CTAs per SM; 80 registers: 25 warps
])
def test_sweep_kernels_leave_the_barriers_free(tmp_path, kernel, most):
    assert barriers(tmp_path, kernel) <= most
