"""What the sweep kernels compile to, as nvcc and ptxas report it (no GPU).
Barriers: an SM has 64, so a kernel that reserves 16 a CTA runs at most
four CTAs per SM, and the one-warp CTAs of a grid with few lines leave it idle."""
import re
import subprocess

import pytest

from paper_2007_03041_gb300 import build


def compile_kernel(tmp_path, kernel, *extra):
    try:
        nvcc = build.nvcc()
    except RuntimeError:
        pytest.skip("needs nvcc")
    src = tmp_path / "k.cu"
    src.write_text('#include "sweep.cuh"\nnamespace molt {\ntemplate __global__ void %s(const SweepArgs);\n}\n' % kernel)
    return subprocess.run([nvcc] + build.ARCH + build.FLAGS + list(extra) + ["-Xptxas", "-v", "-cubin", "-o",
                                                                             str(tmp_path / "k.cubin"), str(src)],
                          capture_output=True, text=True)


@pytest.mark.parametrize("kernel,most", [
    ("sweep_kernel<float, float, float, JQ_D0, EPI_STORE, true, 4>", 1),
    ("sweep_kernel<float, float, float, JQ_D0, EPI_STORE, false, 16>", 1),
    ("sweep_kernel<double, double, double, JQ_D0, EPI_STORE, true, 8>", 1),
    ("sweep_kernel<double, double, double, JQ_D0, EPI_STORE, true, 16>", 5),   # 12 CTAs per SM; 80 registers: 25 warps
])
def test_sweep_kernels_leave_the_barriers_free(tmp_path, kernel, most):
    r = compile_kernel(tmp_path, kernel)
    assert r.returncode == 0, r.stderr
    assert int(re.search(r"used (\d+) barriers", r.stderr).group(1)) <= most


def test_tiles_wider_than_the_scans_are_refused(tmp_path):
    """More than 16 warps to a line: the scan of their totals would drop some."""
    kernel = "sweep_kernel<float, float, float, JQ_D0, EPI_STORE, true, 4>"
    assert compile_kernel(tmp_path, kernel, "-DMOLT_MAX_THREADS=256").returncode == 0
    r = compile_kernel(tmp_path, kernel, "-DMOLT_MAX_THREADS=1024")
    assert r.returncode != 0 and "16 warps a line at most" in r.stderr
