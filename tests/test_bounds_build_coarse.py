"""The bounds-check variant of the coarse-level kernels compiles for sm_103a and carries its own site word (no GPU
needed); the checks run in tests/test_gpu_bounds_build.py."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1709_05660_gb300", "csrc")


@pytest.mark.skipif(shutil.which("nvcc") is None and not os.path.exists("/usr/local/cuda/bin/nvcc"),
                    reason="nvcc not available")
@pytest.mark.parametrize("unit", ["coarse", "slab"])
def test_checked_kernels_compile(unit, tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    obj = str(tmp_path / "unit.o")
    p = subprocess.run([nvcc, "-gencode=arch=compute_103a,code=sm_103a", "-std=c++17", "-O3",
                        "--expt-relaxed-constexpr", "-DFSI_BOUNDS_CHECK", "-I" + os.path.join(ROOT, "include"), "-c",
                        os.path.join(CSRC, f"k_{unit}.cu"), "-o", obj], capture_output=True, text=True, timeout=600)
    assert p.returncode == 0, p.stdout + p.stderr
    names = subprocess.run(["nm", "-C", obj], capture_output=True, text=True, check=True).stdout
    assert f"fsi::bounds_site_{unit}()" in names and "fsi::bounds::g_site" in names
