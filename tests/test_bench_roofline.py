"""The roofline line's peak for the FP64 Schwarz factorisation follows the kernel that ran: blocks of at most 160
unknowns are inverted on the FP64 pipe, larger ones form their trailing products on the integer pipe (CPU only)."""
import importlib.util
import os

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.parametrize("max_block,fixed_point", [(112, False), (160, False), (164, True), (372, True)])
def test_fp64_patch_factor_peak(max_block, fixed_point):
    spec = importlib.util.spec_from_file_location("bench_roofline_mod", os.path.join(ROOT, "bench.py"))
    b = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(b)
    kst = {"patch_factor": {"ms": 10.0, "bytes": 1e9, "flops": 5e9, "launches": 2},
           "assemble": {"ms": 1.0, "bytes": 1e6, "flops": 1e6, "launches": 2}}
    roof, _ = b._roofline(kst, steps=1, max_block=max_block)
    peak = b.FIXED_POINT_PEAK_GFLOPS if fixed_point else b.FP64_ALU_PEAK_GFLOPS
    assert roof["kernel"] == "patch_factor" and roof["bound"] == "alu"
    assert roof["peak"] == pytest.approx(peak / 1e3) and roof["frac"] == pytest.approx(500.0 / peak)
