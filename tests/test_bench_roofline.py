"""The roofline entries of bench.py count the work of the stencil that ran
(CPU only): integer multiply-adds for the fixed-point FP64 stencil, FP64
operations for the FP64 kernels, which serve small solves, links off SU(3)
and calls without memory for the fixed-point links."""
import pytest

import bench

V, M, MHZ = 4096, 3, 2000.0


@pytest.mark.parametrize("per_call,unit", [(5, "Tmad/s"), (4, "TFLOP/s")])
def test_residuals(per_call, unit):
    calls, ms = 7, 2.0
    nbytes = calls * (8.0 * M * 12 * V + 2 * 36 * V) * 16          # the library's count for A
    r = bench.residual_roofline(per_call * calls, nbytes, ms, V, M, MHZ)
    work = {"Tmad/s": 1728, "TFLOP/s": 1368}[unit] * 2 * V * M * calls
    assert r["unit"] == unit and r["fields_per_solve"] == M * calls
    assert r["achieved"] == pytest.approx(work / (ms / 1e3) / 1e12, abs=1e-4)
    assert ("mads_per_solve" in r) == (unit == "Tmad/s")
    assert r["frac"] == pytest.approx(r["achieved"] / r["peak"], abs=1e-3)


@pytest.mark.parametrize("other,dslash,unit", [(3, 6, "Tmad/s"), (0, 6, "TFLOP/s"), (3, 12, "TFLOP/s")])
def test_fp64_applications(other, dslash, unit):
    """A with a conversion per call; without one; repeated by the FP64 kernels."""
    r = bench.fp64_stencil_roofline({"other": other, "dslash": dslash}, 3, 2, 1.5, V, M, MHZ)
    assert r["unit"] == unit and r["ms_per_launch"] == pytest.approx(1.5 / dslash, abs=1e-4)
    per = {"Tmad/s": 1728, "TFLOP/s": 1368}[unit]
    assert r["achieved"] == pytest.approx(per * V * M / (1.5 / dslash / 1e3) / 1e12, abs=1e-4)
