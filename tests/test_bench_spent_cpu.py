"""Roofline fractions of the benchmark are in operations that the kernels execute on the pipe
that bounds them: at times measured on a GB300 each is a fraction, also where the fixed unit of
work holds operations that are no longer executed."""
import importlib.util
import os

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PEAKS = {"hbm_gbs": 6791.4, "sm_max_mhz": 2070.0}


@pytest.fixture(scope="module")
def bench():
    spec = importlib.util.spec_from_file_location("bench_spent", os.path.join(ROOT, "bench.py"))
    mod = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(mod)
    return mod


# class, spec, stats, n, ms per launch, executed per pair, pipe peak in T/s
FP32_T, FP64_T = 152 * 128 * 2070e6 / 1e12, 152 * 1.7 * 2070e6 / 1e12
CASES = [
    ("matvec_fp32", ("fp32", "soft", 64), {"matvec_variant": 2}, 32768, 2.45, 46, FP32_T),
    ("matvec_fp32", ("fp32", "hard", 1), {"matvec_variant": 2}, 32768, 3.0, 52, FP32_T),
    ("matvec_fp64", ("fp32", "soft", 64), {"residual_variant": 2}, 32768, 15.2, 352, FP32_T),
    ("matvec_fp64", ("fp32", "hard", 16), {"residual_variant": 2}, 4096, 0.3, 623, FP32_T),
    ("matvec_fp64", ("fp64", "hard", 16), {}, 4096, 2.1, 42, FP64_T),
    ("matvec_fp64", ("fp64", "soft", 1), {}, 1024, 0.09, 25.5, FP64_T)]


@pytest.mark.parametrize("cls,shape,stats,n,ms,spent,pipe", CASES)
def test_fractions_are_of_executed_operations(bench, cls, shape, stats, n, ms, spent, pipe):
    prec, bc, nrhs = shape
    spec = {"nrhs": nrhs, "bc": bc, "precision": prec, "curve": "kite"}
    r = bench.kernel_rooflines({cls: (10 * ms, 10)}, spec, stats, PEAKS, "measured", n, 1)[cls]
    launches = 2 if bc == "hard" and stats.get("residual_variant") == 2 else 1   # S and C
    want = spent * n * n / (launches * ms / 1e3) / 1e12 / pipe
    assert abs(r["frac_spent"] - want) < 1e-9 * want
    assert 0.05 < r["frac_spent"] <= 1.0 and r["frac"] <= 1.0
    assert abs(r["achieved"] / r["peak"] - r["frac"]) < 1e-9
    assert "frac_spent" in bench._brief({"config": {"workload": "w"}, "roofline": r})["roofline"]
