"""The benchmark's JSON line of a plain FP64 solve, from fake kernel statistics (no GPU needed)."""
import json
import os
import sys
import types

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)


@pytest.mark.parametrize("top,unit", [("gram_fp64", "TFLOP/s"), ("plane_fft_vloc_fp64", "GB/s")])
def test_fp64_roofline(top, unit):
    """An FP64 solve has FP64 classes only.  Its products are rated against the digit products'
    peak (a 34th of the BF16 rate), which no measured rate exceeds, not against the FP64 units'."""
    import bench
    names = ["col_inverse_fft_fp64", "plane_fft_vloc_fp64", "col_forward_fft_fp64", "nonlocal_project_fp64",
             "nonlocal_add_fp64", "gram_fp64", "rotate_fp64", "vector_fp64", "dense_la"]
    stats = {k: dict(launches=0, ms=0.0, bytes=0.0, flops=0.0)
             for k in ("col_inverse_fft", "plane_fft_vloc", "col_forward_fft", "nonlocal_project", "nonlocal_D",
                       "nonlocal_add", "gram", "rotate", "vector")}
    stats.update({k: dict(launches=10, ms=10.0, bytes=1e9, flops=1e11) for k in names})
    stats[top]["ms"] = 1000.0
    stats["gram_fp64"]["flops"] = 15e12                              # 15 TFLOP/s over a second
    args = types.SimpleNamespace(precision="fp64", no_cpu=True, no_fp64=True, steps=1, warmup=3, workload="tiny")
    w = types.SimpleNamespace(n=(16, 16, 32), natom=8, nproj=4, nstates=8, e_ref=0.3, nbands=12)
    ctx = types.SimpleNamespace(npw=1069, gvectors=lambda: np.zeros((1069, 3), dtype=np.int32))
    r = [dict(nconv=8, iters=50, iters_mixed=0, n_hpsi=1000, resid=np.zeros(8), status=0)]
    clocks = {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": []}
    d = bench.make_line(args, w, ctx, r, stats, 8, 1.0, 1.0, 8, clocks, 6793.4, 1980.5, "measured", 1,
                        np.zeros((12, 10), complex))
    roof = d["roofline"]
    assert roof["kernel"] == top and roof["unit"] == unit
    assert 0 < roof["frac"] <= 1 and roof["frac"] == roof["achieved"] / roof["peak"]
    if unit == "TFLOP/s":
        assert roof["bound"] == "tensor" and roof["peak"] == 1980.5 / 34
    json.dumps(d)
