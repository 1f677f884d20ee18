"""The FP64 roofline entry of the benchmark names the kernel that ran and its own bound."""
import importlib.util
import os

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_fp64_roofline_names_the_form():
    spec = importlib.util.spec_from_file_location("bench_labels", os.path.join(ROOT, "bench.py"))
    bench = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(bench)
    kinds = {"iface_apply": "coupled", "local_solve": "local"}
    st = {"iface_apply": {"achieved_GBs": 4000.0, "ms_per_step": 2.0}, "vector": {"achieved_GBs": None, "ms_per_step": 9.0},
          "local_solve": {"achieved_GBs": 3000.0, "ms_per_step": 1.0}}
    fixed = bench._fp64_roofline(st, {"coupled": (100.0, 110.0)}, kinds, 6700.0, "measured", 1.05)
    assert "k_fxgemv" in fixed["kernel"] and fixed["unit"] == "GB/s" and fixed["bound"] != "hbm"
    dense = bench._fp64_roofline(st, {"coupled": (100.0, 100.0)}, kinds, 6700.0, "measured", 1.05)
    assert "k_gemv<double>" in dense["kernel"] and dense["unit"] == "GFLOP/s"
    assert abs(dense["frac"] - 4000.0 / 8.0 * 2.0 / 1050.0) < 1e-12
    st["coarse"] = {"achieved_GBs": 1000.0, "ms_per_step": 5.0}     # always dense
    assert "k_gemv<double>" in bench._fp64_roofline(st, {"coupled": (100.0, 110.0)}, kinds, 6700.0, "measured", 0.0)["kernel"]
