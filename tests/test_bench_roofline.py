"""bench.py names the bound of each kernel: instruction issue for the binary64
transforms (integers), the FP64 pipe for what a binary64 solve leaves there, HBM for
the FP32 form."""
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)
import bench  # noqa: E402

PEAKS = {"hbm_gbs": 6800.0, "source": "test"}
FP64 = {"gflops": 1250.0, "source": "test"}
POINTS = 1 << 22


def rec(name, ms, bytes_, flops=0.0, launches=10):
    return dict(name=name, launches=launches, ms_total=ms * launches, bytes_total=bytes_ * launches, flops_total=flops * launches)


def test_bound_of_each_kernel():
    stats = [rec("atkm_z_f64", 0.23, 4.7e8, 5e9), rec("H_z_f64", 0.11, 72.0 * POINTS, 1e9), rec("H_x_f64", 0.08, 32.0 * POINTS, 1e9),
             rec("vec_dir_dots", 0.12, 80.0 * POINTS), rec("vec_lincomb", 0.055, 64.0 * POINTS), rec("atkm_z_f32", 0.09, 2.4e8, 5e9)]
    r = bench.roofline(stats, PEAKS, FP64, True, POINTS)
    assert r["kernel"] == "atkm_z_f64" and r["bound"] == "issue" and r["frac"] == bench.ISSUE_SLOTS["atkm_z"]
    assert abs(r["hbm_GBs"] - 4.7e8 / 0.23e-3 / 1e9) < 0.1 and os.path.exists(os.path.join(ROOT, bench.ISSUE_PROFILE))
    bound = {p["name"]: p["bound"] for p in r["passes"]}
    assert bound == {"atkm_z_f64": "issue", "H_z_f64": "fp64", "H_x_f64": "issue", "vec_dir_dots": "fp64", "vec_lincomb": "hbm",
                     "atkm_z_f32": "hbm"}
    # 14 instructions a point against half the FMA flops
    frac = {p["name"]: p["frac"] for p in r["passes"]}
    assert abs(frac["vec_dir_dots"] - 14 * POINTS / 0.12e-3 / 1e9 / 625.0) < 1e-3
    f32 = bench.roofline(stats[3:], PEAKS, FP64, False, POINTS)
    assert {p["bound"] for p in f32["passes"]} == {"hbm"}
