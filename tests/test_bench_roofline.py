"""bench.py's rooflines: kernels whose float64 products are formed from integers are measured
against the HBM peak, the eigensolve against the FP64 peak."""
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)


def test_peaks():
    import bench
    rec = {"ms": 2.0, "launches": 2, "bytes": 4e9, "flops": 4e9}
    for name in bench.SINGLE_KERNELS:
        r = bench.class_roofline(name, rec, 5000.0, "measured")
        assert (r["bound"], r["unit"], r["peak"]) == ("hbm", "GB/s", 5000.0)
        assert abs(r["achieved"] - 2000.0) < 1e-6 and abs(r["frac"] - 0.4) < 1e-9 and "integer" in r["limited_by"]
    r = bench.class_roofline("dense_eig", rec, 5000.0, "measured", fp64_unit=True)
    assert (r["bound"], r["unit"]) == ("alu", "TFLOP/s") and abs(r["achieved"] - 2.0) < 1e-9
