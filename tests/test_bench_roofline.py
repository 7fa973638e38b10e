"""The benchmark's roofline entries: a rate of operations that are not all executed
is no fraction of a peak."""
import numpy as np

import bench
from paper_1812_04719_gb300 import stiv as S


def test_fp64_procedure_rate_has_no_fraction():
    counts = np.zeros(S.NCOUNTS, dtype=np.int64)
    counts[S.C_FLOPS], counts[S.C_PATCH] = 450_000_000, 1000
    peaks = {"fp64_gflops": 1057.0, "sm_max_mhz": 2070.0}
    r = bench.kernel_roofline(S, None, "fp64", S.STIV_FP64, {"fp64": 0.4, "narrow": 0.1}, counts, peaks, None, 152)
    assert r["kernel"].startswith("fp64_kernel") and r["frac"] is None
    assert abs(r["achieved"] - 1125.0) < 1e-6          # above the peak: no fraction of it
    assert "procedure" in r["work"] and "not computed" in r["work"]
