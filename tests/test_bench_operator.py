"""The bench's roofline of the operator's application (host arithmetic): rates for
the workload whose entries per step were counted, none for the others."""

import os
import sys

import pytest

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
import bench  # noqa: E402

RATES = ("achieved", "frac", "flops_per_step", "fp64_instructions_per_step", "coefficient_bytes_per_step",
         "hbm_gbs_coefficients")


@pytest.mark.parametrize("workload", sorted(bench.WORKLOADS))
def test_operator_rates_only_where_the_entries_were_counted(workload):
    r = bench.op_roofline(workload, {"replay_ms": 10.0, "replay_steps": 2e9})
    assert r["steps_per_launch"] == 2e9 and r["ms_per_launch"] == 10.0
    if workload == "slab65":
        assert r["achieved"] == pytest.approx(2 * 2.24 * 2e9 / 1e-2 / 1e12, rel=1e-3)
        assert r["frac"] == pytest.approx(r["achieved"] / bench.PEAK_FP64_TFLOPS, rel=1e-3)
        assert r["hbm_gbs_coefficients"] == pytest.approx(8 * 2.24 * 2e9 / 1e-2 / 1e9, rel=1e-3)
    else:
        assert all(r[k] is None for k in RATES)
