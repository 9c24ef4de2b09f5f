"""The DRAM traffic that the bench line reports for the mixed 4M-cell smoother
classes is that of the kernels that run: the committed launch list of the cluster
sweeps, to the 0.1 MB it prints.  The sweeps' latency model counts their steps."""
import os
import re

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
KERNELS = {"ilu_fwd": "k_sweep<float, 0, 0>", "ilu_bwd": "k_sweep<float, 1, 0>",
           "ilu_resid": "k_resid_scaled<float, 0, 0>", "ilu_apply": "k_apply_z<float, 0>"}


@pytest.fixture(scope="module")
def bench():
    import sys
    sys.path.insert(0, ROOT)
    import bench
    return bench


def test_reported_traffic_is_the_present_kernels(bench):
    rows = {}
    with open(os.path.join(ROOT, "profiles", "launch_list_3d-200x200x100-mixed-clusters.md")) as f:
        for line in f:
            m = re.match(r"\| (k_\S.*?) \| \d+ \| [\d.]+ \| [\d.]+% \| ([\d.]+) MB \| ([\d.]+) MB \|", line)
            if m:
                rows[m.group(1).replace("\\", "")] = float(m.group(2)) + float(m.group(3))
    for cls, kern in KERNELS.items():
        assert abs(bench.CLUSTER_TRAFFIC[("3d-200x200x100-mixed", cls)] / 1e6 - rows[kern]) <= 0.15, cls
    with open(os.path.join(ROOT, "paper_1705_05783_gb300", "csrc", "k_sweep.cu")) as f:
        src = f.read()
    for kern in KERNELS.values():
        assert re.search(r"\b" + kern.split("<")[0] + r"\(", src), kern


@pytest.mark.parametrize("precision, steps", [(0, 200 + 200 + 100 - 3), (1, 50 + 200 + 100 - 3)])
def test_latency_model_counts_the_sweeps_steps(bench, precision, steps):
    w = bench.WORKLOADS["3d-200x200x100"].with_(precision=precision)
    out = bench.sweep_latency_bound({"ilu_fwd": (10, 1.0, 10)}, w)
    assert out["steps"] == steps and abs(out["bound_us"] - steps * bench.T_STEP_US[precision]) < 1e-9
    assert abs(out["ilu_fwd"]["frac"] - out["bound_us"] / 100.0) < 1e-9
