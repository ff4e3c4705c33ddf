"""What the benchmark says it launched is the library's own plan (host logic, no GPU)."""
import os
import sys

import pytest

pytest.importorskip("torch")
from conftest import ROOT  # noqa: E402

sys.path.insert(0, ROOT)
import bench  # noqa: E402


@pytest.mark.parametrize("plan,nx,storage,want", [
    (("march", 34, 3, 0), 4096, "fp32", "k_march3<fp32,fluid> (3 steps per launch)"),
    (("tile", 5, 4, 64), 512, "fp32", "k_tile<fp32,fluid> (4 steps per launch)"),
    (("single", 100, 1, 0), 1024, "fp32", "k_step_vec<fp32,4,fluid>"),
    (("single", 100, 1, 0), 1024, "fp16", "k_step_vec<fp16,8,fluid>"),
    (("single", 2, 1, 0), 1023, "bf16", "k_step_scalar<bf16,1,fluid>")])
def test_kernel_label_follows_the_plan(plan, nx, storage, want):
    assert bench.kernel_label(plan, "d2q9", storage, nx, "fluid") == want


def test_no_launch_count_of_the_benchmark_s_own():
    assert not hasattr(bench, "passes") and not hasattr(bench, "STEPS_PER_PASS")
    assert bench.SlabRun.step_plan(None, 7) == ("single", 7, 1, 0)


@pytest.mark.gpu
@pytest.mark.parametrize("size", [512, 1024])
def test_reported_launches_are_the_plan_s(size, tmp_path):
    """A line of the benchmark at sizes that do not march: launches and label of the plan."""
    import json
    import subprocess

    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1312_3297_gb300 import D2Q9

    out = subprocess.run([sys.executable, os.path.join(ROOT, "bench.py"), "--size", str(size),
                          "--mode", "fluid", "--steps", "20", "--no-extras", "--no-e2e",
                          "--no-cpu"], capture_output=True, text=True, check=True).stdout
    line = json.loads(out.strip().splitlines()[-1])
    with D2Q9(size, size, bench.S_RATES) as sim:
        plan = sim.step_plan(20)
    assert line["gpu_launches"] == plan[1]
    assert line["roofline"]["kernel"] == bench.kernel_label(plan, "d2q9", "fp32", size, "fluid")
