"""The kernel whose profiled traffic the benchmark quotes is the one its linear layer runs."""
import os
import re
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)
import bench  # noqa: E402


def test_kernel_is_defined_in_the_files_its_profile_is_bound_to():
    text = "".join(open(os.path.join(ROOT, "paper_2604_16855_b200", "csrc", f)).read() for f in bench.LINEAR_KERNEL_SOURCES)
    assert re.search(r"__global__[^;{]*\b%s\(" % bench.LINEAR_KERNEL, text)
    assert len(bench.kernel_source_hash(bench.LINEAR_KERNEL_SOURCES)) == 64


LAYER = """
import torch
from torch.profiler import ProfilerActivity, profile
from paper_2604_16855_b200 import tdq
M, C, O = 32 * 577, 768, 3072                            # the benchmark's default workload
codes = torch.zeros((M, C // 2), dtype=torch.uint8, device="cuda")
wcodes = torch.zeros((O, C // 2), dtype=torch.uint8, device="cuda")
scale, wscale = torch.ones((M, C // 32), device="cuda"), torch.ones((O,), device="cuda")
y = torch.empty((M, O), device="cuda")
torch.cuda.synchronize()
with profile(activities=[ProfilerActivity.CUDA]) as p:
    tdq.w4a4_linear(codes, scale, wcodes, wscale, y=y)
    torch.cuda.synchronize()
print(max((e.device_time, e.name) for e in p.events() if "tdq::" in e.name)[1])
"""


@pytest.mark.gpu
def test_default_workload_runs_it():
    r = subprocess.run([sys.executable, "-c", LAYER], cwd=ROOT, capture_output=True, text=True, timeout=300)   # the profiler stays out of this process
    assert r.returncode == 0, r.stderr
    assert bench.LINEAR_KERNEL in r.stdout
