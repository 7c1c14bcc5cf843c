"""Launches of the fused round whose dynamic shared memory is at the edge of what a launch gets without asking
(48 KB, the kernel's own variables included): a warp per row with fp32 storage takes 2048 k + 16 n rounds
bytes, which is 49,152 for 32 devices with 22 selected in launches of 8 rounds and with 23 selected in launches
of 4.  Each as the first launch of a process, in which nothing has raised the limit before."""
import os
import subprocess
import sys

import pytest

from gpu_common import require_gpu

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CHILD = """
import sys
import numpy as np, torch
from paper_2111_08274_b200 import runtime, workloads
k, count = int(sys.argv[1]), int(sys.argv[2])
wl = workloads.Workload("edge", 32, 4097, k, count, "fixed", (1,) * 32, grad_std=1e-2, seed=workloads.BASE_SEED + k)
fused, plain = runtime.Arena(wl), runtime.Arena(wl)
got = fused.run_rounds_fused(0, count)
want = np.stack([plain.run_round(r) for r in range(count)])
torch.cuda.synchronize()
assert np.array_equal(got, want)
assert torch.equal(fused.w, plain.w) and torch.equal(fused.m, plain.m)
fused.h.debug_check()
"""


@pytest.mark.parametrize("k,count", [(21, 8), (22, 8), (23, 4), (23, 8)])
def test_first_launch_of_a_process(k, count):
    require_gpu()
    run = subprocess.run([sys.executable, "-c", CHILD, str(k), str(count)], cwd=ROOT, capture_output=True, text=True)
    assert run.returncode == 0, run.stderr[-2000:]
