"""A process that used the library can unload it, and ends normally with and without handles left."""
import os
import subprocess
import sys

import pytest

from gpu_common import require_gpu

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CHILD = """
import _ctypes, sys
from paper_2111_08274_b200 import binding
lib = binding.lib()
handles = [binding.Hadfl(4, 1000) for _ in range(2)]
for h in handles:
    h.round([0, 1, 2, 3], [1] * 4, 0.01, 0, 2, 1)
    h.stats_read()
if sys.argv[1] != "handles_left":
    for h in handles:
        h.destroy()
if sys.argv[1] == "unload":
    binding._lib = None
    _ctypes.dlclose(lib._handle)
    assert not any("libhadfl" in line for line in open("/proc/self/maps"))
print("end", flush=True)
"""


@pytest.mark.parametrize("how", ["unload", "destroyed", "handles_left"])
def test_end_of_a_process(how):
    require_gpu()
    run = subprocess.run([sys.executable, "-c", CHILD, how], cwd=ROOT, capture_output=True, text=True, timeout=120)
    assert run.returncode == 0 and run.stdout == "end\n", run.stderr[-2000:]
