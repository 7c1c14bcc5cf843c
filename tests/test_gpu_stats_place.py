"""Statistics that are read now and then: whether the last launches wrote them to the host or to the device, a
read returns those of the round it names."""
import numpy as np
import pytest

from gpu_common import require_gpu
from paper_2111_08274_b200 import runtime, workloads
from paper_2111_08274_b200.workloads import Workload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("gap", [1, 3, 4, 5, 9])
def test_reads_with_gaps(gap):
    require_gpu()
    wl = Workload("gaps", 4, 20_003, 2, 40, "fixed", (1, 2, 3, 4), grad_std=1e-2, seed=workloads.BASE_SEED + 9)
    always, now_and_then = runtime.Arena(wl), runtime.Arena(wl)
    for r in range(3 * gap):
        always.run_round_fused(r)
        now_and_then.run_round_fused(r)
        want = always.h.stats_read()
        if r % gap == gap - 1:
            got = now_and_then.h.stats_read()
            assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1])
    for a in (always, now_and_then):           # a batch, and the statistics of a reference model after it
        a.run_rounds_fused(3 * gap, 5)
    back = [now_and_then.h.stats_read_round(b) for b in (4, 0, 2)]
    for b, got in zip((4, 0, 2), back):
        want = always.h.stats_read_round(b)
        assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1])
    now_and_then.h.stats_enqueue(1)
    assert now_and_then.h.stats_read()[1][1] == 0.0
    again = now_and_then.h.stats_read_round(3)
    want = always.h.stats_read_round(3)
    assert np.array_equal(again[0], want[0]) and np.array_equal(again[1], want[1])
    always.close()
    now_and_then.close()
