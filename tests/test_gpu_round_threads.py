"""Two threads with a handle each run batches of rounds side by side whose launches take the same kernel with
different amounts of shared memory: rows on the SM with 16 and 32 devices (arenas beyond the L2), a warp per
row with 24 and 31 selected devices (both above 48 KB).  Every call succeeds, and the results are those of
the same rounds run alone, bit for bit."""
import threading

import numpy as np
import pytest
import torch

from gpu_common import require_gpu
from paper_2111_08274_b200 import runtime, workloads
from paper_2111_08274_b200.workloads import Workload

pytestmark = pytest.mark.gpu

PAIRS = {"on_the_sm": ((16, 1_250_001, 4), (32, 620_003, 8)), "warp_per_row": ((32, 4_097, 24), (32, 4_097, 31))}
CALLS, ROUNDS = 150, 4


def arena(n, P, k, seed, stream=None):
    return runtime.Arena(Workload("thr", n, P, k, 1, "fixed", (1,) * n, grad_std=1e-2, seed=workloads.BASE_SEED + seed),
                         stream=stream)


@pytest.mark.parametrize("pair", sorted(PAIRS))
def test_two_handles_in_two_threads(pair):
    require_gpu()
    side = [arena(*shape, seed=i, stream=torch.cuda.Stream()) for i, shape in enumerate(PAIRS[pair])]
    errors, start = [], threading.Barrier(2)

    def work(a):
        try:
            torch.cuda.set_device(0)
            start.wait(timeout=30)
            for c in range(CALLS):
                a.run_rounds_fused(c * ROUNDS, ROUNDS)
            a.h.synchronize()
        except Exception as e:  # noqa: BLE001 - the main thread reports it
            errors.append(repr(e))

    threads = [threading.Thread(target=work, args=(a,)) for a in side]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    for i, shape in enumerate(PAIRS[pair]):
        alone = arena(*shape, seed=i)
        for c in range(CALLS):
            alone.run_rounds_fused(c * ROUNDS, ROUNDS)
        alone.h.synchronize()
        assert torch.equal(alone.w, side[i].w) and torch.equal(alone.m, side[i].m)
        assert all(np.array_equal(x, y) for x, y in zip(alone.h.get_versions(), side[i].h.get_versions()))
        alone.close()
    for a in side:
        a.close()
