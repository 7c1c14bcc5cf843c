"""Statistics that are read now and then: whether the last launches wrote them to the host or to the device, a
read returns those of the round it names - also after a launch that failed, and after a replayed graph."""
import ctypes
import glob
import os

import numpy as np
import pytest
import torch

from gpu_common import require_gpu
from paper_2111_08274_b200 import binding, runtime, workloads
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


def cudart():
    found = glob.glob(os.path.join(os.path.dirname(os.path.dirname(torch.__file__)), "nvidia", "cuda_runtime", "lib",
                                   "libcudart.so*"))
    assert found
    return ctypes.CDLL(found[0])


@pytest.mark.parametrize("launches_since_read", [0, 1, 3, 4, 5, 9])
@pytest.mark.parametrize("call", ["round", "rounds", "stats"])
def test_statistics_stay_readable_after_a_launch_that_failed(call, launches_since_read):
    """The launch is refused by the runtime: the stream is in a capture that a synchronisation has invalidated
    (nothing reaches the GPU)."""
    require_gpu()
    rt, stream = cudart(), torch.cuda.Stream()
    wl = Workload("refused", 4, 20_003, 2, 40, "fixed", (1, 2, 3, 4), grad_std=1e-2, seed=workloads.BASE_SEED + 10)
    a, same = runtime.Arena(wl, stream=stream), runtime.Arena(wl)
    a.run_round_fused(0), same.run_round_fused(0)
    a.h.stats_read()
    for r in range(launches_since_read):
        a.run_rounds_fused(1 + 3 * r, 3), same.run_rounds_fused(1 + 3 * r, 3)
    a.h.synchronize()
    at = ctypes.c_void_p(stream.cuda_stream)
    assert rt.cudaStreamBeginCapture(at, 2) == 0            # relaxed
    assert rt.cudaStreamSynchronize(at) != 0                # not permitted: the capture is invalid from here on
    refused = {"round": lambda: a.run_round_fused(99), "rounds": lambda: a.run_rounds_fused(99, 3),
               "stats": lambda: a.h.stats_enqueue(0)}[call]
    with pytest.raises(binding.HadflError):
        refused()
    graph = ctypes.c_void_p()
    assert rt.cudaStreamEndCapture(at, ctypes.byref(graph)) != 0
    rt.cudaGetLastError()
    got, want = a.h.stats_read(), same.h.stats_read()
    assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1])
    for back in range(3 if launches_since_read else 1):
        got, want = a.h.stats_read_round(back), same.h.stats_read_round(back)
        assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1])
    assert all(np.array_equal(x, y) for x, y in zip(a.h.get_versions(), same.h.get_versions()))
    a.close()
    same.close()


@pytest.mark.parametrize("watched", [False, True])    # whether statistics are being read when the graph is captured
@pytest.mark.parametrize("watched_at_replay", [False, True])
def test_statistics_of_a_replayed_graph(watched, watched_at_replay):
    require_gpu()
    stream = torch.cuda.Stream()
    wl = Workload("graph", 4, 20_003, 2, 40, "fixed", (1, 2, 3, 4), grad_std=1e-2, seed=workloads.BASE_SEED + 11)
    a, same = runtime.Arena(wl, stream=stream), runtime.Arena(wl)
    for r in range(6):
        a.run_round_fused(r), same.run_round_fused(r)
    if watched:
        a.h.stats_read()
    a.h.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        a.h.stats_enqueue(1)
    for r in range(6, 18):
        a.run_round_fused(r), same.run_round_fused(r)
        if watched_at_replay:
            a.h.stats_read()
    graph.replay()
    torch.cuda.synchronize()
    same.h.stats_enqueue(1)
    got, want = a.h.stats_read(), same.h.stats_read()
    assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1])
    a.h.synchronize()
    del graph
    a.close()
    same.close()
