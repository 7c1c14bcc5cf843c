"""The last-block finish of the statistics and of the fused round at the sizes where its loops change
shape: block counts around the group size (128 blocks), around a warp's stride over the partial sums
(32 lanes x 4 loads), one block, and more than one group; a launch with one round and one with several;
finished by one block and in two levels.
The sums must match a double-precision sum over the arena as it stands afterwards.  Bounds, all terms being
positive: in the fused round a term is rounded at most 8 times in a thread's pack (each square is fused to the
sum) and once across a pair of lanes, in the statistics kernel 16 times in a thread's chunk of 4 packs of 4;
the rest is in fp64, and the output is rounded once more."""
import numpy as np
import pytest
import torch

from gpu_common import require_gpu
from paper_2111_08274_b200 import runtime, workloads
from paper_2111_08274_b200.workloads import Workload

pytestmark = pytest.mark.gpu
ROUND, STATS = 10 * 2.0 ** -24, 17 * 2.0 ** -24


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


def sums(arena, ref):
    w = arena.w[:, : arena.wl.n_params].double()
    return (w * w).sum(1).cpu().numpy(), ((w - w[ref]) ** 2).sum(1).cpu().numpy()


def check(got, want, bound):
    assert np.allclose(got[0], want[0], rtol=bound, atol=0)
    # distances are sums over fp32 differences, each rounded once more before it is squared
    assert np.allclose(got[1], want[1], rtol=bound + 2.0 ** -23, atol=0)


@pytest.mark.parametrize("blocks", [1, 2, 31, 32, 33, 127, 128, 129, 255, 257, 300])
@pytest.mark.parametrize("n,k,extra", [(2, 1, 0), (3, 2, 1), (17, 16, -1)])
def test_sums_over_block_counts(blocks, n, k, extra):
    wl = Workload("fin", n, 2048 * blocks + extra, k, 1, "fixed", (1,) * n, grad_std=1e-2,
                  seed=workloads.BASE_SEED + blocks)
    arena = runtime.Arena(wl)
    sel = arena.run_round_fused(0)                       # a launch of one round
    check(arena.h.stats_read(), sums(arena, int(sel[0])), ROUND)
    sel = arena.run_rounds_fused(1, 3)[-1]               # a launch of three
    check(arena.h.stats_read(), sums(arena, int(sel[0])), ROUND)
    ref = n - 1
    check(arena.h.stats(ref), sums(arena, ref), STATS)          # the statistics kernel
    arena.close()


@pytest.mark.parametrize("blocks,rounds", [(481, 1), (482, 1), (160, 3), (161, 3)])
def test_one_group_and_several(blocks, rounds):
    """17 devices, odd numbers of blocks and values: finished by one block (160 and 161 blocks, whatever the rounds; 481 and
    482 with the 34 values of one round)."""
    wl = Workload("fin", 17, 2048 * blocks - 1, 5, 1, "fixed", (1,) * 17, grad_std=1e-2, seed=workloads.BASE_SEED + blocks)
    arena = runtime.Arena(wl)
    for first in (0, rounds):                            # the tickets are back at zero for the second launch
        sel = arena.run_rounds_fused(first, rounds)[-1]
        check(arena.h.stats_read(), sums(arena, int(sel[0])), ROUND)
    arena.close()


@pytest.mark.parametrize("n,blocks,rounds", [(2, 512, 1), (2, 513, 1), (16, 512, 1), (17, 257, 1), (24, 256, 2), (24, 257, 2),
                                             (24, 383, 2), (24, 384, 2), (24, 385, 2), (32, 512, 1), (32, 513, 1), (1, 1024, 1), (1, 1025, 1)])
def test_one_level_and_two(n, blocks, rounds):
    """Both sides of the lines between a finish by one block and one in two levels: 256 blocks, 512 blocks, and the number
    of values in between; in two levels with a last group of 128 blocks, of fewer and of one."""
    wl = Workload("fin", n, 2048 * blocks - 1, max(1, n // 4), 1, "fixed", tuple(1 + i % 2 for i in range(n)), grad_std=1e-2,
                  seed=workloads.BASE_SEED + blocks)
    arena = runtime.Arena(wl)
    for first in (0, rounds):                            # the tickets are back at zero for the second launch
        sel = arena.run_rounds_fused(first, rounds)[-1]
        check(arena.h.stats_read(), sums(arena, int(sel[0])), ROUND)
    arena.h.debug_check()
    arena.close()
