"""The order of the statistics' sums is that of a launch of one round in a batch of any length of the same form of the
kernel: the results are the same bit for bit, also where the order decides them.

A row's squares are 2^53 + 2^29, halfway between two neighbours in fp32, in its first tile, and ones far apart.  In 64
bits a one is lost beside the large sum and two of them are not, so the row's norm in fp32 shows whether ones met
before they came to it."""
import numpy as np
import pytest
import torch

from gpu_common import require_gpu
from paper_2111_08274_b200 import runtime, workloads
from paper_2111_08274_b200.workloads import Workload

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


def check_order(n, P, ones, rounds):
    wl = Workload("order", n, P, 1, 1, "fixed", (0,) * n, seed=workloads.BASE_SEED + P)
    a = runtime.Arena(wl)
    a.w.zero_()
    a.w[:, 0:32:8] = torch.tensor([2.0 ** 26, 2.0 ** 26, 2.0 ** 14, 2.0 ** 14], device=a.device)
    for c in ones:
        a.w[:, c] = 1.0
    torch.cuda.synchronize()
    a.run_round_fused(0)
    single, _ = a.h.stats_read()
    assert np.isin(single, [2.0 ** 53, 2.0 ** 53 + 2.0 ** 30]).all()
    for several in rounds:
        a.run_rounds_fused(1, several)
        for back in range(several):
            assert np.array_equal(a.h.stats_read_round(back)[0], single), (several, back)
    a.h.debug_check()
    a.close()


@pytest.mark.parametrize("blocks", [(32, 64), (128, 160), (33, 129), (256, 128), (256, 288), (1, 300)])
def test_row_walk(blocks):
    """24 devices, 2 groups of blocks and a bit, 3, and 4: one round is finished in one level, several in two."""
    for n_blocks in (257, 301, 384, 512):
        check_order(24, 2048 * n_blocks - 3, [2048 * b + 8 * i for i, b in enumerate(blocks) if b < n_blocks], (2, 3))


@pytest.mark.parametrize("tiles", [(64, 256), (1, 2), (2, 3), (3, 4), (5, 131), (63, 65), (128, 130), (37, 101)])
@pytest.mark.parametrize("n,P", [(1, 37_889), (1, 131_072), (2, 30_001), (2, 100_001), (2, 131_071), (3, 37_888), (3, 113_663), (4, 30_000),
                                 (4, 37_889), (4, 100_000), (4, 131_072), (5, 113_664), (5, 113_665), (7, 70_001), (8, 37_889), (8, 75_776),
                                 (8, 75_777), (8, 131_072), (16, 37_888), (16, 131_072), (24, 87_381), (32, 65_536)])
def test_warp_per_row(n, P, tiles):
    """One to four tiles per block in a batch, where one round has eight, four, two or one: the most that an SM takes in
    one block, one tile more, and in between.  Beyond that, the same blocks in both, up to 512, with a finish in one
    level for one round and in two for several."""
    check_order(n, P, [min(256 * t + 8, P - 1) for t in tiles], (2, 5, 8))
