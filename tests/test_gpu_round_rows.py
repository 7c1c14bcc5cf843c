"""The fused round's form for small vectors (a warp per row) at the sizes where it can go wrong: tiles of 256
columns with and without a ragged end, one row to 32, one or several tiles per block, the ends of the
range that the library takes it for (2^17 parameters in a launch of one round, 2^22 device-parameters in
a launch of several), all rows selected, odd and even numbers of rounds per launch.  Parameters and
momentum bit for bit against the separate calls; statistics against double-precision sums.  Bound: a square
and the additions to it are rounded at most 8 times in a thread's pack (fused) and once across the lanes l and
l ^ 16, all terms positive, the rest is in fp64, and the output is rounded: 10 * 2^-24."""
import numpy as np
import pytest
import torch

from gpu_common import require_gpu
from paper_2111_08274_b200 import runtime, workloads
from paper_2111_08274_b200.workloads import Workload

pytestmark = pytest.mark.gpu
BOUND = 10 * 2.0 ** -24


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


STORAGE = [(0, 0, 0), (1, 0, 0), (1, 1, 1)]
SIZES = [(1, 1, 1), (1, 257, 1), (2, 255, 2), (3, 256, 1), (5, 4_097, 5), (7, 2_305, 3), (8, 131_072, 4), (9, 131_071, 2),
         (16, 131_072, 4), (16, 131_073, 16), (31, 511, 31), (32, 65_537, 3), (32, 131_072, 32), (32, 131_073, 1)]


@pytest.mark.parametrize("dtype,m_dtype,rounding", STORAGE)
@pytest.mark.parametrize("n,P,k", SIZES)
def test_rows_form_against_the_separate_calls(n, P, k, dtype, m_dtype, rounding):
    beta = 0.25 if n % 2 else 1.0
    wl = Workload("rows", n, P, k, 12, "fixed", tuple((3 * i + 1) % 4 for i in range(n)), grad_std=1e-2, dtype=dtype,
                  m_dtype=m_dtype, rounding=rounding, sync_every=3, sync_beta=beta, seed=workloads.BASE_SEED + P + n)
    fused, plain = runtime.Arena(wl), runtime.Arena(wl)
    for a in (fused, plain):                      # what lies behind the vector must stay as it is
        a.w[:, P:] = 3.0
        a.m[:, P:] = 5.0
    want = np.stack([plain.run_round(r) for r in range(12)])
    got = np.concatenate([fused.run_rounds_fused(0, 8), fused.run_rounds_fused(8, 3), fused.run_rounds_fused(11, 1)])
    assert np.array_equal(got, want)
    torch.cuda.synchronize()
    assert torch.equal(fused.w, plain.w) and torch.equal(fused.m, plain.m)
    n2, d2 = fused.h.stats_read()
    w = fused.w[:, :P].double()
    assert np.allclose(n2, (w * w).sum(1).cpu().numpy(), rtol=BOUND, atol=0)
    assert np.allclose(d2, ((w - w[int(want[-1][0])]) ** 2).sum(1).cpu().numpy(), rtol=BOUND + 2.0 ** -23, atol=0)
    fused.h.debug_check()
    fused.close()
    plain.close()


@pytest.mark.parametrize("rounds", [1, 3])
def test_row_sums_beyond_a_lane_pair_are_in_64_bits(rounds):
    """One square of 1 and, in other lanes of the same half-warp, squares that add up to just under half a unit in
    the last place of 1 at each level of a tree over the lanes: a tree in fp32 loses all four (2^-22), sums in
    64 bits none.  Bound: the output's rounding, and that of the squares, 2^-24 each."""
    wl = Workload("lanes", 2, 256, 1, 1, "fixed", (0, 0), seed=workloads.BASE_SEED)
    a = runtime.Arena(wl)
    a.h.set_available([1, 0])
    half = 0.49 * 2.0 ** -23
    v = np.zeros(256)
    v[0] = 1.0
    for lanes in ((8,), (4, 12), (2, 6, 10, 14), (1, 3, 5, 7, 9, 11, 13, 15)):
        v[8 * np.array(lanes)] = np.sqrt(half / len(lanes))
    v = v.astype(np.float32)
    a.h.write_params(0, np.zeros(256, dtype=np.float32))
    a.h.write_params(1, v)
    a.run_rounds_fused(0, rounds)
    want = (v.astype(np.float64) ** 2).sum()
    for back in range(rounds):
        n2, d2 = a.h.stats_read_round(back)
        assert abs(n2[1] - want) <= 2.0 ** -23 * want and abs(d2[1] - want) <= 2.0 ** -23 * want
    a.close()


@pytest.mark.parametrize("n,P", [(1, 1), (1, 2049), (3, 1_025), (4, 100_000), (8, 131_072), (32, 65_537), (4, 131_073), (32, 131_072)])
def test_reported_grid_is_that_of_a_single_round(n, P):
    a = runtime.Arena(Workload("grid", n, P, 1, 1, "fixed", (1,) * n))
    rows = P <= 1 << 17 and n * P <= 1 << 21
    columns = 256 * max(8 // n, 1) if rows else 2048
    assert a.h.round_grid() == -(-P // columns)
    a.close()


@pytest.mark.parametrize("dtype,m_dtype,rounding", STORAGE)
@pytest.mark.parametrize("n,per_sm,over", [(1, 8, 0), (1, 8, 1), (2, 8, 0), (2, 8, 1), (3, 5, 0), (3, 5, 1), (4, 1, 0), (4, 1, 1),
                                           (4, 3, 1), (4, 4, 0), (16, 1, 0), (16, 1, 1)])
def test_batches_with_an_sm_per_block(n, per_sm, over, dtype, m_dtype, rounding):
    """Tiles on both sides of what blocks of 16 warps hold with one block on every SM."""
    tiles = per_sm * torch.cuda.get_device_properties(0).multi_processor_count + over
    test_rows_form_against_the_separate_calls(n, 256 * tiles - 3, max(1, n // 3), dtype, m_dtype, rounding)
