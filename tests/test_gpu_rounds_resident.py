"""Batches of rounds whose replicas stay on the SMs (shared memory and tensor memory) against the same rounds
launched one by one, bit for bit: arenas beyond the L2 with all rows on the SM (few devices), with part of
them (16 devices and more), light and heavy steps, every storage, ragged ends, odd numbers of rounds,
global synchronisation by overwriting and by mixing, devices that run no steps, one and all devices
selected; small arenas of at most 8 devices, which take the form as well; and vectors of more chunks than a
launch has blocks.  The statistics of every round of every launch are compared, those of synchronised rounds
and of rounds inside a batch among them: their fp64 sums are added in another order, and the output is one
fp32 rounding of them."""
import numpy as np
import pytest
import torch

from gpu_common import require_gpu
from paper_2111_08274_b200 import binding, runtime, workloads
from paper_2111_08274_b200.workloads import Workload

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


STORAGE = {"fp32": (0, 0, 0, 8), "bf16": (1, 0, 0, 6), "bf16_m16": (1, 1, 0, 4), "bf16_m16_sr": (1, 1, 1, 4)}


def compare(n, P, k, steps, storage, beta, batches, launches):
    dtype, m_dtype, rounding, _ = STORAGE[storage]
    rounds = sum(batches)
    wl = Workload("res", n, P, k, rounds, "fixed", steps, grad_std=1e-2, dtype=dtype, m_dtype=m_dtype, rounding=rounding,
                  sync_every=3, sync_beta=beta, seed=workloads.BASE_SEED + P + n)
    batch, single = runtime.Arena(wl), runtime.Arena(wl)
    single.h.set_round_batch(1)
    for a in (batch, single):                     # what lies behind the vector must stay as it is
        a.w[:, P:] = 3.0
        a.m[:, P:] = 5.0
    before, first = batch.h.launch_count(), 0
    for count in batches:
        got = batch.run_rounds_fused(first, count)
        stats = []
        for r in range(first, first + count):
            want = single.run_rounds_fused(r, 1)
            assert np.array_equal(got[r - first], want[0])
            stats.append(single.h.stats_read())
        one_launch = launches == len(batches)
        for back in range(count if one_launch else 1):
            a, b = batch.h.stats_read_round(back), stats[count - 1 - back]
            assert np.allclose(a[0], b[0], rtol=2.0 ** -23, atol=0) and np.allclose(a[1], b[1], rtol=2.0 ** -23, atol=0)
        first += count
    assert batch.h.launch_count() - before == launches
    torch.cuda.synchronize()
    assert torch.equal(batch.w, single.w) and torch.equal(batch.m, single.m)
    va, vb = batch.h.get_versions(), single.h.get_versions()
    assert np.array_equal(va[0], vb[0]) and np.array_equal(va[1], vb[1])
    batch.h.debug_check()
    batch.close()
    single.close()


@pytest.mark.parametrize("storage", sorted(STORAGE))
@pytest.mark.parametrize("n,k,hi", [(2, 1, 2), (5, 5, 2), (8, 4, 2), (8, 3, 7), (13, 2, 2), (16, 4, 2), (16, 16, 5), (24, 3, 2),
                                    (32, 8, 2)])
def test_large_arenas(n, k, hi, storage):
    rounding = STORAGE[storage][2]
    P = 150_000_001 // (n * STORAGE[storage][3]) // 1024 * 1024 + {2: 1, 5: 1023, 8: 8, 13: 519}.get(n, 0)
    steps = tuple(i % (hi + 1) for i in range(n))
    compare(n, P, k, steps, storage, 0.25 if n % 2 else 1.0, (8, 7),
            15 if rounding and n > 16 else 2)   # stochastic rounding with many devices: one by one


@pytest.mark.parametrize("storage", ["fp32", "bf16"])
def test_two_steps_of_24_devices(storage):
    compare(24, 150_000_001 // (24 * STORAGE[storage][3]), 5, (2,) * 24, storage, 0.5, (8, 6), 2)


@pytest.mark.parametrize("n,P,k", [(8, 524_289, 4), (3, 1_500_007, 2), (1, 4_200_001, 1), (8, 1_048_576, 8)])
@pytest.mark.parametrize("hi", [1, 6])
def test_small_arenas(n, P, k, hi):
    compare(n, P, k, tuple(i % (hi + 1) for i in range(n)), "fp32", 0.5, (2, 7), 2)


@pytest.mark.parametrize("n,k,beta", [(2, 1, 1.0), (3, 2, 0.25)])
def test_more_chunks_than_blocks(n, k, beta):
    """16,384 blocks and chunks of 1024 parameters: each block has a second chunk, a few a third."""
    compare(n, 2 * 16_384 * 1024 + 5_003, k, tuple(1 + i % 2 for i in range(n)), "bf16_m16", beta, (3,), 1)


@pytest.mark.parametrize("n,storage,per_round,launches", [
    (16, "fp32", (8, 8), [1, 1]), (16, "fp32", (8,) * 8, [1] * 8), (16, "fp32", (1, 1, 8), [2, 1]),
    (16, "fp32", (8, 1, 1, 1, 8), [1, 3, 1]), (16, "fp32", (1, 1, 5), [2, 1]), (16, "fp32", (1, 1, 5, 2), [4]),
    (16, "fp32", (4, 3, 4, 4, 3, 4), [6]), (6, "fp32", (8, 8), [1, 1]), (6, "fp32", (8, 8, 8), [3]), (8, "fp32", (3, 3), [2]),
    (16, "bf16", (8, 8), [1, 1]), (16, "bf16", (8, 8, 8), [3]), (14, "bf16", (8, 8), [2]),
    (16, "bf16_m16_sr", (2, 2, 2, 2), [1] * 4), (16, "bf16_m16_sr", (1, 1), [2]), (14, "bf16_m16_sr", (8, 8, 8), [3])])
def test_rounds_that_do_not_gain_are_launched_apart(n, storage, per_round, launches):
    dtype, m_dtype, rounding, width = STORAGE[storage]
    wl = Workload("apart", n, 166_000_000 // (n * width), 3, 1, "fixed", (1,) * n, grad_std=1e-2, dtype=dtype,
                  m_dtype=m_dtype, rounding=rounding, seed=workloads.BASE_SEED + n)
    batch, single = runtime.Arena(wl), runtime.Arena(wl)
    steps = np.repeat(np.array(per_round, dtype=np.int32)[:, None], n, axis=1)
    before = batch.h.launch_count()
    got = batch.h.rounds(0, steps, wl.lr, wl.k, batch.select_seed, 2)
    assert batch.h.launch_count() - before == len(launches)
    stats = []
    for r in range(len(steps)):
        want = single.h.round(single.ids, steps[r], wl.lr, r, wl.k, single.select_seed, sync_all=r % 2 == 1)
        assert np.array_equal(got[r], want)
        stats.append(single.h.stats_read())
    torch.cuda.synchronize()
    assert torch.equal(batch.w, single.w) and torch.equal(batch.m, single.m)
    assert all(np.array_equal(x, y) for x, y in zip(batch.h.get_versions(), single.h.get_versions()))
    for back in range(launches[-1]):
        for x, y in zip(batch.h.stats_read_round(back), stats[-1 - back]):
            assert np.allclose(x, y, rtol=2.0 ** -23, atol=0)
    with pytest.raises(binding.HadflError):
        batch.h.stats_read_round(launches[-1])
    batch.h.debug_check()
    batch.close()
    single.close()


@pytest.mark.parametrize("n,k,steps,beta", [(16, 1, (0, 1), 1.0), (16, 1, (0, 1), 0.5), (16, 16, (1,), 1.0), (19, 2, (2, 0), 0.25),
                                            (32, 3, (1,), 1.0)])
def test_one_visit_per_row(n, k, steps, beta):
    """fp32, a part of the rows on the SM, fewer than two steps per device: a single selected device without steps,
    all selected, several steps beside none, overwritten and mixed rounds."""
    compare(n, 150_000_001 // (n * 8) + 3, k, tuple(steps[i % len(steps)] for i in range(n)), "fp32", beta, (8, 5), 2)


@pytest.mark.parametrize("n", [9, 10, 12, 13, 16])
@pytest.mark.parametrize("steps", [(1,), (1, 1, 1, 2), (1, 2), (1, 2, 2, 2), (2,)])
def test_one_visit_or_visits_apart(n, steps):
    """Both sides of the lines between one visit per row and visits apart: 9, 10 to 12, and 13 devices; 1.25 and 2 steps per
    device; in two rounds, where six blocks share an SM, and in three."""
    compare(n, 150_000_001 // (n * 8) + 3, 2, tuple(steps[i % len(steps)] for i in range(n)), "fp32", 0.5, (2, 3), 2)
