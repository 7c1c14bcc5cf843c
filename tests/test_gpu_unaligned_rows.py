"""Arenas that start at an odd multiple of 16 bytes (rows not at multiples of 32, which the 32-byte stores of
full fp32 packs need) against the same calls on an aligned arena, bit for bit: every kernel that updates
rows, each storage, with full and ragged chunks."""
import numpy as np
import pytest
import torch

from gpu_common import require_gpu
from paper_2111_08274_b200 import binding
from paper_2111_08274_b200.workloads import Workload

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


def arena(wl, shift_w, shift_m):
    """Rows that start `shift` bytes behind a 512-byte boundary, 7.0 around the vectors."""
    stride = (wl.n_params + 7) // 8 * 8 + 8
    out = []
    for dtype, shift in ((wl.dtype, shift_w), (wl.m_dtype, shift_m)):
        t = torch.full((wl.n_devices * stride + 64,), 7.0, dtype=torch.bfloat16 if dtype else torch.float32, device="cuda")
        out.append(t[shift // t.element_size():][: wl.n_devices * stride].view(wl.n_devices, stride))
    torch.cuda.synchronize()
    h = binding.Hadfl.from_workload(wl, w_ptr=out[0].data_ptr(), m_ptr=out[1].data_ptr(), row_stride_elems=stride,
                                    stream=torch.cuda.current_stream().cuda_stream)
    return out[0], out[1], h


# vectors of a few tiles (a warp per row), of one to two chunks and more (row walk), with an arena of at most 64
# MiB and more than eight devices or fewer (row walk or resident batches)
@pytest.mark.parametrize("storage", [(0, 0, 0), (1, 0, 0), (1, 1, 1)])
@pytest.mark.parametrize("n,P", [(3, 2047), (4, 2048), (2, 300_001), (5, 1_048_577), (12, 524_291)])
@pytest.mark.parametrize("shifts", [(16, 16), (0, 16), (16, 0)])
def test_calls_and_rounds(n, P, storage, shifts):
    wl = Workload("odd16", n, P, 2, 1, "fixed", (1,) * n, grad_std=1e-2, dtype=storage[0], m_dtype=storage[1],
                  rounding=storage[2], seed=77 + P)
    ids = np.arange(n, dtype=np.int32)
    got = []
    for sw, sm in (shifts, (0, 0)):
        w, m, h = arena(wl, sw, sm)
        h.local_step(ids, (1 + ids % 3).astype(np.int32), 0.02)
        h.round(ids, (ids % 4).astype(np.int32), 0.02, 0, 2, 5)
        h.rounds(1, np.stack([(ids + r) % 3 for r in range(6)]).astype(np.int32), 0.02, 2, 5, 4)
        stats = h.stats_read()
        h.debug_check()
        got.append((w.clone(), m.clone(), stats))
        h.destroy()
    (wa, ma, sa), (wb, mb, sb) = got
    assert torch.equal(wa, wb) and torch.equal(ma, mb)
    assert np.array_equal(sa[0], sb[0]) and np.array_equal(sa[1], sb[1])
