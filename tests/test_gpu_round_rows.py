"""The fused round's form for small vectors (a warp per row) at the sizes where it can go wrong: tiles of 256
columns with and without a ragged end, one row to 32, one or several tiles per block, the ends of the
range that the library takes it for (2^17 parameters in a launch of one round, 2^22 device-parameters in
a launch of several), all rows selected, odd and even numbers of rounds per launch.  Parameters and
momentum bit for bit against the separate calls; statistics against double-precision sums (bound as for
the finish: 16 values per lane pair, then trees of 5 levels, all positive)."""
import numpy as np
import pytest
import torch

from gpu_common import require_gpu
from paper_2111_08274_b200 import runtime, workloads
from paper_2111_08274_b200.workloads import Workload

pytestmark = pytest.mark.gpu
BOUND = 18 * 2.0 ** -24


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
