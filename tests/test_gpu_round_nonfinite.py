"""Rounds over models that hold infinities and NaNs, in each form of the fused kernel (row walk, a warp per row,
rows on the SM).

Statistics: a selected device holds the aggregate and is at distance 0 whatever its values; a device that a
global synchronisation overwrites is at the sum over (w - w_ref)^2 with w = w_ref, which is 0, or NaN where
the aggregate is not finite."""
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


# devices, parameters, rounds per call: row walk; a warp per row, alone and in a batch, in blocks of up to 512 threads and
# of more; rows on the SM, in a small arena and with all and with a part of the rows of a large one (with fp32 parameters
# 16 devices take one visit per row, 9 visits apart)
FORMS = {"walk": (4, 140_001, 1), "rows": (4, 1_001, 1), "rows_batch": (4, 1_001, 3), "rows_large": (32, 1_001, 1),
         "rows_large_batch": (32, 1_001, 3), "on_sm_small": (3, 1_500_007, 2), "on_sm_all": (4, 9_400_003, 3),
         "on_sm_part": (16, 2_350_003, 2), "on_sm_part_apart": (9, 4_200_003, 3)}


def arena(n, P, storage, sync_every):
    dtype, m_dtype = storage
    wl = Workload("inf", n, P, 2, 1, "fixed", (0,) * n, dtype=dtype, m_dtype=m_dtype, sync_every=sync_every,
                  seed=workloads.BASE_SEED + P)
    a = runtime.Arena(wl)
    a.h.set_available([1, 1] + [0] * (n - 2))     # devices 0 and 1 are the selected ones
    return a


@pytest.mark.parametrize("storage", [(0, 0), (1, 1)])
@pytest.mark.parametrize("bad", [np.inf, np.nan])
@pytest.mark.parametrize("sync_every", [0, 1])
@pytest.mark.parametrize("form", sorted(FORMS))
def test_statistics(form, sync_every, bad, storage):
    n, P, rounds = FORMS[form]
    a = arena(n, P, storage, sync_every)
    a.h.write_params(1, np.array([1.0, bad], dtype=np.float32))
    sel = a.run_rounds_fused(0, rounds)
    assert sorted(sel[0]) == [0, 1]
    for back in range(min(rounds, 2)):
        n2, d2 = a.h.stats_read_round(back)
        assert (d2[:2] == 0.0).all()
        assert not np.isfinite(n2[:2]).any()
        assert (np.isnan(d2[2:]) if sync_every or np.isnan(bad) else np.isposinf(d2[2:])).all()
        assert np.isfinite(n2[2:]).all() != bool(sync_every)
    a.h.debug_check()
    a.close()


@pytest.mark.parametrize("storage", [(0, 0), (1, 0), (1, 1)])
@pytest.mark.parametrize("form", sorted(FORMS))
def test_untouched_values_keep_their_bits(form, storage):
    """NaNs with a payload, and signalling ones, in the parameters and the momentum of devices that run no steps
    and receive nothing: of the unselected ones, and of the selected one where it is the only one."""
    n, P, rounds = FORMS[form]
    wl = Workload("bits", n, P, 1, 1, "fixed", (0,) * n, dtype=storage[0], m_dtype=storage[1],
                  seed=workloads.BASE_SEED + P)
    a = runtime.Arena(wl)
    bits = {4: [0x7FC12345, -0x003EDCBB, 0x7F812345, -0x80000000, 1], 2: [0x7FC5, -0x0035, 0x7F85, -0x8000, 1]}
    whole = []
    for t in (a.w, a.m):
        t = t.view(torch.int32 if t.element_size() == 4 else torch.int16)
        t[:, :5] = torch.tensor(bits[t.element_size()], dtype=t.dtype, device="cuda")
        t[:, P - 1] = t[:, 0]
        whole.append((t, t.clone()))
    torch.cuda.synchronize()
    a.run_rounds_fused(0, rounds)
    torch.cuda.synchronize()
    for now, before in whole:
        assert torch.equal(now, before)
    a.h.debug_check()
    a.close()
