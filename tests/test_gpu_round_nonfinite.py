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


# devices, parameters, rounds per call: row walk; a warp per row, alone and in a batch; rows on the SM, in a small
# arena and with all and with a part of the rows of a large one
FORMS = {"walk": (4, 140_001, 1), "rows": (4, 1_001, 1), "rows_batch": (4, 1_001, 3), "on_sm_small": (3, 1_500_007, 2),
         "on_sm_all": (4, 9_400_003, 3), "on_sm_part": (16, 2_350_003, 2)}


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
