"""The status that a read returns with the fields, for host buffers of either
kind."""
import dataclasses

import numpy as np
import pytest

from paper_2208_13769_gb300 import lbm
from paper_2208_13769_gb300 import workloads as W

pytestmark = [pytest.mark.gpu, pytest.mark.auto_plan]


@pytest.mark.parametrize("first", ["pageable", "pinned"])
def test_unstable_runs_are_reported_into_any_buffer(first):
    """The status comes with the fields, whether the caller's buffer is pinned
    or not, in either order, and goes back to good with a restored state."""
    import torch
    prob = W.smooth_random(90, 50, W.clamped_free_edges(), seed=5, amp=0.01, lam=0.3, mu=0.3)
    wild = dataclasses.replace(prob, make_initial=None, u0=np.where(np.arange(90)[None, :, None] % 4 < 2, 1.5, -1.5) *
                               np.ones((50, 90, 2)), v0=np.zeros((50, 90, 2)))
    n = 2 * 90 * 50
    bufs = {"pageable": np.empty(n), "pinned": torch.empty(n, dtype=torch.float64, pin_memory=True).numpy()}
    order = [first, "pinned" if first == "pageable" else "pageable", first]
    with lbm.Body(prob, storage="f32") as good, lbm.Body(wild, storage="f32") as bad:
        good.step(5)
        bad.step(5)
        ref = good.read(lbm.LBM_FIELD_U)["u"].ravel()
        for k in order:
            assert lbm.lbm_read_fields(good.ctx, lbm.LBM_FIELD_U, bufs[k])[0] == lbm.LBM_OK
            assert np.array_equal(bufs[k], ref), k
            assert lbm.lbm_read_fields(bad.ctx, lbm.LBM_FIELD_U, bufs[k], allow_unstable=True)[0] == lbm.LBM_E_UNSTABLE
        bad.load_state(good.save_state())
        for k in order:
            assert lbm.lbm_read_fields(bad.ctx, lbm.LBM_FIELD_U, bufs[k])[0] == lbm.LBM_OK
            assert np.array_equal(bufs[k], ref), k
