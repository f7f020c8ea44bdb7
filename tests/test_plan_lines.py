"""Default plans where the rules that pick them change, against other
decompositions: the same bits in FP32 (FP64 to rounding, 5e-13).  FP32 pairs with
20 rows or more a wave (shorter tiles after it) and, with a hole, without; the
extrapolated scheme with the deeper ring in one and in several waves, below its
line and with a hole; FP64 by its own kernel's occupancy; plan 2 on a body without
seams."""
import dataclasses

import numpy as np
import pytest

from paper_2208_13769_gb300 import lbm
from paper_2208_13769_gb300 import workloads as W
from parity_util import rel_l2

pytestmark = [pytest.mark.gpu, pytest.mark.auto_plan]

KEYS = ("u", "v", "P", "r")


def _read(prob, steps, storage, carry, scheme, tuning=None):
    with lbm.Body(prob, storage=storage, compensated=carry, scheme=scheme, tuning=tuning) as b:
        b.step(steps)
        return b.read(lbm.LBM_FIELD_U | lbm.LBM_FIELD_V | lbm.LBM_FIELD_P | lbm.LBM_FIELD_R)


@pytest.mark.parametrize("nx,ny,storage,carry,scheme,hole", [
    (4000, 560, "f32", True, 1, None), (4000, 470, "f32", True, 0, None), (2100, 1300, "f32", True, 1, (900, 1201, 500, 777)),
    (1000, 830, "f32", True, 2, None), (990, 790, "f32", True, 2, None), (4000, 560, "f32", True, 2, None),
    (1301, 2803, "f32", True, 2, None), (1400, 1000, "f32", True, 2, (500, 901, 300, 700)),
    (900, 611, "f64", None, 2, None)])
def test_default_plans_match_other_decompositions(nx, ny, storage, carry, scheme, hole):
    prob = W.smooth_random(nx, ny, W.clamped_free_edges(), seed=7, amp=0.01, lam=0.3, mu=0.3)
    if hole:
        prob = dataclasses.replace(prob, hole=hole)
    got = _read(prob, 9, storage, carry, scheme)
    for tuning in (lbm.lbm_tuning(0, 0, -1, 2), lbm.lbm_tuning(4, 16, 0, 0), lbm.lbm_tuning(6, 48, 2, 0),
                   lbm.lbm_tuning(0, 0, -1, 1)):
        ref = _read(prob, 9, storage, carry, scheme, tuning)
        for k in KEYS:
            if storage == "f64":
                assert rel_l2(got[k], ref[k]) <= 5e-13, k
            else:
                assert np.array_equal(got[k], ref[k]), k
