"""Batches of many small bodies, at the rows a wave where the default tiles
change (short tiles below 12, then chunks of about 32 rows), against fixed rows:
the same bits in FP32 and 16-bit arithmetic, FP64 to rounding (5e-13, as for
single bodies' plans)."""
import numpy as np
import pytest

from paper_2208_13769_gb300 import lbm
from paper_2208_13769_gb300 import workloads as W
from parity_util import rel_l2

pytestmark = [pytest.mark.gpu, pytest.mark.auto_plan]


@pytest.mark.parametrize("storage,count", [("f32", 150), ("f32", 260), ("f16", 260), ("f64", 150)])
def test_many_small_members_match_fixed_rows(storage, count):
    P = W.Edge(W.PERIODIC)
    sides = np.random.default_rng(count).integers(12, 131, (count, 2))
    shapes = [(int(x), int(y)) for x, y in sides]
    probs = [W.smooth_random(nx, ny, [P] * 4 if k % 2 else W.clamped_free_edges(), seed=k % 5, amp=0.01, lam=0.3, mu=0.3)
             for k, (nx, ny) in enumerate(shapes)]
    res = []
    for tuning in (None, lbm.lbm_tuning(0, 16, 0, 0)):
        bodies = [lbm.Body(p, storage=storage) for p in probs]
        try:
            with lbm.Batch(bodies, tuning=tuning) as batch:
                batch.step(9)
                batch.sync()
            res.append([b.read(lbm.LBM_FIELD_U | lbm.LBM_FIELD_R) for b in bodies])
        finally:
            for b in bodies:
                b.close()
    for k, (a, b) in enumerate(zip(*res)):
        for f in ("u", "r"):
            if storage == "f64":
                assert rel_l2(a[f], b[f]) <= 5e-13, (shapes[k], f)
            else:
                assert np.array_equal(a[f], b[f]), (shapes[k], f)
