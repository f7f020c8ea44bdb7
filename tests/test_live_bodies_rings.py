"""Bodies and batches of one format whose rings differ, alive at once: what one
plans leaves the others' launches as they were."""
import numpy as np
import pytest

from paper_2208_13769_gb300 import lbm
from paper_2208_13769_gb300 import workloads as W

pytestmark = [pytest.mark.gpu, pytest.mark.auto_plan]


def _prob(lam=0.3):
    return W.smooth_random(300, 200, W.clamped_free_edges(), seed=3, amp=0.01, lam=lam, mu=0.3)


@pytest.mark.parametrize("storage,carry,scheme", [
    ("f64", None, 1), ("f32", False, 1), ("f32", True, 0), ("f32", "lo16", 1), ("f16", None, 1), ("bf16", None, 1),
    ("f64", None, 2), ("f32", True, 2), ("f16", None, 2)])
def test_bodies_of_different_rings_step_by_turns(storage, carry, scheme):
    """A deep ring's launches go on after a body with a shallower one is planned."""
    bodies = [lbm.Body(_prob(), storage=storage, compensated=carry, scheme=scheme, tuning=lbm.lbm_tuning(r, 0, 0, 2))
              for r in (8, 4, 6)]
    try:
        for n in (3, 1, 2):
            for b in bodies:
                b.step(n)
        got = [b.read() for b in bodies]
    finally:
        for b in bodies:
            b.close()
    for other in got[1:]:
        for k in ("u", "v", "P", "r"):
            assert np.array_equal(other[k], got[0][k]), k


def test_batches_of_different_rings_step_by_turns():
    bodies = [lbm.Body(_prob(), storage="f64") for _ in range(3)]
    try:
        with lbm.Batch(bodies[:1], tuning=lbm.lbm_tuning(8, 0, -1, 0)) as a, \
                lbm.Batch(bodies[1:2], tuning=lbm.lbm_tuning(4, 0, -1, 0)) as b, \
                lbm.Batch(bodies[2:], tuning=lbm.lbm_tuning(6, 0, -1, 0)) as c:
            for n in (3, 1, 2):
                for batch in (a, b, c):
                    batch.step(n)
        got = [b.read() for b in bodies]
    finally:
        for b in bodies:
            b.close()
    for other in got[1:]:
        for k in ("u", "v", "P", "r"):
            assert np.array_equal(other[k], got[0][k]), k
