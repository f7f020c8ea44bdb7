"""The FP64 reciprocal and quotients that the kernels compute by hand.

The reciprocal: the seed of rcp.approx.ftz.f64 takes the first 20 mantissa bits of
its operand and gives 20 of the result, each an error of up to 2^-20 of the value,
2^-19 together.  One third-order step leaves its cube, 2^-57 of the value, which is
2^-4 units in the last place, and one rounding, 0.5; the roundings within the step
add less than 2^-17.  Hence 0.57 at most.  The quotients of the read-out: a
reciprocal, a product and Markstein's correction, the division where that does not
apply, and so the bits of the division everywhere."""
import pytest

from paper_2208_13769_gb300 import lbm


@pytest.mark.gpu
@pytest.mark.parametrize("seed", [0, 1, 2208, 2 ** 63 + 5])
def test_reciprocal_and_quotients_hold_their_bounds(seed):
    worst, differ = lbm.lbm_selftest_quotients(1 << 27, seed)
    assert 0.49 < worst <= 0.5 + 2.0 ** -4 + 2.0 ** -17
    assert differ == 0


def test_bad_counts_are_refused():
    import ctypes as C
    out = (C.c_double * 2)()
    for n in (0, -1, (1 << 30) + 1):
        assert lbm.lib().lbm_selftest_quotients(n, 1, None, out) == lbm.LBM_E_INVALID
    assert lbm.lib().lbm_selftest_quotients(1, 1, None, None) == lbm.LBM_E_INVALID
