"""lbm_launches counts the launches that are issued, lbm_kernel_launches the
level kernels they carry."""
import pytest

from paper_1601_06984_gb300 import workloads as W

pytestmark = pytest.mark.gpu


# two-level LINEAR step without interior bricks on the coarse level: launched
# level by level GFF, GFC, coarse bricks, coarse list, fine interior, fine
# boundary bricks, GFC, fine interior, fine boundary bricks; batched by instant
# GFF, GFC, interior, rest and GFC, interior, rest
@pytest.mark.parametrize("timing,launches", [(1, 9), (0, 7)])
@pytest.mark.parametrize("precision", [0, 1, 2])
def test_launches_of_a_two_level_step(precision, timing, launches):
    from paper_1601_06984_gb300 import lbm
    m = W.config_tgv2d()
    s = lbm.Sim(m, 9, 1.6, precision=precision)
    s.init(*W.tgv_fields(m, 0.01))
    s.timing_enable(timing)
    s.step(1)  # forms the source records of the initial state too
    n, k = s.launches(), s.kernel_launches()
    s.step(5)
    assert s.launches() - n == 5 * launches
    assert s.kernel_launches() - k == 5 * 10  # one more: the GFF fill's records
    n, k = s.launches(), s.kernel_launches()
    s.reduce()
    assert s.launches() - n == 2 and s.kernel_launches() - k == 3
