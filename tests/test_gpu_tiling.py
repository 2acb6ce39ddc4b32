"""The cut of the columns that is in effect (teuk_get_tiling): a strip length that is set is
kept whatever its value."""
import pytest

from paper_1001_3631_gb300 import TeukSolver

pytestmark = pytest.mark.gpu


def params_of(nr, nth, prec):
    return dict(s=-2, m=2, a=0.8, rstar_min=-10.0, rstar_max=30.0, n_rstar=nr, n_theta=nth, rstar_ext=14.0,
                dt_rule=1, courant=0.5, prec=prec)


# the automatic cut is not uniform strips of one wave on any of these
@pytest.mark.parametrize("nr,nth,prec", [(800, 64, "fp64"), (5001, 100, "fp64_df"), (5001, 100, "fp32_kahan"),
                                         (3001, 300, "fp32")])
def test_a_strip_that_is_set_is_kept(nr, nth, prec):
    with TeukSolver(params_of(nr, nth, prec)) as s:
        auto = s.tiling()
        assert auto["automatic"] and 1 <= auto["columns"] <= nr - 2
        for strip in range(1, auto["columns"] + 3):
            pieces = -(-(nr - 2) // strip)
            for put in (lambda v: s.set_tiling(v, 1), lambda v: s.set_instance_tiling(0, v)):
                put(strip)
                t = s.tiling()
                assert (t["automatic"], t["pieces"]) == (False, pieces), (strip, t)
                put(0)
                assert s.tiling() == auto
