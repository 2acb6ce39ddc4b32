"""Batches whose block-size classes run side by side (asserted by teuk_get_tiling): the results
of each instance alone, bit for bit, a wait that gives up while another class runs beside it,
and room on the GPU for every class at once."""
import time

import numpy as np
import pytest

from paper_1001_3631_gb300 import TeukError, TeukSolver, inputs

pytestmark = pytest.mark.gpu


def params_of(nr, nth, m, prec):
    return dict(s=-2, m=m, a=0.8, rstar_min=-10.0, rstar_max=30.0, n_rstar=nr, n_theta=nth, rstar_ext=14.0,
                dt_rule=1, courant=0.5, prec=prec, wave_capacity=64)


def problems(shape, prec):
    return [params_of(nr, nth, 1 + k, prec) for k, (nr, nth) in enumerate(shape)]


def start(s, k, p, moving, instance):
    if moving:
        dt = s.time(instance)[1]
        s.set_trajectory(inputs.eccentric_trajectory(80, dt, semi_latus=7.0, ecc=0.3, incl=0.4, chi0=0.3 * k),
                         instance=instance)
    else:
        s.set_source(7.5 + 0.25 * k, instance=instance)
    s.set_state(inputs.smooth_state(p["n_theta"], p["n_rstar"], seed=k), k, instance=instance)


# two, three and four classes of 1 to 10 warps; a fraction of a column a place up to some 40
SHAPES = [((120, 20), (150, 50), (90, 70)), ((1750, 300), (2152, 96), (2366, 96)),
          ((1500, 32), (700, 32), (2200, 64)), ((3000, 128), (3000, 192), (6000, 64)),
          ((9000, 20), (5600, 33), (7000, 100))]


@pytest.mark.parametrize("moving", [False, True])
@pytest.mark.parametrize("prec", ["fp64", "fp64_df", "fp32_kahan", "fp32"])
@pytest.mark.parametrize("shape", SHAPES)
def test_classes_side_by_side_equal_instances_alone(shape, prec, moving):
    ps = problems(shape, prec)
    with TeukSolver(ps) as s:
        for k, p in enumerate(ps):
            start(s, k, p, moving and k != 1, k)
        assert all(s.tiling(k)["side_by_side"] for k in range(len(ps)))
        for n in (7, 1, 4):
            s.step(n)
        got = [(s.get_state(k), s.extract(instance=k)[0]) for k in range(len(ps))]
        s.sync()
    for k, p in enumerate(ps):
        with TeukSolver(p) as s:
            start(s, k, p, moving and k != 1, 0)
            s.step(12)
            assert np.array_equal(got[k][0], s.get_state()) and np.array_equal(got[k][1], s.extract()[0]), k


def test_a_wait_that_gives_up_beside_another_class():
    # an item number that only the larger class has: its neighbours' waits run out, the other
    # class stops as well, and the context is usable after a reset
    ps = problems(((9000, 64), (600, 32)), "fp32_kahan")
    with TeukSolver(ps) as s:
        t = [s.tiling(k) for k in range(2)]
        assert t[0]["side_by_side"] and t[0]["pieces"] > t[1]["pieces"]
        s.set_fault_injection(skip_release_item=t[1]["pieces"], spin_limit=20000)
        s.step(6)
        with pytest.raises(TeukError) as e:
            s.sync()
        assert e.value.status == 5   # TEUK_ETIMEOUT
        s.set_fault_injection(-1, 0)
        for k, p in enumerate(ps):
            start(s, k, p, False, k)
        s.step(6)
        s.sync()
        got = [s.get_state(k) for k in range(2)]
    for k, p in enumerate(ps):
        with TeukSolver(p) as s:
            start(s, k, p, False, 0)
            s.step(6)
            assert np.array_equal(got[k], s.get_state()), k


def step_time(ps, n):
    with TeukSolver(ps) as s:
        for k in range(len(ps)):
            s.set_source(8.0, instance=k)
        s.step(n)
        s.sync()
        best = np.inf
        for _ in range(8):
            t = time.perf_counter()
            s.step(n)
            s.sync()
            best = min(best, time.perf_counter() - t)
        return best


# side by side the classes take less than one after the other (0.83 to 0.95 of it on these);
# without room for all of them at once they took 1.3 to 1.6 times as long
@pytest.mark.parametrize("prec,shape", [("fp32_kahan", ((12000, 32), (12000, 64), (12000, 32))),
                                        ("fp64", ((856, 128), (1563, 160), (794, 128), (2732, 160)))])
def test_every_class_finds_its_places(prec, shape):
    ps = problems(shape, prec)
    rows = sorted({p["n_theta"] for p in ps})
    with TeukSolver(ps) as s:
        assert s.tiling()["side_by_side"]
    apart = sum(step_time([p for p in ps if p["n_theta"] == r], 40) for r in rows)
    assert step_time(ps, 40) <= 1.15 * apart
