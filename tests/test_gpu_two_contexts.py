"""Several contexts in one process: what a kernel is allowed belongs to the kernel, so no
context may lower it for another."""
import threading

import numpy as np
import pytest

from paper_1001_3631_gb300 import TeukSolver, inputs

pytestmark = pytest.mark.gpu


def params_of(nr, nth, prec):
    return dict(s=-2, m=2, a=0.7, rstar_min=-10.0, rstar_max=30.0, n_rstar=nr, n_theta=nth, rstar_ext=14.0,
                dt_rule=1, courant=0.5, prec=prec)


@pytest.mark.parametrize("prec", ["fp64", "fp64_df", "fp32_kahan"])
def test_a_shorter_reverse_sweep_beside_a_tall_one(prec):
    # 1024 rows take more shared memory than 576, both in the build for up to 1024 rows
    n, nth = 200, 1024
    gw = np.random.default_rng(3).standard_normal((n, nth, 2))
    stop, errors = threading.Event(), []

    def short():
        try:
            with TeukSolver(dict(params_of(40, 576, prec), wave_capacity=2)) as s:
                s.set_source(8.0)
                while not stop.is_set():
                    s.adjoint(1, step0=0, grad_wave=np.ones((1, 576, 2)))
        except Exception as e:   # noqa: BLE001 (reported by the test)
            errors.append(e)

    with TeukSolver(dict(params_of(24, nth, prec), wave_capacity=n + 1)) as s:
        s.set_source(8.0, inputs.amplitudes(n, seed=2))
        alone = s.adjoint(n, step0=0, grad_wave=gw)
        t = threading.Thread(target=short)
        t.start()
        try:
            beside = [s.adjoint(n, step0=0, grad_wave=gw) for _ in range(20)]
        finally:
            stop.set()
            t.join()
    assert not errors
    for ga, gr, _ in beside:
        assert np.array_equal(ga, alone[0]) and gr == alone[1]


@pytest.mark.parametrize("prec", ["fp64", "fp64_df", "fp32_kahan", "fp32"])
def test_a_small_resident_grid_planned_beside_a_large_one(prec):
    # the plan of 241 x 32 takes less shared memory than that of 800 x 64
    u0 = inputs.smooth_state(64, 800, seed=4)

    def states(between):
        with TeukSolver(params_of(800, 64, prec)) as s:
            s.set_resident(1)
            s.set_source(8.0)
            s.set_state(u0)
            s.step(7)
            if between:
                with TeukSolver(params_of(241, 32, prec)) as small:
                    small.set_resident(1)
                    small.step(3)
                    small.sync()
            s.step(7)
            return s.get_state()

    assert np.array_equal(states(False), states(True))
