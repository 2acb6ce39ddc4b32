"""The cut of the columns that is in effect (teuk_get_tiling): a strip length that is set is
kept whatever its value, and the autotuner knows the automatic cut."""
import json

import numpy as np
import pytest

from paper_1001_3631_gb300 import TeukSolver, inputs

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


def test_the_tuner_keeps_an_automatic_cut_that_is_fastest(tmp_path):
    # FP64 2048 x 128 (too large for resident launches): 43.7 us a step, uniform strips 51
    with TeukSolver(params_of(2048, 128, "fp64")) as s:
        s.set_instance_tiling(0, 5)
        chosen = s.autotune(trial_steps=30, cache_path=str(tmp_path / "t.json"))
        t = s.tiling()
        assert t["automatic"] and chosen == [t["columns"]]
    table = json.loads((tmp_path / "t.json").read_text())
    assert list(table.values()) == [0]


@pytest.mark.parametrize("batch", [False, True])
def test_a_cached_automatic_cut_is_each_grids_own(tmp_path, batch):
    # one entry serves every grid of its bucket (a batch: every context of the same shapes)
    cache = tmp_path / "t.json"
    grids = [8000, 8000] if batch else [8000, 5001]
    for k, nr in enumerate(grids):
        ps = [params_of(nr, 128, "fp32_kahan")] * (2 if batch else 1)
        with TeukSolver(ps) as s:
            auto = s.tiling()
            if k == 0:
                s.autotune(trial_steps=2, cache_path=str(cache))
                cache.write_text(json.dumps({key: 0 for key in json.loads(cache.read_text())}))
                continue
            s.set_instance_tiling(0, 7)
            launches = s.kernel_launches()
            assert s.autotune(cache_path=str(cache)) == [auto["columns"]] * len(ps)
            assert s.kernel_launches() == launches and s.tiling() == auto


def test_tables_of_other_cuts_are_not_used(tmp_path):
    cache = tmp_path / "t.json"
    with TeukSolver(params_of(8000, 128, "fp32_kahan")) as s:
        s.autotune(trial_steps=2, cache_path=str(cache))
        (key,) = json.loads(cache.read_text())
        old = key.rsplit("|", 1)[0]   # as written before the cut had a version
        cache.write_text(json.dumps({old: 3}))
        s.autotune(trial_steps=2, cache_path=str(cache))
        assert json.loads(cache.read_text()).keys() == {old, key}


# the record at the two ends of the grid, beside them and inside, by the piece that holds it (a
# launch with a piece for every place) and by a block of its own (one piece)
@pytest.mark.parametrize("prec,tol", [("fp64", 1e-12), ("fp64_df", 1e-12), ("fp32_kahan", 1e-5), ("fp32", 1e-5)])
@pytest.mark.parametrize("ext", [-10.0, -9.99, 14.0, 29.99, 30.0])
def test_record_in_a_launch_that_takes_every_place(orc, prec, tol, ext):
    nr, nth, n = 2500, 100, 3
    p = dict(params_of(nr, nth, prec), rstar_ext=ext)
    u0 = inputs.random_state(nth, nr, seed=5)
    po = orc.params(**{k: v for k, v in p.items() if k != "prec"}, r0=7.5)
    _, wo = orc.run(po, u0, n, orc.orbit_source(po))
    waves = []
    for strip in (0, nr):
        with TeukSolver(p) as s:
            s.set_tiling(strip, 1)
            pieces = s.tiling()["pieces"]
            assert pieces == 1 if strip else pieces % 152 == 0 and pieces >= 3 * 152   # 152 SMs
            s.set_source(7.5)
            s.set_state(u0)
            s.step(n)
            waves.append(s.extract()[0])
    assert np.array_equal(waves[0], waves[1])
    assert np.abs(waves[0] - wo).max() <= tol * max(np.abs(wo).max(), 1.0)
