"""How a launch is cut (pieces of the per-step and reverse-step launches, blocks held per SM,
the record's own block, the builds for tall columns, the batch's branches) never changes a
result: automatic cuts against explicit strips and against each instance alone, bit for bit,
and against the oracle, at sizes around the edges of the rules (152 SMs: a piece more or less
than places, one column a piece, the last build of a register budget)."""
import numpy as np
import pytest

from paper_1001_3631_gb300 import TeukSolver, inputs

pytestmark = pytest.mark.gpu


def rel(a, b):
    return np.linalg.norm(np.asarray(a) - np.asarray(b)) / np.linalg.norm(b)


def params_of(nr, nth, m=2, **kw):
    return dict(dict(s=-2, m=m, a=0.8, rstar_min=-10.0, rstar_max=30.0, n_rstar=nr, n_theta=nth, rstar_ext=14.0,
                     dt_rule=1, courant=0.5), **kw)


def run(p, prec, n, u0, strip=0, persistent=False):
    with TeukSolver(dict(p, prec=prec)) as s:
        s.set_tiling(strip, 0 if persistent else 1)
        s.set_source(7.5)
        s.set_state(u0)
        s.step(n)
        u, w = s.get_state(), s.extract()[0]
        s.sync()
    return u, w


# columns n_rstar - 2 against the pieces of each rule: fewer than SMs, one a place or one more,
# three and four a place at 128 rows, twelve warps an SM of one-warp blocks
GRIDS = [(150, 20), (154, 20), (155, 33), (458, 100), (459, 128), (611, 100), (1826, 20), (306, 256), (307, 250)]


@pytest.mark.parametrize("prec,tol", [("fp64", 1e-12), ("fp64_df", 1e-12), ("fp32_kahan", 1e-6), ("fp32", 1e-5)])
@pytest.mark.parametrize("nr,nth", GRIDS)
def test_automatic_pieces_equal_strips(orc, nr, nth, prec, tol):
    p, n = params_of(nr, nth, m=3), 9
    u0 = inputs.smooth_state(nth, nr, seed=nr)
    u, w = run(p, prec, n, u0)
    for strip, persistent in ((7, False), (nr, False), (0, True)):
        us, ws = run(p, prec, n, u0, strip, persistent)
        assert np.array_equal(u, us) and np.array_equal(w, ws), (strip, persistent)
    po = orc.params(**p, r0=7.5)
    uo, wo = orc.run(po, u0, n, orc.orbit_source(po))
    assert rel(u, uo) <= tol and rel(w, wo) <= tol


# the 256-, 320-, 512-row builds meet at 256/257, 320/321 rows; the persistent kernel has no
# 320-row build
@pytest.mark.parametrize("prec,tol", [("fp64", 1e-12), ("fp32_kahan", 1e-6), ("fp32", 1e-5)])
@pytest.mark.parametrize("nth", [256, 257, 289, 320, 321])
def test_tall_columns(orc, nth, prec, tol):
    p, n = params_of(97, nth), 6
    u0 = inputs.smooth_state(nth, 97, seed=nth)
    u, w = run(p, prec, n, u0)
    us, ws = run(p, prec, n, u0, persistent=True)
    assert np.array_equal(u, us) and np.array_equal(w, ws)
    po = orc.params(**p, r0=7.5)
    uo, wo = orc.run(po, u0, n, orc.orbit_source(po))
    assert rel(u, uo) <= tol and rel(w, wo) <= tol


# the record at the ends of the grid and on a node, in a block of its own and in a piece
# (strip 1 on 152 x 4 columns leaves no place)
@pytest.mark.parametrize("prec", ["fp64", "fp64_df", "fp32_kahan", "fp32"])
@pytest.mark.parametrize("ext", [-10.0, -9.99, 14.0, 29.99, 30.0])
def test_record_of_every_block(orc, prec, ext):
    p, n = params_of(121, 12, rstar_ext=ext), 5
    u0 = inputs.random_state(12, 121, seed=3)
    po = orc.params(**p, r0=7.5)
    _, wo = orc.run(po, u0, n, orc.orbit_source(po))
    tol = 1e-12 if prec.startswith("fp64") else 1e-5
    for strip, persistent in ((0, False), (1, False), (40, False), (0, True)):
        _, w = run(p, prec, n, u0, strip, persistent)
        assert w.shape == wo.shape
        assert np.abs(w - wo).max() <= tol * max(np.abs(wo).max(), 1.0), (strip, persistent)


# classes of one, two and four warps, side by side (a few columns a place) and one after the
# other (too few)
@pytest.mark.parametrize("prec", ["fp64", "fp64_df", "fp32_kahan"])
@pytest.mark.parametrize("shape", [((1500, 32), (2200, 64), (1800, 100), (2500, 128)), ((60, 32), (70, 64), (40, 128))])
def test_batch_of_classes_equals_instances_alone(prec, shape):
    n = 12
    ps = [params_of(nr, nth, m=1 + k) for k, (nr, nth) in enumerate(shape)]
    u0 = [inputs.smooth_state(nth, nr, seed=k) for k, (nr, nth) in enumerate(shape)]
    with TeukSolver([dict(p, prec=prec) for p in ps]) as s:
        for k in range(len(ps)):
            s.set_source(7.5, instance=k)
            s.set_state(u0[k], 0, instance=k)
        s.step(n - 5)
        s.step(5)
        got = [(s.get_state(k), s.extract(instance=k)[0]) for k in range(len(ps))]
        s.sync()
    for k, p in enumerate(ps):
        u, w = run(p, prec, n, u0[k])
        assert np.array_equal(got[k][0], u) and np.array_equal(got[k][1], w), k


# the reverse step's pieces: fewer columns than pieces, a column a piece, two and three blocks
# an SM (FP64: 304 pieces of at least two columns, 456 from 2736 on), capped FP32 launches
@pytest.mark.parametrize("prec,tol", [("fp64", 1e-11), ("fp64_df", 1e-11), ("fp32_kahan", 1e-5)])
@pytest.mark.parametrize("nr,nth", [(8, 4), (9, 33), (305, 12), (609, 8), (1217, 64), (2735, 4), (2736, 5)])
def test_reverse_step_pieces(orc, nr, nth, prec, tol):
    # (the records lie within the particle's window, at its r* = 10.2, on every grid)
    p, n, r0 = params_of(nr, nth, rstar_max=200.0 if nr > 2000 else 30.0, rstar_ext=10.3), 6, 8.0
    amps = inputs.amplitudes(n, seed=nr)
    gw = np.random.default_rng(nr).standard_normal((n, nth, 2))
    po = orc.params(**p, r0=r0)
    ga_o, gr_o, _ = orc.adjoint(po, orc.orbit_source(po), gw, amps=amps)
    with TeukSolver(dict(p, prec=prec, wave_capacity=n + 1)) as s:
        s.set_source(r0, amps)
        ga, gr, _ = s.adjoint(n, step0=0, grad_wave=gw)
    assert rel(ga, ga_o) <= tol
    assert gr == pytest.approx(gr_o, rel=10 * tol)


# mode sum: records that wrap round the ring, one azimuth, more outputs than a block
@pytest.mark.parametrize("n_phi,cap", [(1, 4096), (3, 21), (70, 21)])
def test_mode_sum_ring_wrap(orc, n_phi, cap):
    ms, n = [-1, 0, 2], 50
    base = dict(s=-2, a=0.9, rstar_min=-10.0, rstar_max=30.0, n_rstar=80, n_theta=9, rstar_ext=13.0, dt=0.004)
    u0 = inputs.smooth_state(9, 80, seed=3)
    with TeukSolver([dict(base, m=m, prec="fp64", wave_capacity=cap) for m in ms]) as s:
        for k in range(3):
            s.set_source(7.0, instance=k)
            s.set_state(u0, 0, instance=k)
        s.step(n)
        phi = np.linspace(0.1, 6.0, n_phi)
        h = s.mode_sum(phi, n - 19, 20)
        s.sync()
    ps = [orc.params(**dict(base, m=m), r0=7.0) for m in ms]
    waves = [orc.run(p, u0, n, orc.orbit_source(p))[1][n - 19:n + 1] for p in ps]
    ho = orc.mode_sum(ps, waves, phi)
    assert h.shape == ho.shape == (20, 9, n_phi) and h.dtype == np.complex128
    assert rel(h, ho) <= 1e-12
