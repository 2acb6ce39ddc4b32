"""The checked build on the reverse sweep: rows past n_theta read no record's cotangent (the
last record of the buffer included, n = 1), on columns that end inside a warp."""
import json
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r'''
import json, sys
import numpy as np
sys.path.insert(0, ROOT)
from paper_1001_3631_gb300 import TeukError, TeukSolver, _lib, inputs
from oracle import teuk_oracle as orc
assert _lib.load().teuk_checked_build() == 1
out = {}
for nth in (4, 33, 100):
    for n in (1, 3):
        g = dict(s=-2, m=2, a=0.7, rstar_min=-10.0, rstar_max=30.0, n_rstar=61, n_theta=nth, rstar_ext=10.0,
                 dt_rule=1, courant=0.5)
        amps = inputs.amplitudes(n, seed=nth)
        gw = np.random.default_rng(nth).standard_normal((n, nth, 2))
        p = orc.params(**g, r0=8.0)
        ga_o, _, _ = orc.adjoint(p, orc.orbit_source(p), gw, amps=amps)
        for prec in ("fp64", "fp64_df", "fp32_kahan", "fp32"):
            with TeukSolver(dict(g, prec=prec, wave_capacity=n + 1)) as s:
                s.set_source(8.0, amps)
                try:
                    ga, _, _ = s.adjoint(n, step0=0, grad_wave=gw)
                    s.sync()
                    e = float(np.linalg.norm(ga - ga_o) / np.linalg.norm(ga_o))
                except TeukError as ex:
                    e = "status %d" % ex.status
            out["%d rows, %d steps, %s" % (nth, n, prec)] = e
print("RESULT " + json.dumps(out))
'''


def test_reverse_sweep_stays_within_the_records():
    env = dict(os.environ, TEUK_LIB_VARIANT="check")
    r = subprocess.run([sys.executable, "-c", "ROOT = %r\n" % ROOT + CHILD], env=env, cwd=ROOT,
                       capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr[-3000:]
    line = [x for x in r.stdout.splitlines() if x.startswith("RESULT ")][-1]
    out = json.loads(line[len("RESULT "):])
    assert len(out) == 24
    for key, e in out.items():
        assert not isinstance(e, str) and e <= (1e-11 if "fp64" in key else 1e-5), (key, e)
