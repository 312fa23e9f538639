"""The bounds-checked debug build on the forms whose indexes are computed from
the data: the warp kernel's segments and tasks of an odd number of sources and
its two pixels at a time, the screened FP64 kernel, and the background's nodes,
knots and guessed sources.  Every case passes the checks and matches the
oracle; in a child process, as test_check_build_gpu."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r'''
import numpy as np
import oracle
from paper_2205_07976_gb300 import nbgb
from paper_2205_07976_gb300 import workloads as W
from tests.helpers import masked_rel_err

assert nbgb.load().nb_version().decode().endswith("+check")

def close(got, ref, tol):
    rel, n = masked_rel_err(got, ref, 1e-3)
    assert rel <= tol, (rel, n)

def shot(S, M, os=1, T=1, interp=W.INTERP_TRICUBIC, width=0.005):
    s = W.large_shot(n_src=S, n_mosaic=M)
    s.oversample, s.n_layers, s.interp = os, T, interp
    if T == 1:
        s.thickness_m = 0.0
    s.dirs, s.lambdas, s.weights = W.gaussian_spectrum(S, 9.5, width)
    return W.shrink(s, 37, 29, 2433 - 20, 890 - 15)

# lines: odd and uneven numbers of sources, many lattice points, the most
# sources; halves: few items and steps
for S, M, os, T, width in ((33, 40, 1, 1, 0.005), (101, 12, 1, 2, 0.08),
                           (1023, 2, 1, 1, 0.02), (8, 10, 1, 1, 0.005),
                           (5, 3, 2, 1, 0.005)):
    for interp in (W.INTERP_NEAREST, W.INTERP_TRICUBIC):
        s = shot(S, M, os, T, interp, width)
        ref = oracle.image(s)
        close(nbgb.simulate(s, "mixed", variant="warp"), ref, 1e-5)
s = shot(45, 30)
rng = np.random.default_rng(4)
s.lambdas = 1.305 * (1.0 + 0.004 * rng.standard_normal(45))
close(nbgb.simulate(s, "mixed", variant="warp"), oracle.image(s), 1e-5)
s = shot(100, 12, 2, 1)
close(nbgb.simulate(s, "f64"), oracle.image(s), 1e-12)
# background: 1 to 101 sources, few and many knots, several directions
for S, knots, smax in ((1, 64, 0.5), (9, 512, 0.5), (101, 4096, 0.5),
                       (64, 2, 0.5), (50, 3000, 0.05)):
    s = shot(S, 1, width=0.05)
    bg = W.amorphous_background(knots, stol_max=smax)
    ref = oracle.background(s, bg)
    for prec, tol in (("f64", 1e-12), ("mixed", 1e-5)):
        sim = nbgb.Sim(prec).set_shot(s).set_background(bg)
        sim.add_background()
        close(sim.image(), ref, tol)
        sim.close()
print("check build ok")
'''


def test_check_build_on_computed_indexes():
    env = dict(os.environ, NBGB_VARIANT="check")
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, env=env,
                       capture_output=True, text=True, timeout=900)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-4000:]
    assert "check build ok" in r.stdout
