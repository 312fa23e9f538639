"""The FP64 form's warp-per-pixel kernel (Gaussian shapes; steps that cannot
change the pixel's sum are screened out) against the FP64 oracle, at the sizes
where its work is divided differently.  The tolerance is the FP64 form's own,
1e-12 relative on every pixel: the screened steps add less than 2^-56 of the
sum, far below it."""
import numpy as np
import pytest

import oracle
from tests.helpers import abs_err_frac, rel_err_above
from paper_2205_07976_gb300 import nbgb
from paper_2205_07976_gb300 import workloads as W

pytestmark = pytest.mark.gpu

TOL = 1e-12


def _shot(S, M, os=1, T=1, interp=W.INTERP_TRICUBIC, n_phi=1):
    s = W.large_shot(n_src=S, n_mosaic=M)
    s.oversample, s.n_layers, s.interp = os, T, interp
    if T == 1:
        s.thickness_m = 0.0
    s.n_phi, s.phistep_deg = n_phi, 0.05
    return W.shrink(s, 13, 7, 2429, 886)


def _check(s):
    ref = oracle.image(s)
    got = nbgb.simulate(s, "f64")
    assert ref.max() > 0
    assert rel_err_above(got, ref, 1e-250)[0] <= TOL
    assert abs_err_frac(got, ref) <= TOL


# sources around the 128 whose vectors a warp holds; orientations around the
# 32 lanes and below 17 (several sources at a time); 1, 4 (shared by the
# block's warps), 9 and 36 (more than one pass) units
@pytest.mark.parametrize("interp", [W.INTERP_NEAREST, W.INTERP_TRICUBIC])
@pytest.mark.parametrize("S,M,os,T", [
    (127, 3, 1, 1), (129, 33, 1, 1), (257, 1, 1, 1), (9, 32, 1, 1),
    (64, 17, 2, 1), (100, 11, 2, 2), (40, 5, 3, 1), (33, 4, 6, 1),
    (1, 300, 1, 1), (5, 64, 3, 4)])
def test_matches_oracle_at_the_edges_of_its_work_division(S, M, os, T,
                                                          interp):
    _check(_shot(S, M, os, T, interp))


def test_phi_steps_small_table_and_default_F():
    s = _shot(30, 7, 2, 1, n_phi=3)
    s.F = s.F[50:73, 48:70, 52:69].copy()
    s.hkl_min = np.array([-10, -12, -8], dtype=np.int32)
    s.default_F = 35.0
    _check(s)
    s.interp = W.INTERP_NEAREST
    _check(s)


def test_negative_weights():
    s = _shot(40, 9)
    s.weights = s.weights.copy()
    s.weights[::3] *= -1.0
    ref, got = oracle.image(s), nbgb.simulate(s, "f64")
    # the terms cancel: against the sum of their magnitudes
    s.weights = np.abs(s.weights)
    assert np.max(np.abs(got - ref) / oracle.image(s)) <= TOL


def test_nan_in_the_table_reaches_the_same_pixels():
    s = _shot(40, 9, interp=W.INTERP_NEAREST)
    s = W.shrink(s, 40, 40, -20, -20)
    a, u = s.axes, 1.0 / s.lambdas
    p = s.panels[0]
    pos = p.origin + 20.5 * p.pixel_m * (p.fdir + p.sdir)
    h = (s.umats[0] @ a.T).T @ (pos / np.linalg.norm(pos) - s.dirs[0]) * u[0]
    n = np.ceil(h - 0.5).astype(int) - s.hkl_min
    s.F = s.F.copy()
    s.F[tuple(n)] = np.nan
    ref, got = oracle.image(s), nbgb.simulate(s, "f64")
    bad = np.isnan(ref)
    assert bad.any() and not bad.all()
    np.testing.assert_array_equal(np.isnan(got), bad)
    assert np.max(np.abs(got - ref)[~bad] / ref[~bad]) <= TOL


def test_a_pixel_alone_equals_the_pixel_in_the_image():
    for s in (_shot(100, 11, 2, 2), _shot(60, 9)):
        full = nbgb.simulate(s, "f64")
        sub = np.array([0, 5, 44, 90])
        np.testing.assert_array_equal(nbgb.simulate(s, "f64", pixels=sub),
                                      full[sub])
