"""The amorphous background's sums over runs of sources (one node per knot
interval) against the FP64 oracle: source counts around a run of 8, knots
that fall inside runs or hold whole groups, weights that have no nodes.
Tolerances: the two forms' own, 1e-12 and 1e-5."""
import numpy as np
import pytest

import oracle
from paper_2205_07976_gb300 import workloads as W
from tests.test_background_gpu import TOL, bg_image, check

pytestmark = pytest.mark.gpu


def _shot(S, width=0.02):
    s = W.shrink(W.large_shot(n_src=1, n_mosaic=1), 35, 19, 1400, 900)
    s.dirs, s.lambdas, s.weights = W.gaussian_spectrum(S, 9.5, width)
    return s


@pytest.mark.parametrize("precision", ["f64", "mixed"])
@pytest.mark.parametrize("S,knots", [(1, 64), (7, 3), (8, 512), (9, 512),
                                     (17, 40), (64, 2), (100, 300),
                                     (101, 4096)])
def test_source_runs_and_knots(precision, S, knots):
    s = _shot(S)
    bg = W.amorphous_background(knots, stol_max=0.5)
    check(bg_image(s, bg, precision), oracle.background(s, bg), precision)


@pytest.mark.parametrize("precision", ["f64", "mixed"])
def test_factor_that_changes_sign(precision):
    s = _shot(50, 0.05)
    bg = W.amorphous_background(30)
    bg.F = np.cos(40.0 * bg.stol)
    check(bg_image(s, bg, precision), oracle.background(s, bg), precision)


@pytest.mark.parametrize("precision", ["f64", "mixed"])
def test_zero_and_negative_weights(precision):
    s = _shot(40)
    bg = W.amorphous_background(64)
    s.weights = s.weights.copy()
    s.weights[8:24] = 0.0
    check(bg_image(s, bg, precision), oracle.background(s, bg), precision)
    s.weights[30:] *= -0.5
    check(bg_image(s, bg, precision), oracle.background(s, bg), precision)


@pytest.mark.parametrize("precision", ["f64", "mixed"])
@pytest.mark.parametrize("n_dirs", [2, 1000])
def test_many_directions(precision, n_dirs):
    # 1000 directions and 4096 knots: the FP64 nodes do not fit as well
    s = W.shrink(_shot(1), 9, 5, 3, 4)
    rng = np.random.default_rng(2)
    d = np.concatenate([1e-3 * rng.standard_normal((n_dirs, 2)),
                        np.ones((n_dirs, 1))], 1)
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    s.dirs = d[np.arange(1000) % n_dirs]
    s.lambdas = 1.3 * (1.0 + 0.01 * rng.random(1000))
    s.weights = rng.random(1000) / 500.0
    bg = W.amorphous_background(4096)
    check(bg_image(s, bg, precision), oracle.background(s, bg), precision)
    assert TOL["f64"] < TOL["mixed"]
