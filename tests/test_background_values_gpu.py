"""The background with weights whose products leave the range of FP64, at
the FP64 form's own 1e-12."""
import numpy as np
import pytest

from paper_2205_07976_gb300 import workloads as W
from tests.test_background_gpu import TOL, bg_image

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("c", [1e-200, 1e-170, 1e160, 1e200])
def test_fp64_weights_over_the_range(c):
    s = W.shrink(W.large_shot(n_src=1, n_mosaic=1), 35, 19, 1400, 900)
    s.dirs, s.lambdas, w = W.gaussian_spectrum(60, 9.5, 0.05)
    bg = W.amorphous_background(64)
    bg.F = np.cos(40.0 * bg.stol)  # the variance of a run matters
    s.weights = w
    ref = bg_image(s, bg, "f64")
    s.weights = w * c
    got = bg_image(s, bg, "f64") / c
    assert np.all(np.abs(got - ref) <= TOL["f64"] * ref)
