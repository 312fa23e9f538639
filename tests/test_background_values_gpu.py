"""The background at scattering angles whose square is next to the least
normal FP32 number, with weights whose products leave the range of FP64, and
in every form of the kernels (nodes, nodes or single sources where knots are
dense, single sources): the two forms' own tolerances, 1e-12 and 1e-5."""
import numpy as np
import pytest

import oracle
from paper_2205_07976_gb300 import nbgb
from paper_2205_07976_gb300 import workloads as W
from tests.test_background_gpu import TOL, bg_image, check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["f64", "mixed"])
@pytest.mark.parametrize("e", [-46, -50, -54])
def test_tiny_angles(precision, e):
    """A pixel 2^e m off the beam at 1 m, and knots of that size."""
    s = W.large_shot(n_src=1, n_mosaic=1)
    s.oversample, s.n_layers, s.thickness_m = 1, 1, 0.0
    s.lambdas = np.array([1.0])
    px = 2.0 ** -30
    s.panels = [W.Panel(origin=np.array([-0.5 * px + 2.0 ** e, -0.5 * px, 1.0]),
                        fdir=np.array([1.0, 0.0, 0.0]),
                        sdir=np.array([0.0, 1.0, 0.0]),
                        ndir=np.array([0.0, 0.0, 1.0]), pixel_m=px, nfast=1,
                        nslow=1)]
    # stol = 2^(e - 1): a quarter of the way down from 1000 to 0
    bg = W.Background(stol=np.array([0.0, 2.0 ** (e + 1)]),
                      F=np.array([1000.0, 0.0]), n_molecules=1e10)
    ref = oracle.background(s, bg)
    got = bg_image(s, bg, precision)
    assert ref[0] > 0
    assert abs(got[0] - ref[0]) <= TOL[precision] * ref[0], (got, ref)


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


def _beam(s, S, width, tilt=0.0):
    s.dirs, s.lambdas, s.weights = W.gaussian_spectrum(
        S, 9.5, width, (tilt, 0.0, 1.0))


@pytest.mark.parametrize("precision", ["f64", "mixed"])
def test_tables_follow_the_beam_and_the_curve(precision):
    """One handle through beams and curves of every form of the kernel gives
    bitwise what a fresh handle gives, and the same call twice the same."""
    s = W.shrink(W.large_shot(n_src=1, n_mosaic=1), 35, 19, 1400, 900)
    sim = None
    for S, width, tilt, knots, neg in ((100, 0.005, 0.0, 64, False),
                                       (9, 0.005, 0.0, 4096, False),
                                       (9, 0.005, 0.002, 4096, False),
                                       (50, 0.02, 0.0, 40, True),
                                       (1, 0.005, 0.0, 40, False),
                                       (100, 0.005, 0.0, 512, False)):
        _beam(s, S, width, tilt)
        if neg:
            s.weights = s.weights.copy()
            s.weights[3] *= -1.0
        bg = W.amorphous_background(knots, stol_max=0.5)
        ref = bg_image(s, bg, precision)
        if sim is None:
            sim = nbgb.Sim(precision).set_shot(s)
        sim.set_beam(s)
        sim.set_background(bg)
        for _ in range(2):
            sim.zero()
            sim.add_background()
            np.testing.assert_array_equal(sim.image(), ref)
    # the curve alone, then the beam alone
    sim.set_background(W.amorphous_background(33))
    sim.zero()
    sim.add_background()
    np.testing.assert_array_equal(
        sim.image(), bg_image(s, W.amorphous_background(33), precision))
    _beam(s, 7, 0.01)
    sim.set_beam(s)
    sim.zero()
    sim.add_background()
    np.testing.assert_array_equal(
        sim.image(), bg_image(s, W.amorphous_background(33), precision))
    sim.close()


@pytest.mark.parametrize("precision", ["f64", "mixed"])
@pytest.mark.parametrize("S,knots,dirs,neg", [
    (9, 4096, 1, False), (8, 4096, 1, False), (33, 4096, 1, False),
    (100, 4096, 1, False), (64, 40, 64, False), (65, 40, 1, True),
    (31, 700, 3, True), (2, 4096, 1, False)])
def test_dense_knots_single_sources_and_negative_weights(precision, S, knots,
                                                         dirs, neg):
    s = W.shrink(W.large_shot(n_src=1, n_mosaic=1), 35, 19, 1400, 900)
    _beam(s, S, 0.005)
    rng = np.random.default_rng(2)
    d = np.concatenate([1e-3 * rng.standard_normal((dirs, 2)),
                        np.ones((dirs, 1))], 1)
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    if dirs > 1:
        s.dirs = d[np.arange(S) % dirs]
    if neg:
        s.weights = s.weights.copy()
        s.weights[S // 3] *= -0.5
    bg = W.amorphous_background(knots, stol_max=0.5)
    check(bg_image(s, bg, precision), oracle.background(s, bg), precision)
