"""The FP64 form's sinc: lattice points, sines and reciprocal of its own, and
pixels shared by several lanes, against the oracle at the form's tolerance of
1e-12."""
import numpy as np
import pytest

import oracle
from paper_2205_07976_gb300 import nbgb
from paper_2205_07976_gb300 import workloads as W
from tests.test_parity_gpu import check_f64

pytestmark = pytest.mark.gpu


# 1, 2, 4 and 32 lanes per pixel; more lanes than sources; both lookups
@pytest.mark.parametrize("interp", [W.INTERP_NEAREST, W.INTERP_TRICUBIC])
@pytest.mark.parametrize("S,M,N", [(1, 1, 1), (5, 51, 10), (16, 16, 3),
                                   (1, 600, 50), (3, 300, 200),
                                   (128, 32, 7)])
def test_lanes_per_pixel(S, M, N, interp):
    s = W.precision_shot(N, n_src=S, n_mosaic=M)
    s.interp = interp
    s = W.shrink(s, 19, 11, 610, 630)
    check_f64(nbgb.simulate(s, "f64"), oracle.image(s))
    sub = np.array([0, 18, 100, 19 * 11 - 1])
    np.testing.assert_array_equal(nbgb.simulate(s, "f64", pixels=sub),
                                  nbgb.simulate(s, "f64")[sub])


@pytest.mark.parametrize("os,T", [(2, 2), (3, 1), (2, 3), (1, 2), (8, 1)])
@pytest.mark.parametrize("shape", [W.SHAPE_SINC, W.SHAPE_GAUSS])
def test_units_shared_by_lanes(os, T, shape):
    s = W.precision_shot(10, n_src=3, n_mosaic=4)
    s.shape, s.oversample, s.n_layers = shape, os, T
    s.thickness_m, s.atten_m = 4e-4, 3e-4
    s = W.shrink(s, 19, 11, 610, 630)
    check_f64(nbgb.simulate(s, "f64"), oracle.image(s))


def test_lattice_points_ties_and_far_from_the_table():
    # h, k, l = -+ multiples of 1/2 (ties), exact lattice points, and values
    # beyond 2^30: axes along the components of d - i0 of single pixels
    s = W.single_shot_small(n=8)
    s.umats = W.identity_umats(1)
    s.default_F = 3.0
    s.dirs, s.lambdas, s.weights = W.monochromatic(1.0)
    s.panels = [W.flat_detector(1, 1, 1e-4, 0.1, beam_center=(-250.0, 120.0))]
    p = s.panels[0]
    pos = p.origin + 0.5 * p.pixel_m * (p.fdir + p.sdir)
    v = pos / np.sqrt(pos @ pos) - s.dirs[0]
    for scale in (0.5, -0.5, 1.5, -2.5, 3.0, 12.25, 3e9, 1e17):
        s.axes = np.diag(scale / v)
        s.ncells = np.array([5.0, 5.0, 5.0])
        ref = oracle.image(s)
        got = nbgb.simulate(s, "f64")
        assert np.all(np.abs(got - ref) <= 1e-12 * np.abs(ref)), scale
