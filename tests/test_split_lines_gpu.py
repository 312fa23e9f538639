"""The warp kernel's line form (shots of at least 32 sources and 1200 steps per
pixel: an interval entry's steps are summed along its line through a cell):
segment and task lengths, uneven spectra, lattice points at and beyond the
table's edge, and shots whose batches of items go back and forth between
intervals and source blocks.  Against the oracle with the mixed form's
tolerance, the thread kernel's term count, and bitwise between launches."""
import numpy as np
import pytest

import oracle
from paper_2205_07976_gb300 import nbgb
from paper_2205_07976_gb300 import workloads as W
from tests.test_parity_gpu import check_mixed

pytestmark = pytest.mark.gpu


def _shot(S, M, os=1, T=1, interp=W.INTERP_TRICUBIC, N=25.0):
    s = W.large_shot(n_src=S, n_mosaic=M)
    s.oversample, s.n_layers, s.interp = os, T, interp
    s.ncells = np.array([N, N, N])
    if T == 1:
        s.thickness_m = 0.0
    return W.shrink(s, 37, 29, 2433 - 20, 890 - 15)


def _check(s):
    ref = oracle.image(s)
    assert ref.max() > 0
    sim = nbgb.Sim("mixed").set_shot(s).set_variant("warp")
    sim.add_spots()
    img, (ev, ps) = sim.image(), sim.stats()
    sim.zero()
    sub = np.arange(5, s.npix, 131)
    sim.add_spots(sub)
    part = sim.image()[sub]
    sim.set_variant("thread").zero()
    sim.add_spots()
    ev_thread = sim.stats()[0]
    sim.close()
    check_mixed(img, ref)
    np.testing.assert_array_equal(part, img[sub])
    # the same steps survive the cut, up to its rounding
    assert abs(ev - ev_thread) <= 1e-4 * ev_thread + 2


@pytest.mark.parametrize("interp", [W.INTERP_NEAREST, W.INTERP_TRICUBIC])
@pytest.mark.parametrize("S,M,os,T", [(32, 38, 1, 1), (33, 40, 1, 2),
                                      (64, 5, 2, 1), (127, 3, 2, 2),
                                      (100, 12, 1, 1), (1024, 2, 1, 1)])
def test_line_lengths(S, M, os, T, interp):
    _check(_shot(S, M, os, T, interp))


@pytest.mark.parametrize("interp", [W.INTERP_NEAREST, W.INTERP_TRICUBIC])
def test_uneven_spectrum(interp):
    s = _shot(90, 14, 1, 1, interp)
    rng = np.random.default_rng(4)
    lam = 1.305 * (1.0 + 0.004 * rng.standard_normal(90))
    lam[10:20] = lam[10]  # equal wavelengths
    s.lambdas = lam
    s.weights = rng.random(90)
    _check(s)


@pytest.mark.parametrize("interp", [W.INTERP_NEAREST, W.INTERP_TRICUBIC])
def test_table_edge_and_default_F(interp):
    s = _shot(70, 20, 1, 1, interp)
    # a table that ends among the lattice points of the window
    a = s.axes
    p = s.panels[0]
    pos = p.origin + 18.0 * p.pixel_m * p.fdir + 14.0 * p.pixel_m * p.sdir
    h = a @ (pos / np.linalg.norm(pos) - s.dirs[0]) / s.lambdas[35]
    m = np.rint(h).astype(int)
    lo = m - np.array([6, 7, 5]) - s.hkl_min
    n = np.array([7, 9, 7])
    s.F = s.F[lo[0]:lo[0] + n[0], lo[1]:lo[1] + n[1],
              lo[2]:lo[2] + n[2]].copy()
    s.hkl_min = (lo + s.hkl_min).astype(np.int32)
    s.default_F = 60.0
    _check(s)


@pytest.mark.parametrize("N", [12.0, 15.0, 60.0])
def test_other_crystal_sizes(N):
    # N = 12: the ellipsoids of neighbouring lattice points overlap at the
    # cut; a wide spectrum passes more than 8 lattice points per item
    s = _shot(60, 25, N=N)
    _check(s)
    s.dirs, s.lambdas, s.weights = W.gaussian_spectrum(60, 9.5, 0.08)
    _check(s)
