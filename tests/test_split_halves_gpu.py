"""The warp kernel's form for few items and steps per pixel (up to 16 and 128),
where each half of a warp sums a pixel of its own: numbers of items and pairs
around 16, odd numbers of pixels, tables with pixels that take intervals and
pixels that scan source blocks side by side, unsorted sources.  Against the
oracle with the mixed form's tolerance, the thread kernel's term count, and
bitwise between launches (in both, a pixel has another neighbour)."""
import numpy as np
import pytest

from paper_2205_07976_gb300 import nbgb
from paper_2205_07976_gb300 import workloads as W
from tests.test_split_lines_gpu import _check, _shot

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("interp", [W.INTERP_NEAREST, W.INTERP_TRICUBIC])
@pytest.mark.parametrize("S,M,os,T", [(1, 1, 1, 1), (15, 1, 1, 1),
                                      (128, 1, 1, 1), (7, 15, 1, 1),
                                      (8, 16, 1, 1), (3, 4, 2, 1),
                                      (8, 2, 2, 2), (9, 1, 2, 3)])
def test_items_and_pairs(S, M, os, T, interp):
    _check(_shot(S, M, os, T, interp))


@pytest.mark.parametrize("interp", [W.INTERP_NEAREST, W.INTERP_TRICUBIC])
@pytest.mark.parametrize("N", [12.0, 15.0, 60.0])
def test_intervals_and_blocks_side_by_side(N, interp):
    s = _shot(12, 4, N=N, interp=interp)
    # a wide spectrum passes more than 8 lattice points in some pixels
    for width in (0.01, 0.04, 0.08):
        s.dirs, s.lambdas, s.weights = W.gaussian_spectrum(12, 9.5, width)
        _check(s)
    s.lambdas = s.lambdas[::-1].copy()
    s.lambdas[5] = s.lambdas[2]
    _check(s)


def test_counts_of_the_work():
    s = _shot(9, 8)
    sim = nbgb.Sim("mixed").set_shot(s).set_variant("warp")
    sim.add_spots()
    img, terms = sim.image(), sim.stats()[0]
    sim.count_work().zero()
    sim.add_spots()
    np.testing.assert_array_equal(sim.image(), img)
    assert sim.stats()[0] == terms
    assert sim.work()["pairs"] >= terms
    sim.close()


@pytest.mark.parametrize("nf,ns", [(1, 1), (3, 5), (37, 13)])
def test_server_sums_the_same(nf, ns):
    base = W.serving_detector_shot()
    r = W.serving_requests(1, seed=3, max_src=2, max_mosaic=2)[0]
    rng = np.random.default_rng(9)
    umats = np.stack([np.linalg.qr(np.eye(3) + 1e-3
                                   * rng.standard_normal((3, 3)))[0]
                      for _ in range(9)])
    umats *= np.sign(np.einsum("mii->mi", umats))[:, None, :]
    _, lambdas, weights = W.gaussian_spectrum(11, 9.5, 0.01)
    f0, s0 = 1500, 1400
    srv = nbgb.Server(base, max_slots=1, pool_bytes=1 << 20)
    rid = srv.submit(r.axes, umats, lambdas, weights, r.scale,
                     (f0, s0, nf, ns))
    srv.run_all()
    got = srv.result(rid)
    srv.close()
    s = base.copy()
    s.axes, s.umats, s.lambdas, s.weights = r.axes, umats, lambdas, weights
    s.scale = r.scale
    s.dirs = np.repeat(base.dirs[:1], 11, axis=0)
    pix = ((s0 + np.arange(ns))[:, None] * 3072
           + (f0 + np.arange(nf))[None, :]).ravel()
    sim = nbgb.Sim("mixed").set_shot(s)
    sim.add_spots(pix)
    np.testing.assert_array_equal(got, sim.image()[pix])
    sim.close()
