"""The adjoint's sums over the many steps of a pixel of several subpixels,
layers, orientations and sources, against the oracle's gradient with the
existing 1e-4 (dL/dscale 1e-6), and over the range of dL/dI: the sums are
linear in it, and a power of two changes no rounding."""
import numpy as np
import pytest

import oracle
from paper_2205_07976_gb300 import nbgb
from paper_2205_07976_gb300 import workloads as W
from tests.test_grad_gpu import BKG, THETA, THETA_TRUE, gpu_grad, grad_shot
from tests.test_grad_gpu import with_theta

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def long_shot(interp):
    """16 x 12 pixels of the refinement shot with 2 x 2 subpixels, two layers,
    50 orientations and 100 sources: 40 000 steps per pixel."""
    s, U = grad_shot(100, interp)
    s.umats = W.mosaic_umats(np.random.default_rng(9), 50, 0.05)
    s.oversample, s.n_layers = 2, 2
    s.thickness_m, s.atten_m = 5e-4, 3e-4
    p = s.panels[0]
    p.origin = (p.origin + 30 * p.pixel_m * p.fdir + 28 * p.pixel_m * p.sdir)
    p.nfast, p.nslow = 16, 12
    s.panels = [p]
    return s, U


@pytest.mark.parametrize("interp", [W.INTERP_NEAREST, W.INTERP_TRICUBIC])
def test_long_sums_match_the_oracle(interp):
    shot, U = long_shot(interp)
    truth = oracle.image(with_theta(shot, U, THETA_TRUE))
    y = np.random.default_rng(7).poisson(truth + BKG).astype(np.float64)
    L0, g0, gF0, _ = oracle.loss_grad(with_theta(shot, U, THETA), U,
                                      THETA["cell"], THETA["rot"], y, BKG)
    L, g, gF, _ = gpu_grad(shot, U, y, THETA)
    err = np.abs(g - g0)
    assert abs(L - L0) <= 1e-6 * abs(L0)
    assert np.all(err <= 1e-4 * np.abs(g0) + 1e-6 * np.abs(g0).max())
    # dL/dscale sums terms of a few FP32 roundings each, compensated
    assert err[9] <= 1e-6 * np.abs(g0[9])
    assert np.abs(gF - gF0).max() <= 1e-4 * np.abs(gF0).max()


@pytest.mark.parametrize("interp,powers", [
    (W.INTERP_NEAREST, [-200, -140, 130, 200]),
    (W.INTERP_TRICUBIC, [-30, 100, 140])])
def test_gradient_is_linear_in_dLdI(interp, powers):
    shot, U = grad_shot(4, interp)
    shot.fluence = 1e14  # with it 2^140 is no large weight in the ring kernel
    sim = nbgb.Sim("mixed").set_shot(with_theta(shot, U, THETA))
    sim.set_params(U, THETA["cell"], THETA["rot"], THETA["N"], THETA["scale"])
    w = torch.from_numpy(np.random.default_rng(3).uniform(
        0.5, 1.0, shot.npix)).cuda()
    torch.cuda.synchronize()
    g0 = sim.adjoint(w.data_ptr())
    for e in powers:
        wc = w * 2.0 ** e
        torch.cuda.synchronize()
        g = sim.adjoint(wc.data_ptr())
        assert np.all(np.abs(g * 2.0 ** -e - g0) <= 1e-12 * np.abs(g0)), e
    sim.close()
