"""The refinement kernels at the sizes where their work divides: the adjoint
with more than 32 sources (its lanes take the surviving steps 32 sources at a
time) and many partial rows, and the Poisson loss's logarithm and quotient
over their whole range.  The adjoint's tolerance is the existing 1e-4; the
loss is FP64, and a few roundings of each term are allowed."""
import numpy as np
import pytest

import oracle
from paper_2205_07976_gb300 import nbgb
from paper_2205_07976_gb300 import workloads as W
from tests.test_grad_gpu import BKG, THETA, THETA_TRUE, gpu_grad, grad_shot
from tests.test_grad_gpu import with_theta

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("interp", [W.INTERP_NEAREST, W.INTERP_TRICUBIC])
@pytest.mark.parametrize("n_src", [31, 33, 70])
def test_adjoint_with_many_sources(n_src, interp):
    shot, U = grad_shot(n_src, interp)
    truth = oracle.image(with_theta(shot, U, THETA_TRUE))
    y = np.random.default_rng(7).poisson(truth + BKG).astype(np.float64)
    L0, g0, gF0, _ = oracle.loss_grad(with_theta(shot, U, THETA), U,
                                      THETA["cell"], THETA["rot"], y, BKG)
    L, g, gF, _ = gpu_grad(shot, U, y, THETA)
    assert abs(L - L0) <= 1e-6 * abs(L0)
    assert np.all(np.abs(g - g0) <= 1e-4 * np.abs(g0)
                  + 1e-6 * np.abs(g0).max())
    assert np.abs(gF - gF0).max() <= 1e-4 * np.abs(gF0).max()


def _loss(bkg, y, shot=None):
    shot = shot or W.shrink(W.single_shot_small(), 67, 41, 120, 110)
    sim = nbgb.Sim("mixed").set_shot(shot)
    sim.add_spots()
    img = sim.image()
    yd = torch.from_numpy(y[:img.size].copy()).cuda()
    d = torch.empty_like(yd)
    torch.cuda.synchronize()
    L = sim.poisson_loss(yd.data_ptr(), bkg, d.data_ptr())
    sim.close()
    return L, d.cpu().numpy(), img + bkg


@pytest.mark.parametrize("bkg", [1e-300, 1e-160, 1e-9, 1.0, 1.0078125, 37.5,
                                 1e12, 1e160])
def test_poisson_loss_over_its_range(bkg):
    rng = np.random.default_rng(5)
    y = rng.poisson(3.0, 67 * 41).astype(np.float64)
    y[::7] = 0.0
    y[3::11] = rng.uniform(1e-3, 1e6, y[3::11].size)
    L, d, m = _loss(bkg, y)
    ref = 1.0 - y / m
    assert np.all(np.abs(d - ref) <= 4e-16 * (1.0 + np.abs(y / m)))
    terms = m - y * np.log(m)
    scale = np.sum(np.abs(m) + np.abs(y * np.log(m)))
    assert abs(L - terms.sum()) <= 2e-15 * scale


def test_poisson_loss_of_a_pixel_without_a_logarithm():
    y = np.full(67 * 41, 2.0)
    y[10] = np.inf
    L, d, m = _loss(1.0, y)
    assert np.isnan(L) or np.isinf(L)
    assert d[10] == -np.inf
    keep = np.arange(y.size) != 10
    assert np.all(np.abs(d - (1.0 - 2.0 / m))[keep] <= 2e-15)
