"""The line form (test_split_lines_gpu) where a line's cell changes: sources
right at an offset's sign change.  Tolerance: the mixed form's own, 1e-5."""
import numpy as np
import pytest

import oracle
from paper_2205_07976_gb300 import nbgb
from paper_2205_07976_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _pixel_shot(u, N, axes, d, px=1e-4):
    """One pixel in direction d at 0.1 m, 12 equal orientations, sources at
    1/lambda = u along +z."""
    s = W.large_shot(n_src=1, n_mosaic=1)
    s.oversample, s.n_layers, s.thickness_m = 1, 1, 0.0
    s.umats = W.identity_umats(12)
    s.axes, s.ncells = axes, np.array([N, N, N])
    s.lambdas = 1.0 / u
    s.weights = np.full(u.size, 1.0 / u.size)
    s.dirs = np.repeat(s.dirs[:1], u.size, axis=0)
    n = d / np.linalg.norm(d)
    f = np.cross([0.0, 1.0, 0.0], n)
    f /= np.linalg.norm(f)
    t = np.cross(n, f)
    o = 0.1 * n - 0.5 * px * (f + t)
    s.panels = [W.Panel(origin=o, fdir=f, sdir=t, ndir=n, pixel_m=px, nfast=1,
                        nslow=1)]
    return s


def _cut_shots():
    """Sources of which one, number s, puts h within a few 1e-9 of an
    integer, with k's sign change between the sources s - 2 and s - 1 and l's
    20 sources away: the sources s - 1 and s are a segment of two (or s the
    first of the next one, by the rounding of the sign change)."""
    rng = np.random.default_rng(8)
    for i in range(64):
        S, s = 100, 40 + i % 20
        U = W.random_orientation(rng)
        d = np.array([0.3, 0.2, 0.9]) + 0.05 * rng.standard_normal(3)
        d /= np.linalg.norm(d)
        v = d - np.array([0.0, 0.0, 1.0])
        u = 0.77 * (1.0 + 1e-3 * (np.arange(S) - s))
        e = U * np.sign(U @ v)[:, None]  # rows with e . v > 0
        ev = e @ v
        eps = rng.uniform(-3e-9, 3e-9)
        h = np.array([20.0 + eps, 11.0, 1.02])
        at = np.array([u[s], 0.5 * (u[s - 2] + u[s - 1]), u[s]])
        yield _pixel_shot(u, 16.0, e * (h / (at * ev))[:, None], d)


def test_sources_at_a_sign_change():
    worst = 0.0
    for s in _cut_shots():
        ref = oracle.image(s)
        got = nbgb.simulate(s, "mixed", variant="warp")
        assert ref[0] > 0
        worst = max(worst, abs(got[0] - ref[0]) / ref[0])
    assert worst <= 1e-5, worst
