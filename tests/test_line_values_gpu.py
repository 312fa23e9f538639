"""The line form (test_split_lines_gpu) where a line's cell changes and where
its table is special: sources right at an offset's sign change, and entries
that are not finite.  Tolerances: the mixed form's own, 1e-5; which pixels are
finite is exact."""
import numpy as np
import pytest

import oracle
from paper_2205_07976_gb300 import nbgb
from paper_2205_07976_gb300 import workloads as W

pytestmark = pytest.mark.gpu

CUT = 44.0 * 0.63  # steps with sum N^2 f^2 above this have no FP32 term


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


def _reach(s, entry):
    """Per pixel: whether a step under the cut uses the table entry, and
    whether one might, up to the FP32 rounding of the cut and of a cell's
    boundary."""
    p = s.panels[0]
    ij = np.stack(np.meshgrid(np.arange(p.nslow), np.arange(p.nfast),
                              indexing="ij"), -1).reshape(-1, 2) + 0.5
    pos = (p.origin + p.pixel_m * (ij[:, 1:] * p.fdir + ij[:, :1] * p.sdir))
    v = pos / np.linalg.norm(pos, axis=1, keepdims=True) - s.dirs[0]
    sure = np.zeros(len(pos), bool)
    maybe = np.zeros(len(pos), bool)
    for um in s.umats:
        g = v @ (s.axes @ um.T).T
        h = g[:, None, :] / s.lambdas[None, :, None]
        n = np.rint(h)
        f = h - n
        r = np.sum((s.ncells * f) ** 2, -1)
        if s.interp == W.INTERP_NEAREST:
            use = near = np.all(n == entry, -1)
        else:
            lo = np.floor(h) - 1
            use = np.all((entry >= lo) & (entry <= lo + 3), -1)
            lo_d, lo_u = np.floor(h - 1e-6) - 1, np.floor(h + 1e-6) - 1
            near = np.all((entry >= lo_d) & (entry <= lo_u + 3), -1)
            use &= np.all(lo_d == lo_u, -1)
        sure |= np.any(use & (r <= CUT * (1 - 1e-4)), 1)
        maybe |= np.any(near & (r <= CUT * (1 + 1e-4)), 1)
    return sure, maybe


@pytest.mark.parametrize("interp", [W.INTERP_NEAREST, W.INTERP_TRICUBIC])
@pytest.mark.parametrize("bad", [np.nan, np.inf, 3e38])
def test_table_entries_that_are_not_finite(interp, bad):
    """A pixel is not finite exactly where a step under the cut uses the
    entry (3e38: its square is not)."""
    s = W.large_shot(n_src=100, n_mosaic=12)
    s.oversample, s.n_layers, s.thickness_m, s.interp = 1, 1, 0.0, interp
    s = W.shrink(s, 61, 47, 2433 - 30, 890 - 23)
    p = s.panels[0]
    pos = p.origin + p.pixel_m * (30.0 * p.fdir + 23.0 * p.sdir)
    h = s.axes @ (pos / np.linalg.norm(pos) - s.dirs[0]) / s.lambdas[50]
    entry = np.rint(h).astype(int)
    s.F = s.F.copy()
    s.F[tuple(entry - s.hkl_min)] = bad
    sure, maybe = _reach(s, entry)
    assert sure.any() and not maybe.all()
    for variant in ("warp", "thread"):
        ok = np.isfinite(nbgb.simulate(s, "mixed", variant=variant))
        assert not ok[sure].any(), variant
        assert ok[~maybe].all(), (variant, int((~ok[~maybe]).sum()))


def test_pixels_far_from_every_lattice_point():
    """Windows whose terms all lie far out in a reflection's tail (their
    brightest pixel 1e-12 to 1e-30 of a peak), where a term's error is its
    exponent's: against the FP64 form, window by window, in the geometric mean
    no more than half above the thread kernel's error, which forms every
    exponent from its own offset."""
    err = {"warp": [], "thread": []}
    for S, M, N, interp, f0, s0 in (
            (100, 30, 18.0, 1, 580, 371), (64, 50, 18.0, 1, 940, 2100),
            (64, 50, 25.0, 0, 1855, 2236), (40, 50, 18.0, 1, 942, 2860),
            (100, 30, 25.0, 0, 1859, 1472), (40, 50, 18.0, 0, 1027, 1129),
            (64, 50, 18.0, 1, 2250, 2447), (40, 50, 18.0, 0, 2945, 1956),
            (100, 30, 18.0, 1, 483, 834), (40, 30, 25.0, 1, 2667, 1731),
            (64, 50, 25.0, 1, 2200, 2952), (64, 50, 60.0, 0, 847, 2959)):
        s = W.large_shot(n_src=S, n_mosaic=M)
        s.oversample, s.n_layers, s.thickness_m = 1, 1, 0.0
        s.interp, s.ncells = interp, np.array([N, N, N])
        s = W.shrink(s, 16, 16, f0, s0)
        ref = nbgb.simulate(s, "f64")
        if not 1e-30 < ref.max() / (8e-8 * N ** 6) < 1e-12:
            continue
        m = ref > 1e-2 * ref.max()
        for v in err:
            got = nbgb.simulate(s, "mixed", variant=v)
            e = (got - ref)[m] / ref[m]
            err[v].append(np.mean(e ** 2))
    assert len(err["warp"]) >= 6
    rms = {v: np.exp(0.5 * np.mean(np.log(e))) for v, e in err.items()}
    assert rms["warp"] <= 1.5 * rms["thread"], rms
