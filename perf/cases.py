"""The work that users of this package have it do, as cases that can be timed.

A case is a dict of plain values.  listed() names twelve of them and draw()
gives more of the same ranges; prepare() makes what a program holds before the
call (a handle or server with its tables, and the inputs, from a seed), run()
is one pass through the public entry points, work() what a pass cannot do
without, and exact() the same outputs in 64 bits from plain torch.

Five kinds of work:
  shot        one detector image of a re-oriented crystal: nb_set_crystal
              with the resident structure factors, nb_zero_image,
              nb_add_spots and nb_get_image on the device
  rows        the same for a list of pixels (nb_add_spots_pixels)
  background  the amorphous background of a detector (nb_add_background)
  refine      one refinement step: new structure factors and parameters,
              forward image, Poisson loss, adjoint
  serve       a batch of requests through the continuous-batching server,
              images fetched to the host

Images of the FP32-mixed form are fetched as float32, as the benchmark's
end-to-end leg does; images of the FP64 form as float64.
"""
import math

import numpy as np
import torch

from paper_2205_07976_gb300 import nbgb
from paper_2205_07976_gb300 import workloads as W

R_E = 2.8179403262e-15  # classical electron radius, m


def listed():
    return [
        # the smallest calls: a region of 1e3 pixels, one crystal orientation
        # after another; launches and host set-up count
        {"name": "roi_mixed", "kind": "shot", "optics": "serving",
         "precision": "mixed", "nf": 37, "ns": 27, "n_src": 11,
         "n_mosaic": 9},
        # the plain single shot (256^2, one wavelength, sinc N = 10) in both
        # forms: what a first-time user runs
        {"name": "single_mixed", "kind": "shot", "optics": "single",
         "precision": "mixed", "nf": 256, "ns": 256, "n_src": 1,
         "n_mosaic": 10},
        {"name": "single_f64", "kind": "shot", "optics": "single",
         "precision": "f64", "nf": 256, "ns": 256, "n_src": 1,
         "n_mosaic": 10},
        # an odd-sized window of the large shot's detector (100 energies, 50
        # mosaic domains, oversample 2, 2 layers, Gaussian, tricubic)
        {"name": "window_mixed", "kind": "shot", "optics": "large",
         "precision": "mixed", "nf": 203, "ns": 157, "n_src": 100,
         "n_mosaic": 50},
        # the large shot itself: the benchmark's workload
        {"name": "large_mixed", "kind": "shot", "optics": "large",
         "precision": "mixed", "nf": 3072, "ns": 3072, "n_src": 100,
         "n_mosaic": 50},
        # its FP64 form on a sample of rows, as the reference to a mixed image
        {"name": "rows_f64", "kind": "rows", "optics": "large",
         "precision": "f64", "nf": 3072, "ns": 3072, "every": 768,
         "n_src": 100, "n_mosaic": 50},
        # the precision sweep's shot (sinc, nearest lookup) in both forms
        {"name": "sweep_mixed", "kind": "shot", "optics": "sweep",
         "precision": "mixed", "nf": 1024, "ns": 1024, "n_src": 100,
         "n_mosaic": 20, "ncells": 50},
        {"name": "sweep_f64", "kind": "shot", "optics": "sweep",
         "precision": "f64", "nf": 307, "ns": 211, "n_src": 100,
         "n_mosaic": 20, "ncells": 200},
        # water around the crystal, over the large shot's whole detector
        {"name": "background_mixed", "kind": "background",
         "precision": "mixed", "nf": 3072, "ns": 3072, "n_src": 100,
         "knots": 64},
        # refinement steps on 64 panels of 185x194 pixels, 8 energies, 10
        # mosaic domains, for both lookups
        {"name": "refine_nearest", "kind": "refine", "interp": 0, "tiles": 8,
         "nf": 194, "ns": 185, "n_src": 8, "n_mosaic": 10},
        {"name": "refine_tricubic", "kind": "refine", "interp": 1, "tiles": 8,
         "nf": 194, "ns": 185, "n_src": 8, "n_mosaic": 10},
        # a batch of uneven requests (1-100 energies, 1-50 domains, regions of
        # 1e3 to 4e6 pixels) queued at once
        {"name": "serve_batch", "kind": "serve", "requests": 48,
         "max_src": 100, "max_mosaic": 50, "max_pix": 4000000},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo),
                                                          math.log(hi)))))))


def _sides(rng, lo, hi, most):
    """Two sides of a region: each log-uniform, the product at most `most`."""
    nf, ns = _log_int(rng, lo, hi), _log_int(rng, lo, hi)
    while nf * ns > most and (nf > lo or ns > lo):
        nf, ns = max(lo, int(nf * 0.8)), max(lo, int(ns * 0.8))
    return nf, ns


def draw(rng):
    kind = rng.choice(["mixed", "mixed", "sweep", "f64", "f64", "background",
                       "refine", "serve"])
    S, M = _log_int(rng, 1, 100), _log_int(rng, 1, 50)
    if kind == "mixed":
        optics = rng.choice(["large", "serving", "single"])
        if optics == "single":
            S = 1
        per_pixel = S * M * (8 if optics == "large" else 1)
        nf, ns = _sides(rng, 31, 3072, 8e10 / per_pixel)
        return {"kind": "shot", "optics": optics, "precision": "mixed",
                "nf": nf, "ns": ns, "n_src": S, "n_mosaic": M}
    if kind == "sweep":
        nf, ns = _sides(rng, 31, 1024, 2e9 / (S * M))
        return {"kind": "shot", "optics": "sweep", "precision": "mixed",
                "nf": nf, "ns": ns, "n_src": S, "n_mosaic": M,
                "ncells": rng.choice([10, 50, 200])}
    if kind == "f64":
        optics = rng.choice(["large", "single", "sweep"])
        if optics == "single":
            S = 1
        per_pixel = S * M * (8 if optics == "large" else 1)
        if optics == "large" and rng.random() < 0.5:
            every = _log_int(rng, 192, 1536)
            nf = max(31, min(3072, int(2.5e8 * every / (3072.0 * per_pixel))))
            return {"kind": "rows", "optics": "large", "precision": "f64",
                    "nf": nf, "ns": 3072, "every": every, "n_src": S,
                    "n_mosaic": M}
        nf, ns = _sides(rng, 31, 1024, 2.5e8 / per_pixel)
        c = {"kind": "shot", "optics": optics, "precision": "f64", "nf": nf,
             "ns": ns, "n_src": S, "n_mosaic": M}
        if optics == "sweep":
            c["ncells"] = rng.choice([10, 50, 200])
        return c
    if kind == "background":
        f64 = rng.random() < 0.3
        nf, ns = _sides(rng, 31, 3072, 3e5 if f64 else 1e7)
        return {"kind": "background", "precision": "f64" if f64 else "mixed",
                "nf": nf, "ns": ns, "n_src": S, "knots": _log_int(rng, 2, 512)}
    if kind == "refine":
        return {"kind": "refine", "interp": rng.randrange(2),
                "tiles": rng.randint(1, 8), "nf": _log_int(rng, 31, 194),
                "ns": _log_int(rng, 31, 185), "n_src": rng.randint(1, 8),
                "n_mosaic": rng.randint(4, 12)}
    return {"kind": "serve", "requests": rng.randint(6, 48), "max_src": S,
            "max_mosaic": M, "max_pix": _log_int(rng, 20000, 4000000)}


# --------------------------------------------------------------- inputs


def _shot(case, seed):
    """The shot of a `shot`, `rows` or `background` case."""
    S, M = case["n_src"], case.get("n_mosaic", 1)
    nf, ns = case["nf"], case["ns"]
    optics = case.get("optics", "large")
    if optics == "single":
        s = W.single_shot_small(seed)
        if M != s.n_mosaic:
            s.umats = W.mosaic_umats(np.random.default_rng([seed, 1]), M, 0.05)
        det = 256
    elif optics == "sweep":
        s = W.precision_shot(case["ncells"], seed, n_src=S, n_mosaic=M)
        det = 1024
    elif optics == "serving":
        rng = np.random.default_rng([seed, 2])
        s = W.serving_detector_shot(seed)
        s.axes = W.orthorhombic_axes(79.0, 79.0, 38.0,
                                     W.random_orientation(rng))
        s.umats = W.mosaic_umats(rng, M, 0.05)
        s.dirs, s.lambdas, s.weights = W.gaussian_spectrum(S, 9.5, 0.005)
        det = 3072
    else:
        s = W.large_shot(seed, n_src=S, n_mosaic=M)
        det = 3072
    if (nf, ns) != (det, det):
        # a window off the beam centre, as far as the detector allows
        f0 = max(0, min(det - nf, det // 2 + det // 8))
        s0 = max(0, min(det - ns, det // 2 + det // 8))
        s = W.shrink(s, nf, ns, f0, s0)
    return s


def _refine_inputs(case, seed):
    """(shot, U, theta, F, y): the multi-panel shot, its orientation, the ten
    parameters, the structure factors and a measured image: background counts
    and, in one pixel of fifty, a spot."""
    rng = np.random.default_rng([seed, 3])
    shot = W.multipanel_shot(case["n_src"], seed, n_mosaic=case["n_mosaic"],
                             tiles=(case["tiles"], case["tiles"]),
                             panel=(case["nf"], case["ns"]))
    shot.interp = case["interp"]
    U = W.random_orientation(rng)
    theta = np.concatenate([1e-4 * rng.standard_normal(3),
                            np.array([79.0, 79.0, 38.0])
                            * (1.0 + 5e-4 * rng.standard_normal(3)),
                            15.0 + 0.5 * rng.uniform(-1, 1, 3),
                            [1.0 + 0.1 * rng.uniform(-1, 1)]])
    spots = rng.exponential(40.0, shot.npix) * (rng.random(shot.npix) < 0.02)
    y = rng.poisson(1.0 + spots).astype(np.float64)
    return shot, U, theta, y


def _requests(case, seed):
    """The resident shot and the requests: their sizes belong to the case,
    the orientations, domains and structure factors to the seed."""
    rng = np.random.default_rng([seed, 5])
    base = W.serving_detector_shot(seed)
    reqs = W.serving_requests(case["requests"], max_src=case["max_src"],
                              max_mosaic=case["max_mosaic"],
                              max_pix=float(case["max_pix"]))
    for r in reqs:
        r.axes = W.orthorhombic_axes(79.0, 79.0, 38.0,
                                     W.random_orientation(rng))
        r.umats = W.mosaic_umats(rng, r.umats.shape[0], 0.05)
    return base, reqs


# ------------------------------------------------------ prepare and run


def prepare(case, seed):
    dev = torch.device("cuda", 0)
    kind = case["kind"]
    if kind == "serve":
        base, reqs = _requests(case, seed)
        offs = np.concatenate([[0], np.cumsum([r.npix for r in reqs])])
        host = torch.empty(int(offs[-1]), dtype=torch.float64,
                           pin_memory=True)
        return {"kind": kind, "reqs": reqs, "offs": offs, "host": host,
                "srv": nbgb.Server(base, max_slots=64, pool_bytes=4 << 30,
                                   step_budget=2_000_000_000)}
    if kind == "refine":
        shot, U, theta, y = _refine_inputs(case, seed)
        sim = nbgb.Sim("mixed").set_shot(shot)
        yd = torch.from_numpy(y).to(dev)
        return {"kind": kind, "sim": sim, "U": U, "theta": theta, "y": yd,
                "dLdI": torch.empty_like(yd),
                "F": torch.from_numpy(shot.F).to(dev)}
    shot = _shot(case, seed)
    sim = nbgb.Sim(case["precision"]).set_shot(shot)
    dtype = torch.float64 if case["precision"] == "f64" else torch.float32
    state = {"kind": kind, "sim": sim, "shot": shot,
             "code": (nbgb.NB_DTYPE_F64 if case["precision"] == "f64"
                      else nbgb.NB_DTYPE_F32),
             "image": torch.empty(shot.npix, dtype=dtype, device=dev)}
    if kind == "rows":
        state["pixels"] = W.strided_rows(shot, case["every"])
        state["index"] = torch.from_numpy(state["pixels"]).to(dev)
    if kind == "background":
        sim.set_background(_background(case, seed))
    return state


def _background(case, seed):
    bg = W.amorphous_background(case["knots"])
    bg.n_molecules *= 0.5 + np.random.default_rng([seed, 4]).random()
    return bg


def run(state):
    kind = state["kind"]
    if kind == "serve":
        return _run_serve(state)
    sim = state["sim"]
    if kind == "refine":
        th, F = state["theta"], state["F"]
        sim.set_fcell_device(F.data_ptr(), F.numel())
        sim.set_params(state["U"], th[3:6], th[0:3], th[6:9], th[9])
        sim.zero()
        sim.add_spots()
        loss = sim.poisson_loss(state["y"].data_ptr(), 1.0,
                                state["dLdI"].data_ptr())
        gF = torch.zeros(F.shape, dtype=torch.float64, device=F.device)
        g = sim.adjoint(state["dLdI"].data_ptr(), gF.data_ptr())
        # gradients in the precision of the structure factors
        return {"loss": torch.tensor(loss, dtype=torch.float32),
                "grad": torch.from_numpy(g).float(), "grad_F": gF.float()}
    image = state["image"]
    if kind == "background":
        sim.zero()
        sim.add_background()
    else:
        sim.set_crystal(state["shot"], with_F=False)
        sim.zero()
        sim.add_spots(state.get("pixels"))
    sim.image_to_device(image.data_ptr(), image.numel(), state["code"])
    return image[state["index"]] if kind == "rows" else image


def _run_serve(state):
    srv, host, offs = state["srv"], state["host"], state["offs"]
    buf = host.numpy()
    place = {}
    for i, r in enumerate(state["reqs"]):
        rid = srv.submit(r.axes, r.umats, r.lambdas, r.weights, r.scale,
                         r.roi)
        place[rid] = i
    left = len(place)
    while left:
        srv.step()
        for rid in srv.completed():
            i = place[rid]
            srv.result(rid, out=buf[offs[i]:offs[i + 1]])
            left -= 1
    # the images as they are stored: float32
    return host.float()


# ----------------------------------------------------------------- work


def _spot_flops(npix, units, PM, S, shape, interp, N):
    """The method's own arithmetic on npix pixels of `units` subpixel x layer
    units: per unit 60 flops, per (unit, orientation) 21, per step 9 for h
    and its offset and 8 (Gaussian exponent) or 96 (sinc); and per term whose
    Gaussian factor does not vanish in FP32 the lookup and the product."""
    n_units = float(npix) * units
    steps = n_units * PM * S
    share = 1.0
    if shape == W.SHAPE_GAUSS:
        share = min(1.0, 4.0 / 3.0 * math.pi * (44.0 * 0.63) ** 1.5 / N ** 3)
    term = 4 + (3 if shape == W.SHAPE_GAUSS else 0) + (
        198 if interp == W.INTERP_TRICUBIC else 0)
    return (60 * n_units + 21 * n_units * PM
            + steps * (17 if shape == W.SHAPE_GAUSS else 105)
            + term * share * steps)


def _optics(case):
    """(units per pixel, shape, interp, N, table entries) of a shot case."""
    return {"single": (1, W.SHAPE_SINC, W.INTERP_NEAREST, 10.0, 61 ** 3),
            "sweep": (1, W.SHAPE_SINC, W.INTERP_NEAREST,
                      float(case.get("ncells", 10)), 121 ** 3),
            "serving": (1, W.SHAPE_GAUSS, W.INTERP_TRICUBIC, 25.0, 121 ** 3),
            "large": (8, W.SHAPE_GAUSS, W.INTERP_TRICUBIC, 25.0, 121 ** 3),
            }[case["optics"]]


def work(case):
    kind = case["kind"]
    if kind == "serve":
        _, reqs = _requests(case, 0)
        flops = sum(_spot_flops(r.npix, 1, r.umats.shape[0], len(r.lambdas),
                                W.SHAPE_GAUSS, W.INTERP_TRICUBIC, 25.0)
                    for r in reqs)
        return {"bytes": 121 ** 3 * 4 + 8 * sum(r.npix for r in reqs),
                "flops": flops}
    if kind == "refine":
        npix = case["tiles"] ** 2 * case["nf"] * case["ns"]
        fwd = _spot_flops(npix, 1, case["n_mosaic"], case["n_src"],
                          W.SHAPE_GAUSS, case["interp"], 15.0)
        # the adjoint repeats the sum and differentiates it; the measured
        # image is read, the table read and its gradient written
        return {"bytes": 8 * npix + 12 * 81 ** 3, "flops": 3 * fwd}
    npix = case["nf"] * case["ns"]
    if kind == "background":
        return {"bytes": 8 * npix,
                "flops": npix * 8 * (60 + 7.0 * case["n_src"])}
    if kind == "rows":
        npix = case["nf"] * len(range(0, case["ns"], case["every"]))
    units, shape, interp, N, table = _optics(case)
    return {"bytes": 8 * npix + 4 * table,
            "flops": _spot_flops(npix, units, case["n_mosaic"],
                                 case["n_src"], shape, interp, N)}


# ---------------------------------------------------------------- exact


def _f64(a):
    return torch.as_tensor(np.asarray(a, dtype=np.float64), device="cuda")


def _unit_directions(shot, pixels=None):
    """Unit directions d [P, units, 3] and the factors solid angle x capture
    x polarization [P, units] of the (listed) pixels of a shot whose sources
    share one direction."""
    pos, nrm, px2 = [], [], []
    for p in shot.panels:
        f = torch.arange(p.nfast, dtype=torch.float64, device="cuda")
        s = torch.arange(p.nslow, dtype=torch.float64, device="cuda")
        S, Fa = torch.meshgrid(s, f, indexing="ij")
        pos.append(torch.stack([S.reshape(-1), Fa.reshape(-1)], 1))
    where = torch.cat(pos)
    panel = torch.repeat_interleave(
        torch.arange(len(shot.panels), device="cuda"),
        torch.tensor([p.npix for p in shot.panels], device="cuda"))
    if pixels is not None:
        where, panel = where[pixels], panel[pixels]
    O, Fd, Sd, Nd = (_f64([getattr(p, k) for p in shot.panels])[panel]
                     for k in ("origin", "fdir", "sdir", "ndir"))
    px = _f64([p.pixel_m for p in shot.panels])[panel]
    os, T = shot.oversample, shot.n_layers
    dt = shot.thickness_m / T
    i0, e = _f64(shot.dirs[0]), _f64(shot.evec)
    e = e - (e @ i0) * i0
    e = e / e.norm()
    b = torch.linalg.cross(i0, e)
    ds, facs = [], []
    for i in range(os):
        for j in range(os):
            for t in range(T):
                P = (O + ((where[:, 1] + (i + 0.5) / os) * px)[:, None] * Fd
                     + ((where[:, 0] + (j + 0.5) / os) * px)[:, None] * Sd
                     + t * dt * Nd)
                R = P.norm(dim=1)
                d = P / R[:, None]
                fac = px * px * (Nd * P).sum(1) / R ** 3
                if shot.thickness_m > 0:
                    L = shot.atten_m * (d * Nd).sum(1)
                    fac = fac * (torch.exp(-t * dt / L)
                                 - torch.exp(-(t + 1) * dt / L))
                fac = fac * 0.5 * (1 + (d @ i0) ** 2 - shot.kahn
                                   * ((d @ e) ** 2 - (d @ b) ** 2))
                ds.append(d)
                facs.append(fac)
    return torch.stack(ds, 1), torch.stack(facs, 1)


def _lagrange(x):
    """Weights of the nodes -1, 0, 1, 2 at x in [0, 1), last axis."""
    return torch.stack([-x * (x - 1) * (x - 2) / 6,
                        (x + 1) * (x - 1) * (x - 2) / 2,
                        -(x + 1) * x * (x - 2) / 2,
                        (x + 1) * x * (x - 1) / 6], -1)


def _lookup(F, hmin, interp, default, h, n):
    """F at h [.., 3] with nearest lattice points n: nearest or tricubic."""
    hn = torch.tensor(F.shape, device="cuda")
    flat = F.reshape(-1)

    def nearest(m):
        i = m.long() - hmin
        ok = ((i >= 0) & (i < hn)).all(-1)
        i = torch.where(ok[..., None], i, torch.zeros_like(i))
        v = flat[(i[..., 0] * hn[1] + i[..., 1]) * hn[2] + i[..., 2]]
        return torch.where(ok, v, torch.full_like(v, default))

    if interp == W.INTERP_NEAREST:
        return nearest(n)
    fl = torch.floor(h.detach()).long()
    i = fl - hmin
    ok = ((i >= 1) & (i + 2 < hn)).all(-1)
    base = torch.where(ok[..., None], i - 1, torch.zeros_like(i))
    w = _lagrange(h - fl)
    r = torch.arange(4, device="cuda")
    idx = (((base[:, 0, None, None, None] + r[:, None, None]) * hn[1]
            + (base[:, 1, None, None, None] + r[None, :, None])) * hn[2]
           + (base[:, 2, None, None, None] + r[None, None, :]))
    v = (flat[idx] * w[:, 2, None, None, :]).sum(-1)
    v = (v * w[:, 1, None, :]).sum(-1)
    v = (v * w[:, 0, :]).sum(-1)
    return torch.where(ok, v, nearest(n))


def _spots(shot, F, axes, N, d, fac):
    """sum over (unit, orientation, source) of F_cell^2 F_latt^2 w fac for
    the pixels of d [P, units, 3], without the prefactor.  Differentiable in
    F, axes and N.  Gaussian terms below exp(-400) of the peak are left out
    of the lookup."""
    umats = _f64(shot.umats)
    A = torch.einsum("mij,vj->mvi", umats, axes)  # rows a, b, c per domain
    v = d - _f64(shot.dirs[0])
    G = torch.einsum("pui,mvi->pumv", v, A)
    u, w = 1.0 / _f64(shot.lambdas), _f64(shot.weights)
    wf = (fac[:, :, None, None] * w).expand(*G.shape[:3], len(u))
    hmin = torch.as_tensor(np.asarray(shot.hkl_min, dtype=np.int64),
                           device="cuda")
    P = d.shape[0]
    if shot.shape == W.SHAPE_SINC:
        lat, hs, ns = 1.0, [], []
        for x in range(3):
            h = G[..., x, None] * u
            n = torch.ceil(h - 0.5)
            f = h - n
            zero = f.abs() < 1e-100
            f = torch.where(zero, torch.ones_like(f), f)
            r = torch.sin(math.pi * N[x] * f) / torch.sin(math.pi * f)
            lat = lat * torch.where(zero, N[x].expand_as(r), r)
            hs.append(h)
            ns.append(n)
        h, n = torch.stack(hs, -1), torch.stack(ns, -1)
        fc = _lookup(F, hmin, shot.interp, shot.default_F, h.reshape(-1, 3),
                     n.reshape(-1, 3)).reshape(lat.shape)
        return (fc * fc * lat * lat * wf).sum((1, 2, 3))
    with torch.no_grad():
        rad = 0.0
        for x in range(3):
            h = G[..., x, None] * u
            rad = rad + (N[x] * (h - torch.ceil(h - 0.5))) ** 2 / 0.63
        at = (rad < 200.0).nonzero()
        del rad, h
    p, q, m, k = at.unbind(1)
    if shot.interp == W.INTERP_TRICUBIC and len(at) > 4_000_000:
        out = torch.zeros(P, dtype=torch.float64, device="cuda")
        for c in at.split(4_000_000):
            out = out + _terms(shot, F, hmin, N, G, u, wf, c, P)
        return out
    return _terms(shot, F, hmin, N, G, u, wf, at, P)


def _terms(shot, F, hmin, N, G, u, wf, at, P):
    p, q, m, k = at.unbind(1)
    h = G[p, q, m] * u[k][:, None]
    n = torch.ceil(h.detach() - 0.5)
    f = h - n
    lat = N.prod() * torch.exp(-((N * f) ** 2).sum(1) / 0.63)
    fc = _lookup(F, hmin, shot.interp, shot.default_F, h, n)
    t = fc * fc * lat * lat * wf[p, q, m, k]
    return torch.zeros(P, dtype=torch.float64,
                       device="cuda").index_add(0, p, t)


def _prefactor(shot):
    return R_E ** 2 * shot.fluence / (shot.oversample ** 2 * shot.n_mosaic)


def _exact_image(shot, pixels=None):
    """The image, or None where no pixel holds a spot (the FP32 forms leave
    out Gaussian tails that underflow, so such an image has no one value)."""
    d, fac = _unit_directions(shot, pixels)
    F, axes, N = _f64(shot.F), _f64(shot.axes), _f64(shot.ncells)
    per = shot.oversample ** 2 * shot.n_layers * shot.n_mosaic * shot.n_src
    c = max(1, int(2e7 // per))
    out = [_spots(shot, F, axes, N, d[i:i + c], fac[i:i + c])
           for i in range(0, d.shape[0], c)]
    image = _prefactor(shot) * torch.cat(out)
    return image if float(image.max()) > 1e-12 else None


def _exact_background(shot, bg):
    d, fac = _unit_directions(shot)
    u, w = 1.0 / _f64(shot.lambdas), _f64(shot.weights)
    st, Fb = _f64(bg.stol), _f64(bg.F)
    half = 0.5 * (d - _f64(shot.dirs[0])).norm(dim=2)
    pre = R_E ** 2 * shot.fluence * bg.n_molecules / shot.oversample ** 2
    out = []
    for hc, fc in zip(half.split(60000), fac.split(60000)):
        x = (hc[:, :, None] * u).clamp(st[0], st[-1])
        j = (torch.bucketize(x, st, right=True) - 1).clamp(0, len(st) - 2)
        slope = (Fb[1:] - Fb[:-1]) / (st[1:] - st[:-1])
        v = Fb[j] + slope[j] * (x - st[j])
        out.append(((v * v * w).sum(2) * fc).sum(1))
    return pre * torch.cat(out)


def _rotation(t):
    c, s, o, z = torch.cos(t), torch.sin(t), torch.ones_like(t[0]), \
        torch.zeros_like(t[0])
    X = torch.stack([o, z, z, z, c[0], -s[0], z, s[0], c[0]]).reshape(3, 3)
    Y = torch.stack([c[1], z, s[1], z, o, z, -s[1], z, c[1]]).reshape(3, 3)
    Z = torch.stack([c[2], -s[2], z, s[2], c[2], z, z, z, o]).reshape(3, 3)
    return X @ Y @ Z


def _exact_refine(case, seed):
    shot, U, theta, y = _refine_inputs(case, seed)
    d, fac = _unit_directions(shot)
    yd = _f64(y)
    F = _f64(shot.F).requires_grad_()
    th = _f64(theta).requires_grad_()
    c = max(1, int(1e7 // (shot.n_mosaic * shot.n_src)))
    loss, gth, gF = 0.0, torch.zeros_like(th), torch.zeros_like(F)
    for i in range(0, d.shape[0], c):
        axes = ((_rotation(th[0:3]) @ _f64(U)) * th[3:6]).T
        I = _prefactor(shot) * th[9] * _spots(shot, F, axes, th[6:9],
                                              d[i:i + c], fac[i:i + c])
        m = I + 1.0
        L = (m - yd[i:i + c] * torch.log(m)).sum()
        a, b = torch.autograd.grad(L, (th, F))
        loss, gth, gF = loss + L.detach(), gth + a, gF + b
    return {"loss": loss.cpu(), "grad": gth.cpu(), "grad_F": gF}


def exact(case, seed):
    kind = case["kind"]
    if kind == "refine":
        return _exact_refine(case, seed)
    if kind == "serve":
        base, reqs = _requests(case, seed)
        if sum(r.pixel_steps for r in reqs) > 4e10:
            return None
        images = [_exact_image(W.request_shot(base, r)) for r in reqs]
        return torch.cat([torch.zeros(r.npix, dtype=torch.float64)
                          if v is None else v.cpu()
                          for v, r in zip(images, reqs)])
    shot = _shot(case, seed)
    if kind == "background":
        return _exact_background(shot, _background(case, seed))
    pixels = None
    if kind == "rows":
        pixels = torch.from_numpy(W.strided_rows(shot, case["every"])).cuda()
    steps = shot.steps_per_pixel * (shot.npix if pixels is None
                                    else len(pixels))
    if steps > 3e10:
        return None
    return _exact_image(shot, pixels)
