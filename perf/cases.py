"""Timing cases of the library: the calls a program that reduces detector images makes, over
the sizes, image types, splits and options it makes them with.

listed() are the cases that are followed, draw(rng) gives more of the same ranges,
prepare(case, seed) makes what a program holds before the call (the integrator, its correction
arrays, the frames), run(state) is one pass through the public entry points and returns its
outputs, work(case) the bytes and operations a pass cannot do without, and exact(case, seed)
the same outputs in 64-bit torch arithmetic written out here (no code of the library).

Kinds of a case:
  frame     one image through Integrator.integrate (FP32 compensated or FP64, 1D or 2D)
  bound     a batch of frames against corrections bound once (integrate_batch_bound)
  batch     a batch of frames with the corrections passed per call (integrate_batch)
  variance  the propagated counting variance of a batch of frames
  grad      one differentiable integration and its gradients (autograd.integrate)
  multi     several detectors in one graph launch (MultiPlan)
  setup     a new geometry: matrix built, corrections computed, first frame integrated
  host      frames in pinned host memory through integrate_batch_host
"""
from __future__ import annotations

import math

import torch

UNIT_Q, UNIT_2TH = "q_nm^-1", "2th_deg"
ALL, NORM, NONE = "dark+flat+sa+pol", "sa+pol", ""
POL_FACTOR = 0.99


def _case(name, kind, ny, nx, npt, azim=0, unit=UNIT_Q, split="full", dtype="uint32", corr=ALL,
          mask=False, frames=1, precision="fp32", pixel=172e-6, dist=0.3, off1=0.0, off2=0.0,
          rot1=0.0, rot2=0.0, rot3=0.0, geom_seed=0):
    """off1, off2: the foot point (PONI) from the detector centre, as a share of the side."""
    c = dict(kind=kind, ny=ny, nx=nx, npt=npt, azim=azim, unit=unit, split=split, dtype=dtype,
             corr=corr, mask=mask, frames=frames, precision=precision, pixel=pixel, dist=dist,
             off1=off1, off2=off2, rot1=rot1, rot2=rot2, rot3=rot3, geom_seed=geom_seed)
    if name:
        c["name"] = name
    return c


def listed():
    pilatus6m = dict(ny=2527, nx=2463, npt=1000, split="full", dtype="uint32", corr=ALL, mask=True,
                     pixel=172e-6, dist=0.3, off1=0.0028, off2=0.0106, rot1=0.02, rot2=0.01)
    pilatus1m = dict(ny=1043, nx=981, npt=1000, split="bbox", dtype="int32", corr=ALL, mask=True,
                     pixel=172e-6, dist=0.2, off1=0.0068, off2=0.0267, rot1=0.02, rot2=0.01)
    cake = dict(ny=2048, nx=2048, npt=500, azim=360, unit=UNIT_2TH, split="full", dtype="float32",
                pixel=50e-6, dist=0.15, rot1=0.05)
    return [
        # the smallest call: a small float image, no corrections, as an interactive program or
        # a test makes it -- launches and latency are all of it
        _case("frame_256_f32", "frame", 256, 256, 200, unit=UNIT_2TH, split="bbox", dtype="float32",
              corr=NONE, pixel=100e-6, dist=0.1, off1=-0.03, off2=0.002),
        # one signed 1-Mpixel frame with every correction passed per call: live view of a
        # running measurement, a frame at a time
        _case("frame_1m_i32", "frame", **pilatus1m),
        # one 6-Mpixel frame in double precision: the reference-quality result of a single shot
        _case("frame_6m_fp64", "frame", precision="fp64", **pilatus6m),
        # one 2D (radial x azimuthal) pattern of a 4-Mpixel float image: texture and strain work
        _case("cake_4m_f32", "frame", corr=ALL, **cake),
        # a scan on one detector: 128 frames against corrections bound once
        _case("bound_6m_128", "bound", frames=128, **pilatus6m),
        # a short scan of an unmasked 4.5-Mpixel detector at fine binning, an odd number of
        # frames, dark and flat passed with the call
        _case("batch_4m_37", "batch", 2167, 2070, 2000, dtype="uint32", corr="dark+flat", frames=37,
              pixel=75e-6, dist=0.2, rot1=0.013, rot2=-0.021, rot3=0.4),
        # a scan reduced to 2D patterns, solid angle and polarisation only
        _case("cake_batch_16", "batch", corr=NORM, frames=16, **cake),
        # error bars of a scan of signed 1-Mpixel frames
        _case("variance_1m_24", "variance", frames=24, **dict(pilatus1m, corr=NONE)),
        # a training or refinement step: the pattern and the gradients for image and flat field
        _case("grad_6m", "grad", **dict(pilatus6m, dtype="float32")),
        # several detectors of uneven shape and binning, one launch per exposure
        _case("multi_16", "multi", 2167, 2070, 5000, corr=NONE, frames=16, pixel=75e-6, dist=0.2,
              geom_seed=3),
        # a new geometry (calibration, a moved detector): build, corrections, first frame
        _case("setup_1m", "setup", corr="dark+flat+sa+pol", **{k: v for k, v in pilatus1m.items() if k != "corr"}),
        # frames as a detector's receiver leaves them in host memory, results wanted there
        _case("host_1m_64", "host", frames=64, **pilatus1m),
    ]


MAX_FRAME_PIXELS = 128 * 2527 * 2463  # the largest listed case's pixels


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["frame"] * 6 + ["bound"] * 3 + ["batch"] * 4 + ["variance", "grad", "grad", "multi",
                                                                     "setup", "host"])
    ny = _log(rng, 200, 2540)
    nx = max(150, min(2540, int(ny * rng.uniform(0.7, 1.4))))
    azim = rng.choice([0, 0, 0, rng.randint(36, 360)]) if kind in ("frame", "bound", "batch", "grad") else 0
    npt = _log(rng, 100, 500) if azim else _log(rng, 100, 5000 if ny > 800 else 1500)
    frames = {"bound": _log(rng, 2, 128), "batch": _log(rng, 2, 128), "variance": _log(rng, 1, 48),
              "host": _log(rng, 2, 64), "multi": rng.randint(4, 16)}.get(kind, 1)
    if kind != "multi":
        frames = max(1, min(frames, MAX_FRAME_PIXELS // (2 * ny * nx), (4 if azim else 8) * 10 ** 8 // (ny * nx)))
    if kind == "host":
        frames = max(1, min(frames, 64 * 1043 * 981 // (ny * nx)))
    corner = rng.random() < 0.2  # the beam near a corner of the detector
    return _case(
        None, kind, ny, nx, npt, azim, unit=rng.choice([UNIT_Q, UNIT_2TH]),
        split=rng.choice(["full", "full", "full", "bbox", "bbox", "none"]),
        dtype="float32" if kind == "grad" else rng.choice(["uint32", "int32", "float32"]),
        corr="" if kind in ("variance", "multi") else rng.choice([ALL, ALL, NORM, "dark+flat", NONE]),
        mask=rng.random() < 0.5 and kind != "multi", frames=frames,
        precision=rng.choice(["fp32", "fp32", "fp64"]) if kind in ("frame", "grad") else "fp32",
        pixel=rng.choice([75e-6, 100e-6, 172e-6]), dist=round(rng.uniform(0.1, 0.5), 3),
        off1=round(0.46 if corner else rng.uniform(-0.05, 0.05), 4),
        off2=round(-0.47 if corner else rng.uniform(-0.05, 0.05), 4),
        rot1=round(rng.uniform(-0.05, 0.05), 4), rot2=round(rng.uniform(-0.05, 0.05), 4),
        rot3=round(rng.uniform(-3.0, 3.0), 3), geom_seed=rng.randint(1, 10 ** 6))


# --------------------------------------------------------------------------------------
# geometry and inputs (plain torch)
# --------------------------------------------------------------------------------------
MULTI_SHAPES = ((512, 1028, 75e-6), (1679, 1475, 172e-6), (2167, 2070, 75e-6))
MULTI_BINS = (500, 2000, 5000)


def _instances(c):
    """The detectors of a multi case: uneven shapes, bins, distances and tilts."""
    g = torch.Generator().manual_seed(1000 + c["geom_seed"])
    r = lambda a, b: float(torch.rand(1, generator=g, dtype=torch.float64) * (b - a) + a)  # noqa: E731
    out = []
    for k in range(c["frames"]):
        ny, nx, px = MULTI_SHAPES[int(torch.randint(3, (1,), generator=g))]
        bins = [b for b in MULTI_BINS if b <= c["npt"]] or [c["npt"]]
        d = dict(c, kind="frame", ny=ny, nx=nx, pixel=px, npt=bins[int(torch.randint(len(bins), (1,), generator=g))],
                 dist=r(0.1, 0.5), off1=r(-0.02, 0.02), off2=r(-0.02, 0.02), rot1=r(-0.05, 0.05),
                 rot2=r(-0.05, 0.05), rot3=r(-0.05, 0.05), frames=1)
        out.append(d)
    return out


def _params(c):
    """(dist, poni1, poni2, rot1, rot2, rot3, pixel1, pixel2, wavelength)"""
    return (c["dist"], c["ny"] * c["pixel"] * (0.5 + c["off1"]), c["nx"] * c["pixel"] * (0.5 + c["off2"]),
            c["rot1"], c["rot2"], c["rot3"], c["pixel"], c["pixel"], 1e-10)


def _lab(c, i, j):
    """Laboratory vector Rz Ry Rx (d1 - poni1, d2 - poni2, dist) of detector coordinates (in
    pixels) i, j; also the untilted offsets."""
    dist, p1, p2, r1, r2, r3, px1, px2, _ = _params(c)
    x, y = i * px1 - p1, j * px2 - p2
    z = torch.full_like(x * y, dist)
    x, y = x + 0 * z, y + 0 * z
    x0, y0 = x, y
    y, z = math.cos(r1) * y - math.sin(r1) * z, math.sin(r1) * y + math.cos(r1) * z
    x, z = math.cos(r2) * x + math.sin(r2) * z, -math.sin(r2) * x + math.cos(r2) * z
    x, y = math.cos(r3) * x - math.sin(r3) * y, math.sin(r3) * x + math.cos(r3) * y
    return x, y, z, x0, y0


def _angles(c, i, j):
    """(radial value in the case's unit, chi in degrees, 2theta, chi in radians)"""
    x, y, z, _, _ = _lab(c, i, j)
    tth = torch.atan2(torch.sqrt(x * x + y * y), z)
    chi = torch.atan2(x, y)
    rad = tth * (180.0 / math.pi) if c["unit"] == UNIT_2TH else 4.0 * math.pi * torch.sin(0.5 * tth) / 1e-10 * 1e-9
    return rad, chi * (180.0 / math.pi), tth, chi


def _grid(c, centres, dev):
    o = 0.5 if centres else 0.0
    n1, n2 = (c["ny"], c["nx"]) if centres else (c["ny"] + 1, c["nx"] + 1)
    i = torch.arange(n1, dtype=torch.float64, device=dev).add(o).unsqueeze(1)
    j = torch.arange(n2, dtype=torch.float64, device=dev).add(o).unsqueeze(0)
    return i, j


def _corrections64(c, dev):
    """Solid angle (dist / |t|)^3 and polarisation of the pixel centres, in 64 bits."""
    i, j = _grid(c, True, dev)
    _, _, _, x0, y0 = _lab(c, i, j)
    sa = (c["dist"] / torch.sqrt(x0 * x0 + y0 * y0 + c["dist"] ** 2)) ** 3
    _, _, tth, chi = _angles(c, i, j)
    pol = 0.5 * (1.0 + torch.cos(tth) ** 2 - POL_FACTOR * torch.cos(2.0 * chi) * torch.sin(tth) ** 2)
    return sa, pol


def _mask(c, dev):
    """Gaps between modules of 195 x 487 pixels (17 rows, 7 columns), 1 = masked."""
    if not c["mask"]:
        return None
    i = torch.arange(c["ny"], device=dev) % 212 >= 195
    j = torch.arange(c["nx"], device=dev) % 494 >= 487
    return (i.unsqueeze(1) | j.unsqueeze(0)).to(torch.uint8)


def _arrays(c, seed, dev):
    """{dark, flat, sa, pol}: float32 arrays of the corrections a case has."""
    have = c["corr"].split("+")
    g = torch.Generator(device=dev).manual_seed(7919 * seed + 17)
    shape = (c["ny"], c["nx"])
    dark = torch.randn(shape, generator=g, device=dev) + 10.0
    flat = torch.rand(shape, generator=g, device=dev) * 0.1 + 0.95
    sa, pol = _corrections64(c, dev) if "sa" in have or "pol" in have else (None, None)
    return {"dark": dark if "dark" in have else None, "flat": flat if "flat" in have else None,
            "sa": sa.float() if "sa" in have else None, "pol": pol.float() if "pol" in have else None}


def _frames(c, seed, dev, mask):
    """[frames, ny, nx] counts: Poisson noise on a falling background with twenty rings (in 2D
    with an azimuthal modulation); the gaps of a masked detector hold -1 (all bits set)."""
    i, j = _grid(c, True, dev)
    rad, _, _, chi = _angles(c, i, j)
    top = float(rad.max())
    x = rad.clamp_min(0.004 * top)
    lam = 12.0 * top / x
    for k in range(20):
        xk = top * (0.1 + 0.8 * k / 19)
        lam = lam + 2000.0 * torch.exp(-((x - xk) ** 2) / (2 * (0.004 * top) ** 2))
    if c["azim"]:
        lam = lam * (1.0 + 0.3 * torch.cos(2.0 * chi))
    lam = lam.float()
    g = torch.Generator(device=dev).manual_seed(104729 * seed + 5)
    n = 1 if c["kind"] in ("frame", "grad", "setup") else c["frames"]
    ints = c["dtype"] != "float32"
    out = torch.empty((n,) + tuple(lam.shape), dtype=torch.int32 if ints else torch.float32, device=dev)
    for a in range(0, n, 16):
        b = min(n, a + 16)
        out[a:b] = torch.poisson(lam.expand(b - a, -1, -1), generator=g)
    if mask is not None:
        out.masked_fill_(mask.bool(), -1)
    return out.view(torch.uint32) if c["dtype"] == "uint32" else out


# --------------------------------------------------------------------------------------
# prepare and run
# --------------------------------------------------------------------------------------
def _build(api, c, mask):
    return api.Integrator.build(api.Geometry(*_params(c)), (c["ny"], c["nx"]), c["npt"], c["azim"],
                                c["unit"], c["split"], mask)


def prepare(case, seed):
    from paper_1412_6367_gb300 import api, autograd
    dev = torch.device("cuda")
    kind = case["kind"]
    if kind == "multi":
        cs = _instances(case)
        igs = [_build(api, c, None) for c in cs]
        images = [_frames(c, 64 * seed + k, dev, None)[0] for k, c in enumerate(cs)]
        return {"kind": kind, "plan": api.MultiPlan(igs, images)}
    mask = _mask(case, dev)
    frames = _frames(case, seed, dev, mask)
    a = _arrays(case, seed, dev)
    corr = (a["dark"], a["flat"], a["sa"], a["pol"])
    st = {"kind": kind, "api": api, "frames": frames, "corr": corr, "precision": case["precision"],
          "case": case, "mask": mask}
    if kind == "setup":
        return st
    st["ig"] = ig = _build(api, case, mask)
    if kind == "bound":
        ig.set_corrections(*corr)
    elif kind == "host":
        host = torch.empty(frames.shape, dtype=torch.int32 if case["dtype"] == "uint32" else frames.dtype,
                           pin_memory=True)
        host.copy_(frames.view(torch.int32) if case["dtype"] == "uint32" else frames)
        st["frames"] = host.view(frames.dtype)
    elif kind == "grad":
        g = torch.Generator(device=dev).manual_seed(31 * seed + 2)
        shape = (case["azim"], case["npt"]) if case["azim"] else (case["npt"],)
        dt = torch.float64 if case["precision"] == "fp64" else torch.float32
        st["autograd"] = autograd
        st["upstream"] = torch.randn(shape, generator=g, device=dev, dtype=torch.float32).to(dt)
        st["image"] = frames[0].requires_grad_(True)
        flat = corr[1] if corr[1] is not None else torch.ones_like(frames[0])
        st["flat"] = flat.detach().requires_grad_(True)
    return st


def run(state):
    kind, corr = state["kind"], state.get("corr")
    if kind == "frame":
        return tuple(state["ig"].integrate(state["frames"][0], *corr, precision=state["precision"]))
    if kind == "bound":
        return tuple(state["ig"].integrate_batch_bound(state["frames"]))
    if kind == "batch":
        return tuple(state["ig"].integrate_batch(state["frames"], *corr))
    if kind == "variance":
        return state["ig"].variance(state["frames"])
    if kind == "grad":
        I = state["autograd"].integrate(state["image"], state["flat"], state["ig"], corr[0], corr[2], corr[3],
                                        state["precision"])
        gi, gf = torch.autograd.grad(I, (state["image"], state["flat"]), state["upstream"])
        return I, gi, gf
    if kind == "multi":
        return [tuple(r) for r in state["plan"].launch(use_graph=True)]
    if kind == "host":
        return state["ig"].integrate_batch_host(state["frames"], *corr)
    api, c = state["api"], state["case"]
    g = api.Geometry(*_params(c))
    shape = (c["ny"], c["nx"])
    ig = api.Integrator.build(g, shape, c["npt"], c["azim"], c["unit"], c["split"], state["mask"])
    sa, pol = g.solid_angle(*shape), g.polarization(*shape, POL_FACTOR)
    r = ig.integrate(state["frames"][0], corr[0], corr[1], sa, pol)
    return tuple(r) + (sa, pol, ig.radial_axis())


# --------------------------------------------------------------------------------------
# bytes and operations
# --------------------------------------------------------------------------------------
def _entries(c):
    """(matrix entries, unmasked pixels), the entries estimated from a sample of pixels: the
    bins a pixel's extent crosses."""
    dev = torch.device("cpu")
    s = max(1, int(math.sqrt(c["ny"] * c["nx"] / 40000)))
    i = torch.arange(0, c["ny"], s, dtype=torch.float64).unsqueeze(1)
    j = torch.arange(0, c["nx"], s, dtype=torch.float64).unsqueeze(0)
    m = _mask(c, dev)
    ok = torch.ones(i.shape[0], j.shape[1], dtype=torch.bool) if m is None else m[::s, ::s] == 0
    share = float(ok.double().mean())
    pixels = c["ny"] * c["nx"] * share
    if c["split"] == "none":
        return pixels, pixels
    rads, chis = zip(*[_angles(c, i + di, j + dj)[:2] for di, dj in ((0, 0), (0, 1), (1, 1), (1, 0))])
    rads, chis = torch.stack(rads), torch.stack(chis)
    width = float(rads.max() - rads.min()) / c["npt"]
    r = (rads.amax(0) - rads.amin(0)) / width
    n = 1.0 + r
    if c["azim"]:
        d = chis.amax(0) - chis.amin(0)
        d = torch.where(d > 180.0, 360.0 - d, d) / (360.0 / c["azim"])
        n = n + d + (r * d if c["split"] == "bbox" else 0.5 * r * d)
    return pixels * float(n[ok].mean()), pixels


def work(case):
    if case["kind"] == "multi":
        each = [work(dict(c, kind="frame")) for c in _instances(case)]
        return {k: sum(w[k] for w in each) for k in ("bytes", "flops")}
    nnz, pixels = _entries(case)
    rows = case["npt"] * max(1, case["azim"])
    f64 = case["precision"] == "fp64"
    entry = 12 if f64 else 8     # pixel index and weight
    narr = len([k for k in case["corr"].split("+") if k])
    frames = 1 if case["kind"] in ("frame", "grad", "setup") else case["frames"]
    out = rows * (8 if f64 else 4)
    b = frames * pixels * 4 + narr * pixels * 4
    if case["kind"] == "setup":  # the matrix is written once and read once, two corrections written
        return {"bytes": b + 2 * nnz * entry + 2 * case["ny"] * case["nx"] * 4 + 4 * out, "flops": 2.0 * nnz}
    b += nnz * entry + (2 * frames + 2) * out
    fl = 2.0 * nnz * frames
    if case["kind"] == "grad":   # the matrix again for the gradients, two gradient images written
        b += nnz * entry + 2 * case["ny"] * case["nx"] * 4 + 2 * pixels * 4
        fl += 4.0 * nnz
    return {"bytes": b, "flops": fl}


# --------------------------------------------------------------------------------------
# the outputs in 64 bits
# --------------------------------------------------------------------------------------
def _quad_area(x, y, lo, hi, c=None, d=None):
    """Area of straight-edged quadrilaterals (x, y: [n, 4]) with lo <= x <= hi and, if given,
    c <= y <= d: the edges' integrals of y (clamped to [c, d], from c) over the clamped span."""
    s = torch.zeros_like(lo)
    for k in range(4):
        x0, y0, x1, y1 = x[:, k], y[:, k], x[:, (k + 1) % 4], y[:, (k + 1) % 4]
        u, v = torch.minimum(torch.maximum(x0, lo), hi), torch.minimum(torch.maximum(x1, lo), hi)
        flat = x0 == x1
        slope = (y1 - y0) / torch.where(flat, torch.ones_like(x0), x1 - x0)
        yu, yv = y0 + (u - x0) * slope, y0 + (v - x0) * slope
        if c is None:
            mean = 0.5 * (yu + yv)
        else:
            p, q = torch.minimum(yu, yv), torch.maximum(yu, yv)
            span = torch.where(q > p, q - p, torch.ones_like(p))
            under = ((c - p) / span).clamp(0.0, 1.0)
            over = ((q - d) / span).clamp(0.0, 1.0)
            mid = (1.0 - under - over) * (0.5 * (torch.maximum(p, c) + torch.minimum(q, d)) - c)
            mean = over * (d - c) + mid
            mean = torch.where(q <= c, torch.zeros_like(mean), torch.where(p >= d, d - c, mean))
            mean = torch.where((q == p) & (q > c) & (p < d), p - c, mean)
        s = s + torch.where(flat, torch.zeros_like(s), (v - u) * mean)
    return s.abs()


def _box(fmin, fmax, lo, hi, b):
    """Share of [fmin, fmax] that lies in bin b of the bins lo .. hi it crosses."""
    span = torch.where(fmax > fmin, fmax - fmin, torch.ones_like(fmin))
    w = torch.where(b == lo, (lo + 1.0) - fmin, torch.where(b == hi, fmax - hi, torch.ones_like(span))) / span
    return torch.where(lo == hi, torch.ones_like(w), w)


def _expand(counts):
    """(owner of each of sum(counts) candidates, its number within the owner)"""
    own = torch.repeat_interleave(torch.arange(counts.numel(), device=counts.device), counts)
    first = torch.cumsum(counts, 0) - counts
    return own, torch.arange(own.numel(), device=counts.device) - first[own]


def _matrix(c, dev):
    """The bins x pixels matrix in 64 bits (rows, pixels, weights) and the radial range."""
    npt, azim = c["npt"], c["azim"]
    m = _mask(c, dev)
    pix = torch.arange(c["ny"] * c["nx"], device=dev)
    if m is not None:
        pix = pix[m.reshape(-1) == 0]
    pi, pj = pix // c["nx"], pix % c["nx"]
    if c["split"] == "none":
        rad, chi, _, _ = _angles(c, *_grid(c, True, dev))
        x = rad.reshape(-1)[pix]
        lo, hi = x.min(), x.max()
        row = ((x - lo) / ((hi - lo) / npt)).floor().long().clamp_max(npt - 1)
        if azim:
            row = row + npt * (((chi.reshape(-1)[pix] + 180.0) / (360.0 / azim)).floor().long() % azim)
        return row, pix, torch.ones_like(x), float(lo), float(hi)
    rad, chi, _, _ = _angles(c, *_grid(c, False, dev))
    corner = lambda t: torch.stack([t[pi, pj], t[pi, pj + 1], t[pi + 1, pj + 1], t[pi + 1, pj]], 1)  # noqa: E731
    R, X = corner(rad), corner(chi)
    lo, hi = R.min(), R.max()
    F = (R - lo) / ((hi - lo) / npt)
    X = torch.where((X.amax(1) - X.amin(1) > 180.0).unsqueeze(1) & (X < 0), X + 360.0, X)
    centre = X.amax(1) - X.amin(1) > 180.0  # the pixel that holds the beam centre
    fmin, fmax = F.amin(1), F.amax(1)
    b0 = fmin.floor().clamp_max(npt - 1)
    b1 = torch.minimum(torch.maximum(b0, fmax.ceil() - 1), torch.full_like(b0, npt - 1))
    inf = torch.full((1,), 1e30, dtype=torch.float64, device=dev)
    if not azim:
        own, k = _expand((b1 - b0 + 1).long())
        b = b0[own] + k
        w = _box(fmin[own], fmax[own], b0[own], b1[own], b)
        if c["split"] == "full":
            f0 = F[own, :1]
            a = _quad_area(F[own] - f0, X[own] - X[own, :1],
                           torch.where(b == 0, -inf, b - f0[:, 0]), torch.where(b == npt - 1, inf, b + 1 - f0[:, 0]))
            tot = torch.zeros_like(fmin).index_add_(0, own, a)
            use = ~centre & (b0 != b1) & (tot > 0)
            w = torch.where(use[own], a / torch.where(tot > 0, tot, torch.ones_like(tot))[own], w)
        return b.long(), pix[own], w, float(lo), float(hi)
    G = (X + 180.0) / (360.0 / azim)
    gmin, gmax = G.amin(1), G.amax(1)
    g0 = gmin.floor()
    g1 = torch.maximum(g0, gmax.ceil() - 1)
    g0, g1 = torch.where(centre, torch.zeros_like(g0), g0), torch.where(centre, torch.full_like(g1, azim - 1), g1)
    nb, ng = (b1 - b0 + 1).long(), (g1 - g0 + 1).long()
    own, k = _expand(nb * ng)
    b, g = b0[own] + k // ng[own], g0[own] + k % ng[own]
    w = _box(fmin[own], fmax[own], b0[own], b1[own], b)
    wg = torch.where(centre[own], torch.full_like(w, 1.0 / azim), _box(gmin[own], gmax[own], g0[own], g1[own], g))
    w = w * wg
    if c["split"] == "full":
        f0, h0 = F[own, :1], G[own, :1]
        a = _quad_area(F[own] - f0, G[own] - h0, torch.where(b == 0, -inf, b - f0[:, 0]),
                       torch.where(b == npt - 1, inf, b + 1 - f0[:, 0]), g - h0[:, 0], g + 1 - h0[:, 0])
        tot = torch.zeros_like(fmin).index_add_(0, own, a)
        a = torch.where(a > 1e-12 * tot[own], a, torch.zeros_like(a))
        kept = torch.zeros_like(fmin).index_add_(0, own, a)
        use = ~centre & (kept > 0)
        w = torch.where(use[own], a / torch.where(kept > 0, kept, torch.ones_like(kept))[own], w)
    keep = w > 0
    return ((g % azim).long() * npt + b.long())[keep], pix[own][keep], w[keep], float(lo), float(hi)


def _values64(frames, dtype):
    if dtype == "uint32":
        v = frames.view(torch.int32).to(torch.int64)
        return (v & 0xffffffff).double()
    return frames.double()


def _exact_frames(c, seed, dev):
    row, pix, w, lo, hi = _matrix(c, dev)
    rows, npix = c["npt"] * max(1, c["azim"]), c["ny"] * c["nx"]
    order = torch.argsort(row, stable=True)
    row, pix, w = row[order], pix[order], w[order]
    ptr = torch.zeros(rows + 1, dtype=torch.int64, device=dev)
    ptr[1:] = torch.cumsum(torch.bincount(row, minlength=rows), 0)
    A = lambda v: torch.sparse_csr_tensor(ptr, pix, v, (rows, npix))  # noqa: E731
    mask = _mask(c, dev)
    ok = torch.ones(npix, dtype=torch.bool, device=dev) if mask is None else mask.reshape(-1) == 0
    a = _arrays(c, seed, dev)
    if c["kind"] == "setup":
        a["sa"], a["pol"] = _corrections64(c, dev)
    norm = torch.ones(npix, dtype=torch.float64, device=dev)
    for k in ("flat", "sa", "pol"):
        if a[k] is not None:
            norm = norm * a[k].double().reshape(-1)
    raw = _frames(c, seed, dev, mask)
    n = raw.shape[0]
    m = A(w * w if c["kind"] == "variance" else w)
    S = torch.empty((n, rows), dtype=torch.float64, device=dev)
    for f in range(0, n, 16):
        X = _values64(raw[f:f + 16], c["dtype"]).reshape(-1, npix)
        if c["kind"] == "variance":
            X = X.clamp_min(0.0)
        elif a["dark"] is not None:
            X = X - a["dark"].double().reshape(1, -1)
        X = torch.where(ok, X, torch.zeros_like(X))
        S[f:f + 16] = (m @ X.t().contiguous()).t()
    if c["kind"] == "variance":
        return S
    NC = A(w) @ torch.stack([norm, torch.ones_like(norm)], 1)
    N, C = NC[:, 0].contiguous(), NC[:, 1].contiguous()
    I = torch.where(N != 0, S / torch.where(N != 0, N, torch.ones_like(N)), torch.zeros_like(S))
    if c["kind"] == "grad":
        g = torch.Generator(device=dev).manual_seed(31 * seed + 2)
        up = torch.randn((max(1, c["azim"]), c["npt"]), generator=g, device=dev).double().reshape(-1)
        u = torch.where(N != 0, up / torch.where(N != 0, N, torch.ones_like(N)), torch.zeros_like(N))
        gi = torch.zeros(npix, dtype=torch.float64, device=dev).index_add_(0, pix, w * u[row])
        gf = torch.zeros(npix, dtype=torch.float64, device=dev).index_add_(0, pix, w * (u * I[0])[row])
        for k in ("sa", "pol"):
            if a[k] is not None:
                gf = gf * a[k].double().reshape(-1)
        shape = (c["azim"], c["npt"]) if c["azim"] else (c["npt"],)
        return I[0].reshape(shape), gi.reshape(c["ny"], c["nx"]), -gf.reshape(c["ny"], c["nx"])
    if c["kind"] in ("frame", "setup"):
        shape = (c["azim"], c["npt"]) if c["azim"] else (c["npt"],)
        out = tuple(t.reshape(shape) for t in (I[0], S[0], N, C))
        if c["kind"] == "setup":
            axis = lo + (torch.arange(c["npt"], dtype=torch.float64, device=dev) + 0.5) * ((hi - lo) / c["npt"])
            out += (a["sa"], a["pol"], axis)
        return out
    return (I, S) if c["kind"] == "host" else (I, S, N, C)


def exact(case, seed):
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    if case["kind"] == "multi":
        return [_exact_frames(dict(c, corr=""), 64 * seed + k, dev) for k, c in enumerate(_instances(case))]
    return _exact_frames(case, seed, dev)
