"""The calls that a user of this library spends GPU time on, as measurable cases.

Each case is one public entry point (or one FramePipeline / SegmentBatch call) on seeded synthetic
IMX455-like star fields: `prepare` makes what the caller holds before the call (inputs, reference and
calibration frames, plans, weights), `run` is one pass, `exact` is the result in 64 bits where it is
a computed number, written out in torch without the library, and `work` counts the bytes and
operations that one pass cannot do without.

Kinds of case and what they stand for:
  frame      the reduction of one raw frame, raw u16 to source list (FramePipeline.run_fused)
  subtract   difference image and variance with a kernel kept from an earlier fit
  coadd      sigma-clipped mean of a stack of raw frames
  segments   one kernel fit, subtraction and detection per image segment of a batch
  forward    the learned kernel of a frame's stamps
  train      one training step of the learned kernel
  zogy       proper (ZOGY) subtraction of a frame's tiles, PSFs given or kept from the pointing
  proper     proper coaddition of a stack's tiles
  products   background map, low-resolution map and minipix stamping of one calibrated frame
  healpix    resampling of a frame into its HEALPix segments
"""
from __future__ import annotations

import math

import numpy as np
import torch
import torch.nn.functional as F

from paper_2207_14304_gb300 import _binding as B
from paper_2207_14304_gb300.learned import KernelNet
from paper_2207_14304_gb300.pipeline import FramePipeline
from paper_2207_14304_gb300.segments import SegmentBatch
from paper_2207_14304_gb300.synth import pitch_for, segment_origins, segment_sides

FULL_W, FULL_H = 9576, 6388          # IMX455 frame
STAR_DENSITY = 150_000 / (FULL_W * FULL_H)
SIGMAS, DEGREES = (0.7, 1.5, 3.0), (6, 4, 2)
BIAS, READ_NOISE, SAT = 100, 1.7, 65535


# --------------------------------------------------------------------------- cases
def listed():
    return [
        # one 61-Mpix camera frame with a spatially varying 21 x 21 kernel: the headline workload
        dict(name="frame_full", kind="frame", w=FULL_W, h=FULL_H, ksize=21, sdeg=2, grid=20, precision="tf32"),
        # a small cutout frame with a constant kernel: latency and launches
        dict(name="frame_1k", kind="frame", w=1024, h=1024, ksize=11, sdeg=0, grid=8, precision="fp32"),
        # subtraction alone with the pointing's kernel, at a ragged size
        dict(name="subtract_ragged", kind="subtract", w=3001, h=2047, ksize=21, sdeg=2),
        # a 15-minute coadd of 30 s exposures
        dict(name="coadd_30", kind="coadd", w=FULL_W, h=FULL_H, frames=30),
        # a short stack of a ragged cutout
        dict(name="coadd_ragged", kind="coadd", w=2043, h=1501, frames=13),
        # the segments of four cameras, 512 each, 64 to 512 px
        dict(name="segments_4x512", kind="segments", cameras=4, per=512, smin=64, smax=512, ksize=15),
        # the learned kernels of one frame's stamps
        dict(name="forward_400", kind="forward", n=400, precision="bf16_split"),
        # one training step at the default batch
        dict(name="train_512", kind="train", n=512, precision="bf16_split"),
        # a frame's tiles on a new pointing: a PSF pair for every tile
        dict(name="zogy_frame", kind="zogy", w=FULL_W, h=FULL_H, tile=512, per_tile=True, kept=False),
        # a deep coadd by matched filter, one PSF per exposure
        dict(name="proper_30", kind="proper", w=FULL_W, h=FULL_H, frames=30, tile=512, per_tile=False),
        # what is archived of a frame beside the difference
        dict(name="products_full", kind="products", w=FULL_W, h=FULL_H, box=64, filt=3, cell=9, factor=10),
        # a frame into its NSIDE 256 segments
        dict(name="healpix_full", kind="healpix", w=FULL_W, h=FULL_H, dec=30.0, k=9),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["frame", "subtract", "coadd", "segments", "forward", "train", "zogy", "proper", "products",
                       "healpix"])
    w, h = _log_int(rng, 700, FULL_W), _log_int(rng, 700, FULL_H)
    if kind == "frame":
        return dict(kind=kind, w=w, h=h, ksize=rng.choice([11, 21]), sdeg=rng.choice([0, 1, 2]),
                    grid=max(6, min(20, min(w, h) // 160)), precision=rng.choice(["tf32", "fp32", "bf16_split"]))
    if kind == "subtract":
        return dict(kind=kind, w=w, h=h, ksize=rng.choice([7, 9, 11, 15, 21]), sdeg=rng.choice([0, 1, 2]))
    if kind == "coadd":
        n = _log_int(rng, 3, 64)
        return dict(kind=kind, w=w, h=min(h, int(30 * FULL_W * FULL_H / (n * w))), frames=n)
    if kind == "segments":
        smin = rng.randint(40, 120)
        return dict(kind=kind, cameras=1, per=_log_int(rng, 8, 512), smin=smin, smax=rng.randint(smin + 1, 512),
                    ksize=rng.choice([11, 15]))
    if kind == "forward":
        return dict(kind=kind, n=_log_int(rng, 9, 1024), precision=rng.choice(["bf16_split", "bf16", "fp32"]))
    if kind == "train":
        return dict(kind=kind, n=_log_int(rng, 64, 1024), precision=rng.choice(["bf16_split", "bf16", "fp32"]))
    if kind in ("zogy", "proper"):
        tile = rng.choice([256, 512, 1024])
        w, h = max(w, tile + 1), max(h, tile + 1)
        if kind == "zogy":
            return dict(kind=kind, w=w, h=h, tile=tile, per_tile=rng.random() < 0.5, kept=rng.random() < 0.5)
        n = _log_int(rng, 2, 64)
        per_tile = rng.random() < 0.3
        most = FULL_W * FULL_H * 30 / (n * (2.5 if per_tile else 1.0))
        return dict(kind=kind, w=w, h=max(tile + 1, min(h, int(most / w))), frames=n, tile=tile, per_tile=per_tile)
    if kind == "products":
        return dict(kind=kind, w=w, h=h, box=rng.choice([16, 32, 48, 63, 64]), filt=rng.choice([1, 3, 5]),
                    cell=rng.randint(5, 32), factor=rng.randint(4, 16))
    return dict(kind=kind, w=w, h=h, dec=round(rng.uniform(-40.0, 80.0), 2), k=rng.choice([5, 7, 8, 9]))


# --------------------------------------------------------------------------- star fields
def _rand(seed):
    return np.random.RandomState((int(seed) * 1_000_003 + 12_345) % (1 << 31))


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) % (1 << 62))


def _catalog(w, h, seed):
    """Star positions and power-law fluxes (dN/dF ~ F^-1.5 on [1e2, 1e6] electrons)."""
    r = _rand(seed)
    n = max(64, int(STAR_DENSITY * w * h))
    a, b = 1e2 ** -0.5, 1e6 ** -0.5
    return r.uniform(0, w, n), r.uniform(0, h, n), (a + r.uniform(0, 1, n) * (b - a)) ** -2.0


def _deltas(cat, w, h, weight=None, shift=(0.0, 0.0)):
    """[h, w] image holding each star's flux at its nearest pixel (the first of stars that share one)."""
    x, y = np.rint(cat[0] - shift[0]).astype(np.int64), np.rint(cat[1] - shift[1]).astype(np.int64)
    f = cat[2] if weight is None else cat[2] * weight
    ok = (x >= 0) & (y >= 0) & (x < w) & (y < h)
    idx, first = np.unique((y * w + x)[ok], return_index=True)
    img = torch.zeros(h * w, device="cuda")
    img[torch.from_numpy(idx).cuda()] = torch.from_numpy(f[ok][first].astype(np.float32)).cuda()
    return img.view(h, w)


def _blur(img, sigma):
    """Separable Gaussian blur by shifted sums (the same sums in the same order on every run)."""
    r = int(math.ceil(4.5 * sigma))
    t = np.exp(-0.5 * (np.arange(-r, r + 1) / sigma) ** 2)
    t /= t.sum()
    for axis in (0, 1):
        out = torch.zeros_like(img)
        n = img.shape[axis]
        for d, c in zip(range(-r, r + 1), t):
            if abs(d) < n:
                dst = out.narrow(axis, max(d, 0), n - abs(d))
                dst.add_(img.narrow(axis, max(-d, 0), n - abs(d)), alpha=float(c))
        img = out
    return img


def _field_blur(cat, w, h, s0, s1):
    """A PSF that widens from s0 at the centre to s1 at the corners."""
    cx, cy = (w - 1) / 2, (h - 1) / 2
    r2 = np.clip(((cat[0] - cx) ** 2 + (cat[1] - cy) ** 2) / (cx * cx + cy * cy), 0, 1)
    return _blur(_deltas(cat, w, h, 1 - r2), s0) + _blur(_deltas(cat, w, h, r2), s1)


def _noisy(expected, var, g):
    return expected + torch.randn(expected.shape, generator=g, device="cuda") * var.sqrt()


def _pitched(a):
    h, w = a.shape
    p = pitch_for(w)
    if p == w:
        return a.contiguous()
    t = torch.zeros((h, p), dtype=a.dtype, device=a.device)
    t[:, :w] = a
    return t


def _camera(w, h, seed):
    """Dark, flat and bad-pixel map of a camera."""
    g = _gen(seed * 7 + 1)
    dark = torch.full((h, w), 0.5, device="cuda")
    dark += (torch.rand((h, w), generator=g, device="cuda") < 1e-4) * 80.0
    yy = (torch.arange(h, device="cuda") - (h - 1) / 2) / h
    xx = (torch.arange(w, device="cuda") - (w - 1) / 2) / w
    flat = (1 - 0.2 * (yy[:, None] ** 2 + xx[None, :] ** 2)) * (
        1 + 0.01 * torch.randn((h, w), generator=g, device="cuda"))
    bpm = (torch.rand((h, w), generator=g, device="cuda") < 1e-4).to(torch.uint8)
    return dark, flat, bpm


def _raw(expected, cam, g, cosmics=0.0):
    """A raw u16 exposure of the expected electrons."""
    lam = expected * cam[1] + cam[0]
    e = _noisy(lam, lam + READ_NOISE ** 2, g)
    if cosmics:
        hit = torch.rand(e.shape, generator=g, device="cuda") < cosmics
        e += hit * torch.exp(math.log(1e3) + math.log(30.0) * torch.rand(e.shape, generator=g, device="cuda"))
    return (e + BIAS).round_().clamp_(0, 65535).to(torch.int32).to(torch.uint16)


def _psf(sigma, half=15):
    u = np.arange(-half, half + 1)
    g = np.exp(-(u[None, :] ** 2 + u[:, None] ** 2) / (2 * sigma * sigma))
    return (g / g.sum()).astype(np.float32)


def _tiles(w, h, t):
    return [(x, y) for y in range(0, max(h - t, 0) + 1, t) for x in range(0, max(w - t, 0) + 1, t)]


class _Net(KernelNet):
    """A network that lives as long as anything that points into its memory."""

    def __del__(self):
        self.close()


class _State:
    """What the caller holds: attributes, and the library handles given back at the end."""

    def __init__(self, case, **kw):
        self.case, self.closers = case, []
        self.__dict__.update(kw)

    def __del__(self):
        for c in self.closers:
            c()


def _basis(case):
    return B.make_basis(case["ksize"], SIGMAS, DEGREES, case.get("sdeg", 0), case.get("sdeg", 0))


# --------------------------------------------------------------------------- inputs (torch only)
def _frame_inputs(case, seed):
    w, h = case["w"], case["h"]
    cat, g = _catalog(w, h, seed), _gen(seed)
    cam = _camera(w, h, seed)
    raw = _raw(_field_blur(cat, w, h, 1.3, 2.2) + 305.0, cam, g)
    e = _blur(_deltas(cat, w, h), 1.2) + 300.0
    rv = (e + READ_NOISE ** 2) / 30
    return dict(raw=_pitched(raw), dark=_pitched(cam[0]), flat=_pitched(cam[1]), bpm=_pitched(cam[2]),
                ref=_pitched(_noisy(e, rv, g)), ref_var=_pitched(rv))


def _subtract_inputs(case, seed):
    w, h, ks = case["w"], case["h"], case["ksize"]
    cat, g = _catalog(w, h, seed), _gen(seed)
    e = _field_blur(cat, w, h, 1.3, 2.2) + 305.0
    var = e + READ_NOISE ** 2
    r = _blur(_deltas(cat, w, h), 1.2) + 300.0
    rv = (r + READ_NOISE ** 2) / 30
    flags = (torch.rand((h, w), generator=g, device="cuda") < 1e-4).to(torch.uint8)
    # a matching kernel that widens outwards, with a slow gradient, and a background gradient
    terms = [(i, j) for i in range(case["sdeg"] + 1) for j in range(case["sdeg"] + 1 - i)]
    base, wide = _psf(max(0.7, ks / 20), ks // 2), _psf(ks / 9, ks // 2)
    shape = {(0, 0): 0.7 * base + 0.3 * wide, (1, 0): 0.02 * (wide - base), (0, 1): -0.03 * (wide - base),
             (2, 0): 0.2 * (wide - base), (0, 2): 0.15 * (wide - base), (1, 1): 0.01 * (wide - base)}
    amp = 0.002 * _rand(seed + 9).standard_normal((len(terms), ks, ks)).astype(np.float32)
    K = np.stack([shape[t] for t in terms]).astype(np.float32) + amp / ks
    bg = np.array([5.0, 0.3, -0.2, 0.1, 0.05, -0.1][:len(terms)])
    return dict(sci=_pitched(_noisy(e, var, g)), var=_pitched(var), ref=_pitched(_noisy(r, rv, g)),
                ref_var=_pitched(rv), flags=_pitched(flags), K=torch.from_numpy(K.reshape(-1)).cuda(),
                bg=torch.from_numpy(bg).cuda())


def _coadd_inputs(case, seed):
    w, h, n = case["w"], case["h"], case["frames"]
    cat, g = _catalog(w, h, seed), _gen(seed)
    cam = _camera(w, h, seed)
    sh = _rand(seed + 1).uniform(-0.5, 0.5, (n, 2)).astype(np.float32)
    stack = torch.zeros((n, h, pitch_for(w)), dtype=torch.uint16, device="cuda")
    field = _blur(_deltas(cat, w, h), 1.5) + 300.0
    for f in range(n):
        stack[f, :, :w] = _raw(field, cam, g, cosmics=0.01)
    return dict(stack=stack, shifts=torch.from_numpy(sh).cuda(), dark=_pitched(cam[0]), flat=_pitched(cam[1]),
                bpm=_pitched(cam[2]))


def _net_inputs(case, seed):
    """Stamp pairs (science, reference) of one star each, divided by the reference flux, the kernels
    between them, and He-scaled weights with the moments of a training in progress."""
    n, r = case["n"], _rand(seed)
    g = _gen(seed)
    u = torch.arange(21, device="cuda") - 10.0
    col = lambda a: torch.from_numpy(a.astype(np.float32)).cuda()[:, None]  # noqa: E731

    def star(s, cx, cy):
        gx = torch.exp(-0.5 * ((u - cx) / s) ** 2) / (s * math.sqrt(2 * math.pi))
        gy = torch.exp(-0.5 * ((u - cy) / s) ** 2) / (s * math.sqrt(2 * math.pi))
        return gy[:, :, None] * gx[:, None, :]

    cx, cy, s = col(r.uniform(-0.5, 0.5, n)), col(r.uniform(-0.5, 0.5, n)), col(r.uniform(1.1, 3.0, n))
    flux = col(np.exp(r.uniform(math.log(1e3), math.log(3e4), n)))[:, :, None]
    sci, ref = star(s, cx, cy) * flux, star(torch.ones_like(s), cx, cy) * flux
    sci = _noisy(sci, sci + 13.0, g)
    ref = _noisy(ref, (ref + 13.0) / 30, g)
    x = (torch.stack([sci, ref], -1) / flux[..., None]).reshape(n, 441, 2).contiguous()
    z = torch.zeros_like(s)
    target = star(torch.sqrt(s * s - 1.0), z, z).reshape(n, 441).contiguous()
    parts = [r.standard_normal(64) * 1.0, r.standard_normal(32) * 0.05]
    for _ in range(4):
        parts += [r.standard_normal(49 * 1024) * math.sqrt(2 / (49 * 32)), r.standard_normal(32) * 0.05]
    parts += [r.standard_normal(32) * math.sqrt(2 / 32), np.ones(1)]
    p = np.concatenate(parts)
    m, v = r.standard_normal(p.size) * 1e-4, np.exp(r.standard_normal(p.size)) * 1e-8
    dev = lambda a: torch.from_numpy(a.astype(np.float32)).cuda()  # noqa: E731
    return dict(x=x, target=target, params=dev(p), m=dev(m), v=dev(v), step=200, lr=1e-3)


def _zogy_inputs(case, seed):
    w, h, t = case["w"], case["h"], case["tile"]
    cat, g = _catalog(w, h, seed), _gen(seed)
    N = _blur(_deltas(cat, w, h), 1.8)
    R = _blur(_deltas(cat, w, h), 1.2)
    N += torch.randn((h, w), generator=g, device="cuda") * 18.0
    R += torch.randn((h, w), generator=g, device="cuda") * 3.0
    org = _tiles(w, h, t)
    n, r = len(org), _rand(seed + 3)
    rec = np.zeros(n, B.ZOGY_TILE_DTYPE)
    rec["x0"], rec["y0"] = [o[0] for o in org], [o[1] for o in org]
    rec["Fn"], rec["Fr"] = r.uniform(0.8, 1.2, n), r.uniform(0.8, 1.2, n)
    rec["sn"], rec["sr"] = r.uniform(15, 20, n), r.uniform(2.5, 3.5, n)
    m = n if case["per_tile"] else 1
    pn, pr = (np.stack([_psf(s) for s in r.uniform(a, b, m)]) for a, b in ((1.3, 2.2), (1.15, 1.25)))
    return dict(N=_pitched(N), R=_pitched(R), rec=rec, pn=torch.from_numpy(pn).cuda(), pr=torch.from_numpy(pr).cuda())


def _proper_inputs(case, seed):
    w, h, t, n = case["w"], case["h"], case["tile"], case["frames"]
    cat, g, r = _catalog(w, h, seed), _gen(seed), _rand(seed + 4)
    org = _tiles(w, h, t)
    d = _deltas(cat, w, h)
    stack = torch.zeros((n, h, pitch_for(w)), device="cuda")
    sig, scale, noise = r.uniform(1.3, 2.2, n), r.uniform(0.8, 1.2, n), r.uniform(12, 25, n)
    for f in range(n):
        stack[f, :, :w] = _blur(d, float(sig[f])) * float(scale[f])
        stack[f, :, :w] += torch.randn((h, w), generator=g, device="cuda") * float(noise[f])
    if case["per_tile"]:
        psf = np.stack([np.stack([_psf(s * (1 + 0.1 * i / len(org))) for s in sig]) for i in range(len(org))])
    else:
        psf = np.stack([_psf(s) for s in sig])
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).cuda()  # noqa: E731
    return dict(stack=stack, org=torch.tensor(org, dtype=torch.int32, device="cuda"), F=dev(scale), sigma=dev(noise),
                psf=dev(psf))


def _products_inputs(case, seed):
    w, h = case["w"], case["h"]
    cat, g = _catalog(w, h, seed), _gen(seed)
    img = _blur(_deltas(cat, w, h), 1.5) + 300.0
    img += torch.linspace(0, 20, w, device="cuda")[None, :] + torch.randn((h, w), generator=g, device="cuda") * 18.0
    flags = (torch.rand((h, w), generator=g, device="cuda") < 1e-4).to(torch.uint8)
    nt, nd = max(8, int(7.5e-5 * w * h)), max(4, int(6.5e-6 * w * h))
    targets = torch.from_numpy(np.stack([cat[0], cat[1]], 1)[:nt].astype(np.int32)).cuda()
    src = torch.zeros((nd, B.SOURCE_BYTES // 4), dtype=torch.int32, device="cuda")
    src[:, 7] = torch.randint(0, w, (nd,), generator=g, device="cuda", dtype=torch.int32)
    src[:, 8] = torch.randint(0, h, (nd,), generator=g, device="cuda", dtype=torch.int32)
    return dict(img=_pitched(img), flags=_pitched(flags), targets=targets, src=src,
                n_src=torch.tensor([nd], dtype=torch.int32, device="cuda"))


def _healpix_wcs(case):
    return (math.radians(60.0), math.radians(case["dec"]), math.radians(1.38 / 3600.0), 0.1,
            (case["w"] - 1) / 2, (case["h"] - 1) / 2)


def _healpix_inputs(case, seed):
    """A frame and the segments whose centre falls in it, or the one nearest to its centre."""
    w, h = case["w"], case["h"]
    cat, g = _catalog(w, h, seed), _gen(seed)
    img = _blur(_deltas(cat, w, h), 1.5) + 300.0 + torch.randn((h, w), generator=g, device="cuda") * 18.0
    flags = (torch.rand((h, w), generator=g, device="cuda") < 1e-4).to(torch.uint8)
    every = torch.arange(12 * 256 * 256, dtype=torch.int64, device="cuda")
    x, y = _hp_positions(every, 256, 0, _healpix_wcs(case))
    x, y = x.reshape(-1), y.reshape(-1)
    inside = (x >= 0) & (y >= 0) & (x <= w - 1) & (y <= h - 1)
    if not bool(inside.any()):
        d = (x - w / 2) ** 2 + (y - h / 2) ** 2
        inside = torch.arange(every.numel(), device="cuda") == torch.nan_to_num(d, nan=math.inf).argmin()
    return dict(img=_pitched(img), flags=_pitched(flags), segs=every[inside].contiguous())


# --------------------------------------------------------------------------- prepare
def prepare(case, seed):
    kind = case["kind"]
    if kind == "segments":
        return _prepare_segments(case, seed)
    i = globals()[f"_{kind}_inputs" if kind not in ("forward", "train") else "_net_inputs"](case, seed)
    st = _State(case, **i)
    z = lambda *s, dtype=torch.float32: torch.zeros(s, dtype=dtype, device="cuda")  # noqa: E731
    if kind in ("frame", "subtract", "coadd", "products"):
        w, h = case["w"], case["h"]
        p = pitch_for(w)
        st.shape = B.argus_shape(w, h, p)
    if kind == "frame":
        st.calib = B.make_calib(BIAS, st.dark, st.flat, st.bpm, 1.0, READ_NOISE, SAT)
        st.pipe = FramePipeline(w, h, basis=_basis(case), grid=(case["grid"], case["grid"]),
                                precision=case["precision"])
        st.closers.append(st.pipe.close)
    elif kind == "subtract":
        st.ctx = B.argus_create(0, h * p, 16, 64, 1 << 10)
        st.closers.append(lambda c=st.ctx: B.argus_destroy(c))
        st.diff, st.diff_var = z(h, p), z(h, p)
    elif kind == "coadd":
        st.calib = B.make_calib(BIAS, st.dark, st.flat, st.bpm, 1.0, READ_NOISE, SAT)
        st.ctx = B.argus_create(0, h * p, 16, 64, 1 << 10)
        st.closers.append(lambda c=st.ctx: B.argus_destroy(c))
        st.out, st.var, st.used = z(h, p), z(h, p), z(h, p, dtype=torch.uint8)
    elif kind in ("forward", "train"):
        st.net = _Net(max_batch=case["n"], seed=1, precision=case["precision"])
        st.held = st.net.tensors()
        for dst, src in zip(st.held, (st.params, st.m, st.v)):
            dst.copy_(src)
            dst.owner = st.net          # these are views of the library's memory
        B.argus_cnn_set_state(st.net.net, case["precision"], st.step)
        st.y, st.loss = z(case["n"], 441), z(1, dtype=torch.float64)
    elif kind == "zogy":
        n, t = len(st.rec), case["tile"]
        st.shape = B.argus_shape(case["w"], case["h"], st.N.shape[1])
        st.tiles = torch.from_numpy(st.rec.view(np.uint8).copy()).cuda()
        st.plan = B.proper_plan_create(0, t, n)
        st.closers.append(lambda q=st.plan: B.proper_plan_destroy(q))
        st.D, st.S, st.sigma_S = z(n, t, t), z(n, t, t), z(n, dtype=torch.float64)
        if case["kept"]:        # the pointing's first frame gives the PSFs
            _zogy(st, st.pn, st.pr)
    elif kind == "proper":
        n, t = st.org.shape[0], case["tile"]
        st.shape = B.argus_shape(case["w"], case["h"], st.stack.shape[2])
        st.plan = B.proper_plan_create(0, t, n)
        st.closers.append(lambda q=st.plan: B.proper_plan_destroy(q))
        st.S, st.R, st.F_R, st.sigma_S = z(n, t, t), z(n, t, t), z(1, dtype=torch.float64), z(n, dtype=torch.float64)
    elif kind == "products":
        st.ctx = B.argus_create(0, h * p, 16, 64, 1 << 10)
        st.closers.append(lambda c=st.ctx: B.argus_destroy(c))
        cell, f, box = case["cell"], case["factor"], case["box"]
        up = lambda a, b: -(-a // b)  # noqa: E731
        st.mesh, st.map = z(up(h, box), up(w, box), dtype=torch.float64), z(h, p)
        st.low = z(up(h, f), pitch_for(up(w, f)))
        st.cap = 2 * (st.targets.shape[0] + st.src.shape[0])
        st.keep, st.out = z(up(h, cell), up(w, cell), dtype=torch.uint8), z(h, p)
        st.packed, st.index = z(st.cap, cell * cell), z(st.cap, dtype=torch.int32)
        st.n_kept = z(1, dtype=torch.int32)
    elif kind == "healpix":
        m, n = 1 << case["k"], st.segs.numel()
        st.shape = B.argus_shape(case["w"], case["h"], st.img.shape[1])
        st.wcs, st.out, st.cov = _healpix_wcs(case), z(n, m, m), z(n, m, m, dtype=torch.uint8)
    return st


def _prepare_segments(case, seed):
    w, h, per, cams = FULL_W, FULL_H, case["per"], case["cameras"]
    sides = segment_sides(per * cams, 4, case["smin"], case["smax"])
    st = _State(case)
    st.batch = b = SegmentBatch(sides, basis=B.make_basis(case["ksize"], SIGMAS, DEGREES, 0, 0),
                                cfg=B.argus_seg_config(128, 1, 8, 0), src_cap=1 << 16)
    st.closers.append(b.close)
    for c in range(cams):
        cat, g = _catalog(w, h, seed * 64 + c), _gen(seed * 64 + c)
        e = _field_blur(cat, w, h, 1.3, 2.2) + 305.0
        var = e + READ_NOISE ** 2
        r = _blur(_deltas(cat, w, h), 1.2) + 300.0
        rv = (r + READ_NOISE ** 2) / 30
        fl = (torch.rand((h, w), generator=g, device="cuda") < 1e-4).to(torch.uint8)
        src = (_noisy(e, var, g), var, _noisy(r, rv, g), rv, fl)
        own = sides[c * per:(c + 1) * per]
        for j, ((x0, y0), s) in enumerate(zip(segment_origins(own, w, h, seed % (1 << 31) + c), own)):
            for dst, a in zip((b.sci, b.var, b.ref, b.ref_var, b.flags), src):
                b.view(dst, c * per + j).copy_(a[y0:y0 + s, x0:x0 + s])
    st.K = torch.zeros((b.n, case["ksize"] ** 2), device="cuda")
    st.bg = torch.zeros(b.n, dtype=torch.float64, device="cuda")
    return st


# --------------------------------------------------------------------------- run
def _zogy(st, pn, pr):
    B.argus_zogy(st.plan, st.N, st.R, st.shape, st.tiles, len(st.rec), pn, pr, 31, 1e-8, st.D, st.S, None, st.sigma_S,
                 psf_per_tile=st.case["per_tile"])


def _sources(buf):
    """The source records as their five measured and four whole fields."""
    return [buf.view(torch.float32).view(-1, 9)[:, :5], buf.view(torch.int32).view(-1, 9)[:, 5:]]


def run(st):
    c, kind = st.case, st.case["kind"]
    if kind == "frame":
        p = st.pipe
        p.run_fused(st.raw, st.calib, st.ref, st.ref_var)
        # the coefficients themselves are those of a nearly degenerate basis: K and bg say what they mean
        return {"img": p.img, "var": p.var, "flags": p.flags, "centers": p.centers, "n_stamps": p.n_stamps, "K": p.K,
                "bg": p.bg, "diff": p.diff, "diff_var": p.diff_var, "mask": p.mask, "sources": _sources(p.sources),
                "n_found": p.n_found}
    if kind == "subtract":
        B.argus_subtract(st.ctx, st.sci, st.var, st.ref, st.ref_var, st.flags, st.shape, c["w"], c["h"], 0, 0,
                         c["ksize"], c["sdeg"], st.K, c["sdeg"], st.bg, st.diff, st.diff_var)
        return [st.diff, st.diff_var]
    if kind == "coadd":
        B.argus_coadd(st.ctx, st.stack, c["frames"], st.shape, st.shifts, st.calib, 3.0, 5, st.out, st.var, st.used)
        return [st.out, st.var, st.used]
    if kind == "segments":
        b = st.batch
        b.run(use_graph=True)
        B.argus_segments_kernels(b.plan, st.K, st.bg)
        return {"K": st.K, "bg": st.bg, "diff": b.diff, "diff_var": b.diff_var, "mask": b.mask,
                "sources": _sources(b.sources), "n_found": b.n_found}
    if kind == "forward":
        return [st.net.forward(st.x, st.y)]
    if kind == "train":
        B.argus_cnn_train_step(st.net.net, st.x, st.target, c["n"], st.lr, st.loss)
        return [st.loss, *st.held]
    if kind == "zogy":
        _zogy(st, *((None, None) if c["kept"] else (st.pn, st.pr)))
        return [st.D, st.S, st.sigma_S]
    if kind == "proper":
        B.argus_proper_coadd(st.plan, st.stack, c["frames"], st.shape, st.org, st.org.shape[0], st.F, st.sigma, st.psf,
                             31, 1e-8, st.S, st.R, None, st.F_R, st.sigma_S, psf_per_tile=c["per_tile"])
        return [st.S, st.R, st.F_R, st.sigma_S]
    if kind == "products":
        B.argus_background(st.ctx, st.img, st.flags, st.shape, c["box"], c["filt"], 0.5, st.mesh, st.map)
        B.argus_lowres(st.ctx, st.img, st.flags, st.shape, c["factor"], st.low, st.low.shape[1])
        B.argus_minipix(st.ctx, st.img, st.shape, c["cell"], st.targets, st.targets.shape[0], st.src, st.n_src,
                        st.src.shape[0], st.keep, st.out, st.packed, st.index, st.cap, st.n_kept)
        return {"mesh": st.mesh, "map": st.map, "low": st.low, "keep": st.keep, "out": st.out, "packed": st.packed,
                "index": st.index, "n_kept": st.n_kept}
    B.argus_healpix_resample(st.img, st.flags, st.shape, st.wcs, 256, c["k"], st.segs, st.segs.numel(), st.out, st.cov)
    return [st.out, st.cov]


# --------------------------------------------------------------------------- exact
def exact(case, seed):
    kind = case["kind"]
    if kind == "segments":
        return None
    i = globals()[f"_{kind}_inputs" if kind not in ("forward", "train") else "_net_inputs"](case, seed)
    return globals()[f"_exact_{kind}"](case, i)


def _calibrated(raw, i):
    """(value, variance, unusable) of raw frames in 64 bits."""
    n = raw.to(torch.int32).double() - BIAS
    flat = i["flat"].double()
    none = ~((flat > 0) & torch.isfinite(flat))
    flat = torch.where(none, 1.0, flat)
    img = torch.where(none, 0.0, (n - i["dark"].double()) / flat)
    var = torch.where(none, 0.0, (n.clamp(min=0) + float(np.float32(READ_NOISE)) ** 2) / flat ** 2)
    return img, var, none | (i["bpm"] != 0) | (raw.to(torch.int32) >= SAT)


def _exact_frame(case, i):
    img, var, _ = _calibrated(i["raw"], i)
    img[:, case["w"]:] = 0
    var[:, case["w"]:] = 0
    return {"img": img, "var": var}


def _poly(case, x, y):
    """Spatial terms at frame positions x [n], y [m]: [terms, m, n]."""
    xt = (2 * x - (case["w"] - 1)) / (case["w"] - 1)
    yt = (2 * y - (case["h"] - 1)) / (case["h"] - 1)
    d = case["sdeg"]
    return torch.stack([yt[:, None] ** j * xt[None, :] ** i for i in range(d + 1) for j in range(d + 1 - i)])


def _exact_subtract(case, i):
    w, h, ks = case["w"], case["h"], case["ksize"]
    r = ks // 2
    sci, var, ref, rv = (i[k][:, :w].double() for k in ("sci", "var", "ref", "ref_var"))
    K, bg = i["K"].double().view(-1, ks, ks), i["bg"]
    px, py = torch.arange(w, device="cuda").double(), torch.arange(h, device="cuda").double()
    diff, dv = sci.clone(), var.clone()
    for y0 in range(0, h, 128):                      # rows of tiles, as the variance's kernels are per tile
        y1 = min(h, y0 + 128)
        terms = _poly(case, px, py[y0:y1])
        rows = F.pad(ref, (r, r, r, r))[y0:y1 + 2 * r]
        win = rows.unfold(1, ks, 1)                  # [rows, w, ks]; out(x) = sum_u K(u) ref(x - u)
        conv = torch.zeros((len(K), y1 - y0, w), dtype=torch.float64, device="cuda")
        for v in range(ks):
            conv += torch.einsum("ywu,ku->kyw", win[v:v + y1 - y0], K[:, ks - 1 - v].flip(-1))
        diff[y0:y1] -= (terms * (conv + bg[:, None, None])).sum(0)
        rows = F.pad(rv, (r, r, r, r))[y0:y1 + 2 * r].unfold(1, ks, 1)
        yc = torch.full((1,), y0 + 63.5, dtype=torch.float64, device="cuda")
        for x0 in range(0, w, 128):
            x1 = min(w, x0 + 128)
            xc = torch.full((1,), x0 + 63.5, dtype=torch.float64, device="cuda")
            kc2 = (_poly(case, xc, yc)[:, 0, 0][:, None, None] * K).sum(0) ** 2
            for v in range(ks):
                dv[y0:y1, x0:x1] += rows[v:v + y1 - y0, x0:x1] @ kc2[ks - 1 - v].flip(-1)
    keep = i["flags"][:, :w] == 0
    keep[:r] = keep[h - r:] = False
    keep[:, :r] = keep[:, w - r:] = False
    pad = i["sci"].shape[1] - w
    return [F.pad(torch.where(keep, diff, 0.0), (0, pad)), F.pad(torch.where(keep, dv, 0.0), (0, pad))]


def _exact_coadd(case, i):
    w, h, n = case["w"], case["h"], case["frames"]
    p = i["stack"].shape[2]
    out, ovar = (torch.zeros((h, p), dtype=torch.float64, device="cuda") for _ in range(2))
    sh = i["shifts"].double().cpu().numpy()
    nan, inf = math.nan, math.inf
    step = max(8, int(2.5e7 / (n * w)))
    for y0 in range(0, h, step):
        y1 = min(h, y0 + step)
        a, b = max(0, y0 - 1), min(h, y1 + 2)        # shifts stay within a pixel
        cal = {k: i[k][a:b, :w] for k in ("dark", "flat", "bpm")}
        vals, vars_ = [], []
        for f in range(n):
            v, q, bad = _calibrated(i["stack"][f, a:b, :w], cal)
            v = F.pad(torch.where(bad, nan, v), (1, 2, 1, 2), value=nan)
            q = F.pad(q, (1, 2, 1, 2))
            ix, iy = math.floor(sh[f, 0]), math.floor(sh[f, 1])
            fx, fy = float(np.float32(sh[f, 0] - ix)), float(np.float32(sh[f, 1] - iy))
            r0 = y0 - a + 1 + iy
            at = lambda t, j, k: t[r0 + j:r0 + j + y1 - y0, 1 + ix + k:1 + ix + k + w]  # noqa: E731
            v00, v01, v10, v11 = (at(v, j, k) for j in (0, 1) for k in (0, 1))
            if fx == 0:
                v01, v11 = v00, v10
            if fy == 0:
                v10, v11 = v00, v01
            top, bot = v00 + fx * (v01 - v00), v10 + fx * (v11 - v10)
            vals.append(top + fy * (bot - top))
            vars_.append(((1 - fx) * (1 - fy)) ** 2 * at(q, 0, 0) + (fx * (1 - fy)) ** 2 * at(q, 0, 1)
                         + ((1 - fx) * fy) ** 2 * at(q, 1, 0) + (fx * fy) ** 2 * at(q, 1, 1))
        V, Q = torch.stack(vals), torch.stack(vars_)
        S = torch.where(torch.isfinite(V), V, inf).sort(0).values
        k = torch.arange(n, device="cuda")[:, None, None]
        lo, hi = torch.zeros_like(S[0]).long(), torch.isfinite(S).sum(0)     # the samples kept: S[lo:hi]
        for it in range(6):
            m = hi - lo
            mid = [S.gather(0, (lo + q).clamp(0, n - 1)[None])[0] for q in ((m - 1) // 2, m // 2)]
            c = torch.where(m > 0, 0.5 * (mid[0] + mid[1]), 0.0)
            d = torch.where((k >= lo) & (k < hi), S - c, 0.0)
            mean = d.sum(0) / m.clamp(min=1)
            if it == 5:
                break
            sd = (torch.where((k >= lo) & (k < hi), (d - mean) ** 2, 0.0).sum(0) / m.clamp(min=1)).sqrt()
            low, high = (d < -3.0 * sd).sum(0), (d > 3.0 * sd).sum(0)
            some = low + high < m
            lo, hi = lo + low * some, hi - high * some
        first, last = (S.gather(0, q.clamp(0, n - 1)[None])[0] for q in (lo, hi - 1))
        ok = (V >= first) & (V <= last) & (m > 0)
        mm = m.clamp(min=1).double()
        out[y0:y1, :w] = torch.where(m > 0, c + mean, 0.0)
        ovar[y0:y1, :w] = torch.where(m > 0, torch.where(ok, Q, 0.0).sum(0) / mm ** 2, 0.0)
    return [out, ovar, None]


def _net_forward(p, x):
    n = x.shape[0]
    at = 0

    def take(*s):
        nonlocal at
        k = math.prod(s)
        at += k
        return p[at - k:at].view(*s)

    w1, b1 = take(32, 2), take(32)
    a = (x @ w1.T + b1).transpose(1, 2).reshape(n, 32, 21, 21)
    for _ in range(4):
        w, b = take(7, 7, 32, 32), take(32)
        a = F.relu(F.conv2d(a, w.permute(3, 2, 0, 1), b, padding=3))
    w6, b6 = take(32), take(1)
    return ((a * w6[:, None, None]).sum(1).reshape(n, 441) + b6) / 441


def _used_weights(case, i):
    return (i["params"] if case["precision"] == "fp32" else i["params"].bfloat16()).double()


def _exact_forward(case, i):
    p = _used_weights(case, i)
    return [torch.cat([_net_forward(p, i["x"][s:s + 64].double()) for s in range(0, case["n"], 64)])]


def _exact_train(case, i):
    p = _used_weights(case, i).requires_grad_(True)
    n, loss, grad = case["n"], 0.0, torch.zeros_like(p)
    for s in range(0, n, 64):
        part = (_net_forward(p, i["x"][s:s + 64].double()) - i["target"][s:s + 64].double()).square().sum() / (n * 441)
        grad += torch.autograd.grad(part, p)[0]
        loss += float(part.detach())
    m = 0.9 * i["m"].double() + 0.1 * grad
    v = 0.999 * i["v"].double() + 0.001 * grad ** 2
    t = i["step"] + 1
    new = i["params"].double() - i["lr"] * (m / (1 - 0.9 ** t)) / ((v / (1 - 0.999 ** t)).sqrt() + 1e-8)
    return [torch.tensor([loss], dtype=torch.float64, device="cuda"), new, m, v]


def _tile_of(img, w, x0, y0, t):
    a = img[y0:y0 + t, x0:min(x0 + t, w)].double()
    return F.pad(a, (0, t - a.shape[1], 0, t - a.shape[0]))


def _psf_hat(psf, t):
    k = psf.shape[-1]
    p = F.pad(psf.double(), (0, t - k, 0, t - k)).roll((-(k // 2), -(k // 2)), (-2, -1))
    return torch.fft.fft2(p)


def _exact_zogy(case, i):
    t, w, rec = case["tile"], case["w"], i["rec"]
    D, S, sig = [], [], []
    for k in range(len(rec)):
        q = 0 if not case["per_tile"] else k
        Pn, Pr = _psf_hat(i["pn"][q], t), _psf_hat(i["pr"][q], t)
        x0, y0 = int(rec["x0"][k]), int(rec["y0"][k])
        Fn, Fr, sn, sr = (float(rec[c][k]) for c in ("Fn", "Fr", "sn", "sr"))
        N, R = (torch.fft.fft2(_tile_of(i[a], w, x0, y0, t)) for a in ("N", "R"))
        den = torch.sqrt((sn * Fr) ** 2 * Pr.abs() ** 2 + (sr * Fn) ** 2 * Pn.abs() ** 2)
        inv = torch.where(torch.maximum(Pn.abs(), Pr.abs()) < 1e-8, 0.0, 1 / den)
        Dh = (Fr * Pr * N - Fn * Pn * R) * inv
        FD = Fr * Fn / math.sqrt((sn * Fr) ** 2 + (sr * Fn) ** 2)
        PD = Fr * Fn * Pr * Pn * inv / FD
        D.append(torch.fft.ifft2(Dh).real)
        S.append(torch.fft.ifft2(FD * Dh * PD.conj()).real)
        sig.append(FD * torch.fft.ifft2(PD).real.square().sum().sqrt())
    return [torch.stack(D), torch.stack(S), torch.stack(sig)]


def _exact_proper(case, i):
    t, w, org = case["tile"], case["w"], i["org"].cpu().tolist()
    Fj, sj = i["F"].double().cpu().tolist(), i["sigma"].double().cpu().tolist()
    S, R, sig = [], [], []
    shared = None if case["per_tile"] else [_psf_hat(p, t) for p in i["psf"]]
    for k, (x0, y0) in enumerate(org):
        Sh = torch.zeros((t, t), dtype=torch.complex128, device="cuda")
        den2, top, var = torch.zeros((t, t), dtype=torch.float64, device="cuda"), 0.0, 0.0
        for j, (f, s) in enumerate(zip(Fj, sj)):
            P = _psf_hat(i["psf"][k, j], t) if shared is None else shared[j]
            Sh += (f / (s * s)) * P.conj() * torch.fft.fft2(_tile_of(i["stack"][j], w, x0, y0, t))
            den2 += (f / s) ** 2 * P.abs() ** 2
            top = torch.maximum(P.abs(), top) if j else P.abs()
            p = (i["psf"][k, j] if shared is None else i["psf"][j]).double()
            var = var + (f / s) ** 2 * (p * p).sum()
        S.append(torch.fft.ifft2(Sh).real)
        R.append(torch.fft.ifft2(torch.where(top < 1e-8, 0.0, Sh / den2.sqrt())).real)
        sig.append(var.sqrt())
    FR = math.sqrt(sum((f / s) ** 2 for f, s in zip(Fj, sj)))
    return [torch.stack(S), torch.stack(R), torch.tensor([FR], dtype=torch.float64, device="cuda"), torch.stack(sig)]


def _median(v, ok):
    """Median over the last axis of the values that are ok, NaN where none is."""
    s = torch.where(ok, v, math.inf).sort(-1).values
    n = ok.sum(-1)
    lo = s.gather(-1, ((n - 1).clamp(min=0) // 2)[..., None])[..., 0]
    hi = s.gather(-1, (n // 2).clamp(max=v.shape[-1] - 1)[..., None])[..., 0]
    return torch.where(n > 0, 0.5 * (lo + hi), math.nan)


def _exact_products(case, i):
    w, h, box, filt, f, cell = (case[k] for k in ("w", "h", "box", "filt", "factor", "cell"))
    img, ok = i["img"][:, :w], i["flags"][:, :w] == 0
    pw = i["img"].shape[1]

    def blocks(a, b, value):
        a = F.pad(a, (0, -w % b, 0, -h % b), value=value)
        return a.view(a.shape[0] // b, b, a.shape[1] // b, b).permute(0, 2, 1, 3).reshape(
            a.shape[0] // b, a.shape[1] // b, b * b)

    mask = blocks(ok.to(torch.uint8), box, 0) != 0
    there = blocks(torch.ones_like(ok, dtype=torch.uint8), box, 0).sum(-1)
    med = torch.stack([_median(a.double(), m) for a, m in zip(blocks(img, box, 0.0), mask)])
    med = torch.where(mask.sum(-1) >= 0.5 * there, med, math.nan)
    e = F.pad(med, (filt // 2,) * 4, value=math.nan).unfold(0, filt, 1).unfold(1, filt, 1).reshape(*med.shape, -1)
    have = med[torch.isfinite(med)]
    fill = _median(have, torch.ones_like(have, dtype=torch.bool)) if have.numel() else torch.zeros(1).cuda()
    mesh = _median(e, torch.isfinite(e))
    mesh = torch.where(torch.isnan(mesh), fill, mesh)

    def axis(n):
        a = torch.arange(0, n, box, device="cuda").double()
        c = (a + torch.clamp(a + box, max=n) - 1) / 2
        p = torch.arange(n, device="cuda").double()
        if c.numel() == 1:
            return torch.zeros(n, dtype=torch.int64, device="cuda"), torch.zeros_like(p).long(), torch.zeros_like(p)
        k = (torch.searchsorted(c, p, right=True) - 1).clamp(0, c.numel() - 2)
        return k, k + 1, ((p - c[k]) / (c[k + 1] - c[k])).clamp(0, 1)

    (x0, x1, tx), (y0, y1, ty) = axis(w), axis(h)
    bmap = torch.zeros((h, pw), dtype=torch.float64, device="cuda")
    top, bot = (mesh[k][:, x0] + (mesh[k][:, x1] - mesh[k][:, x0]) * tx for k in (y0, y1))
    bmap[:, :w] = top + (bot - top) * ty[:, None]
    sums = torch.where(ok, img, 0.0)
    cnt = blocks(ok.to(torch.uint8), f, 0).sum(-1)
    low = torch.zeros((-(-h // f), pitch_for(-(-w // f))), dtype=torch.float64, device="cuda")
    low[:, :cnt.shape[1]] = torch.where(cnt > 0, blocks(sums, f, 0.0).double().sum(-1) / cnt.clamp(min=1), 0.0)
    at = torch.cat([i["targets"], i["src"][:, 7:9]]).long()
    at = at[(at[:, 0] >= 0) & (at[:, 1] >= 0) & (at[:, 0] < w) & (at[:, 1] < h)] // cell
    keep = torch.zeros((-(-h // cell), -(-w // cell)), dtype=torch.bool, device="cuda")
    keep[at[:, 1], at[:, 0]] = True
    out = torch.zeros((h, pw), dtype=torch.float64, device="cuda")
    big = keep.repeat_interleave(cell, 0)[:h].repeat_interleave(cell, 1)[:, :w]
    out[:, :w] = torch.where(big, img, 0.0)
    cells = keep.flatten().nonzero()[:, 0]
    packed = torch.zeros((2 * (i["targets"].shape[0] + i["src"].shape[0]), cell * cell), dtype=torch.float64,
                         device="cuda")
    packed[:cells.numel()] = blocks(img, cell, 0.0).flatten(0, 1)[cells].double()
    return {"mesh": mesh, "map": bmap, "low": low, "out": out, "packed": packed}


def _hp_positions(segs, nside, k, wcs):
    """Frame positions of the pixel centres of nested segments: x, y of [n, 2^k, 2^k] (NaN behind)."""
    face = segs // (nside * nside)
    sub = segs - face * nside * nside
    X, Y = torch.zeros_like(segs), torch.zeros_like(segs)
    for b in range(int(math.log2(nside)) + 1):
        X |= ((sub >> (2 * b)) & 1) << b
        Y |= ((sub >> (2 * b + 1)) & 1) << b
    m, n = 1 << k, nside << k
    g = torch.arange(m, device="cuda")
    ix, iy = (X[:, None, None] << k) + g[None, None, :], (Y[:, None, None] << k) + g[None, :, None]
    face = face[:, None, None]
    jr = (2 + face // 4) * n - ix - iy - 1
    pl = torch.where((face >= 4) & (face < 8), 2 * (face % 4), 2 * (face % 4) + 1)
    north, south = jr < n, jr > 3 * n
    nr = torch.where(north, jr, torch.where(south, 4 * n - jr, n)).double()
    cap = nr * nr / (3.0 * n * n)
    z = torch.where(north, 1 - cap, torch.where(south, cap - 1, (2 * n - jr).double() * 2 / (3.0 * n)))
    s = torch.where(north | south, torch.sqrt(cap * (2 - cap)), torch.sqrt((1 - z) * (1 + z)))
    phi = (pl * nr + (ix - iy).double()) / nr * (math.pi / 4)      # pixel centres lie on this straight line
    v = (s * torch.cos(phi), s * torch.sin(phi), z)
    al, de, scale, rot, cx, cy = wcs
    ca, sa, cd, sd = math.cos(al), math.sin(al), math.cos(de), math.sin(de)
    dot = lambda a: v[0] * a[0] + v[1] * a[1] + v[2] * a[2]  # noqa: E731
    d = dot((cd * ca, cd * sa, sd))
    d = torch.where(d > 0, d, math.nan)
    xi, eta = dot((-sa, ca, 0.0)) / d, dot((-sd * ca, -sd * sa, cd)) / d
    cr, sr = math.cos(rot), math.sin(rot)
    return cx + (cr * xi + sr * eta) / scale, cy + (-sr * xi + cr * eta) / scale


def _exact_healpix(case, i):
    w, h = case["w"], case["h"]
    img = torch.where(i["flags"] == 0, i["img"].double(), math.nan)
    out = []
    for s in i["segs"].split(8):
        x, y = _hp_positions(s, 256, case["k"], _healpix_wcs(case))
        inside = (x >= 0) & (y >= 0) & (x <= w - 1) & (y <= h - 1)
        x, y = torch.where(inside, x, 0.0), torch.where(inside, y, 0.0)
        x0, y0 = x.floor().long(), y.floor().long()
        tx, ty = x - x0, y - y0
        x1, y1 = torch.where(tx > 0, x0 + 1, x0), torch.where(ty > 0, y0 + 1, y0)
        top, bot = (img[r, x0] + tx * (img[r, x1] - img[r, x0]) for r in (y0, y1))
        v = top + ty * (bot - top)
        out.append(torch.where(inside & torch.isfinite(v), v, 0.0))
    return [torch.cat(out), None]


# --------------------------------------------------------------------------- work
def work(case):
    kind, npx = case["kind"], float(case.get("w", 0) * case.get("h", 0))
    nb = sum((d + 1) * (d + 2) // 2 for d in DEGREES)
    if kind in ("frame", "subtract"):
        ks, d = case["ksize"], case["sdeg"]
        terms = (d + 1) * (d + 2) // 2
        conv = 2.0 * (terms + 1) * ks * ks * npx
        if kind == "subtract":
            return {"bytes": 25.0 * npx, "flops": conv}      # 4 float images and flags in, 2 float images out
        nc, rows = 1 + (nb - 1) * terms + terms, case["grid"] ** 2 * 441.0
        # raw, dark, flat, bad pixels, reference and its variance in; img, var, flags, D, V_D, mask out
        return {"bytes": 37.0 * npx, "flops": conv + rows * (2.0 * nb * ks * ks + nc * (nc + 1.0))}
    if kind == "coadd":
        n = case["frames"]                                   # calibration, sample (value and variance), clip
        return {"bytes": (2.0 * n + 18) * npx, "flops": (8.0 + 20 + 15) * n * npx}
    if kind == "segments":
        lo, hi = math.log(case["smin"]), math.log(case["smax"])
        px = case["cameras"] * case["per"] * (math.exp(2 * hi) - math.exp(2 * lo)) / (2 * (hi - lo))
        return {"bytes": 26.0 * px, "flops": px * (2.0 * (nb + 2) * case["ksize"] ** 2 + (nb + 2) * (nb + 3.0))}
    if kind in ("forward", "train"):
        n = float(case["n"])
        f = n * 441 * (2 * 4 * 49 * 1024 + 4 * 64)
        if kind == "forward":
            return {"bytes": n * 441 * 12 + 4.0 * 200_961, "flops": f}
        return {"bytes": n * 441 * 12 + 24.0 * 200_961, "flops": 3 * f}
    if kind in ("zogy", "proper"):
        t, n = case["tile"], len(_tiles(case["w"], case["h"], case["tile"]))
        fft = 5.0 * t * t * math.log2(t * t)
        if kind == "zogy":                                   # two real images in, two out, PSFs beside them
            k = 2 if case["kept"] else 2 + (1 if case["per_tile"] else 1.0 / n)
            return {"bytes": 16.0 * n * t * t, "flops": n * (k * fft + 60.0 * t * t)}
        j = case["frames"]
        k = j / 2 + 1 + (j / 2 if case["per_tile"] else j / 2 / n)
        return {"bytes": (4.0 * j + 8) * n * t * t, "flops": n * (k * fft + 20.0 * j * t * t)}
    if kind == "products":                                   # three calls: each reads the frame, two write one
        return {"bytes": (5.0 + 4) * npx + 5.0 * npx + 4 * npx, "flops": 10.0 * npx}
    m = 1 << case["k"]
    n = max(1.0, npx * (1.38 / 3600) ** 2 / (4 * math.pi * (180 / math.pi) ** 2 / (12 * 256 * 256)))
    return {"bytes": 5.0 * n * m * m + 5.0 * npx, "flops": 60.0 * n * m * m}
