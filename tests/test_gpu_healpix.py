"""HEALPix segmentation on the GPU (Sec. 3.3; Table 2 GPU stage "Image
segmentation and resampling to HEALPix grid") against the FP64 oracle:
coverage bit-exact, values within 4 ulps of the largest frame value, on both
the exact per-pixel path (k < 6, polar-cap rows) and the row path (k >= 6 in
the equatorial belt).

The kernel has not run on a GPU yet, so the file is skipped until it has.
"""
import math

import numpy as np
import pytest
import torch

from paper_2207_14304_gb300 import _binding as B
from paper_2207_14304_gb300.synth import pitch_for
from tests.gpu_helpers import F32_EPS, dev_pitched

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    B.load()


@pytest.mark.parametrize("nside_seg,k,delta0", [(64, 4, 0.4), (256, 6, -0.3), (32, 5, 1.45), (256, 9, 0.2),
                                               (128, 7, 1.1)])
def test_healpix_resample_parity(ora, nside_seg, k, delta0):
    from oracle import healpix as hp
    rng = np.random.default_rng(nside_seg + k)
    w, h = 900, 700
    scale = 1.2 * math.sqrt(4 * math.pi / (12.0 * (nside_seg << k) ** 2))
    wcs = (2.1, delta0, scale, -0.4, (w - 1) / 2, (h - 1) / 2)
    yy, xx = np.mgrid[0:h, 0:w]
    frame = (300 + 0.05 * xx - 0.02 * yy + rng.normal(0, 10, (h, w))).astype(np.float32)
    frame.flat[11::701] = np.nan
    fl = (rng.random((h, w)) < 0.01).astype(np.uint8)
    p = np.arange(12 * nside_seg * nside_seg)
    ix, iy, f = hp.nest2xyf(p, nside_seg)
    x, y = hp.gnomonic(hp.xyf2vec(ix, iy, f, nside_seg), *wcs)
    near = p[np.isfinite(x) & (x > -20) & (y > -20) & (x < w + 20) & (y < h + 20)]
    segs = rng.choice(near, size=min(8, near.size), replace=False).astype(np.int64)
    m = 1 << k
    out = torch.full((segs.size, m, m), -7.0, device="cuda")
    cov = torch.full((segs.size, m, m), 7, dtype=torch.uint8, device="cuda")
    B.argus_healpix_resample(dev_pitched(frame), dev_pitched(fl), B.argus_shape(w, h, pitch_for(w)), wcs,
                             nside_seg, k, torch.from_numpy(segs).cuda(), segs.size, out, cov)
    torch.cuda.synchronize()
    out, cov = out.cpu().numpy(), cov.cpu().numpy()
    tol = 4 * F32_EPS * float(np.nanmax(np.abs(frame)))
    for i, s in enumerate(segs):
        o, oc = hp.resample_segment(frame, fl, int(s), nside_seg, k, wcs)
        np.testing.assert_array_equal(cov[i], oc)
        assert np.abs(out[i] - o).max() <= tol


@pytest.mark.parametrize("nside_seg,k,delta0,step,rot", [(256, 6, 0.3, 1.0, 0.8),     # staged, axes near 45 degrees
                                                         (64, 7, -0.2, 6.0, 0.0),     # rectangles too large to stage
                                                         (128, 7, 0.7297, 1.1, 0.3),  # the belt's edge inside the patches
                                                         (256, 8, 0.1, 0.2, -2.0)])   # several image pixels per frame pixel
def test_healpix_patches(ora, nside_seg, k, delta0, step, rot):
    """The patch path's forms (staged and gathered pixels, halves across the belt's edge, segments
    hanging off the frame, values beyond FP32's differences) at the bars of the parity test; `step` is the
    image's pixel in frame pixels."""
    from oracle import healpix as hp
    rng = np.random.default_rng(nside_seg + k)
    w, h = 333, 287
    scale = math.sqrt(4 * math.pi / (12.0 * (nside_seg << k) ** 2)) / step
    wcs = (0.9, delta0, scale, rot, (w - 1) / 2, (h - 1) / 2)
    frame = (300 + rng.normal(0, 10, (h, w))).astype(np.float32)
    frame.flat[11::701] = np.nan
    frame.flat[13::997] = -np.inf
    fl = (rng.random((h, w)) < 0.01).astype(np.uint8)
    p = np.arange(12 * nside_seg * nside_seg)
    ix, iy, f = hp.nest2xyf(p, nside_seg)
    x, y = hp.gnomonic(hp.xyf2vec(ix, iy, f, nside_seg), *wcs)
    d = np.where(np.isfinite(x), (x - w / 2) ** 2 + (y - h / 2) ** 2, np.inf)
    segs = np.concatenate([p[np.argsort(d)[:4]], [12 * nside_seg * nside_seg]]).astype(np.int64)
    m = 1 << k
    for big in (False, True):
        if big:
            frame[::3, ::2] = 3.0e38
            frame[1::3, ::2] = -3.0e38
        out = torch.full((segs.size, m, m), -7.0, device="cuda")
        cov = torch.full((segs.size, m, m), 7, dtype=torch.uint8, device="cuda")
        B.argus_healpix_resample(dev_pitched(frame), dev_pitched(fl), B.argus_shape(w, h, pitch_for(w)), wcs,
                                 nside_seg, k, torch.from_numpy(segs).cuda(), segs.size, out, cov)
        torch.cuda.synchronize()
        out, cov = out.cpu().numpy(), cov.cpu().numpy()
        tol = 4 * F32_EPS * float(np.abs(frame[np.isfinite(frame)]).max())
        for i, s in enumerate(segs[:-1]):
            o, oc = hp.resample_segment(frame, fl, int(s), nside_seg, k, wcs)
            np.testing.assert_array_equal(cov[i], oc)
            if big:     # a gradient of 6e38 per pixel: a position's 1e-7 pixel is 6e31 there, so only the range
                assert np.isfinite(out[i]).all() and np.abs(out[i]).max() <= 3.0e38 * (1 + F32_EPS)
            else:
                assert np.abs(out[i] - o).max() <= tol
        assert not out[-1].any() and not cov[-1].any()      # not a pixel of this NSIDE


@pytest.mark.parametrize("cx", [2.9e5, 5.0e5, 5.5e5])
def test_healpix_frame_wider_than_the_fixed_point(ora, cx):
    """A frame of more than 2^19 columns, whose last one is past the fixed-point positions' range:
    segments below the patch path's limit of 5e5 pixels, across it and above, at the bars of the parity test."""
    from oracle import healpix as hp
    rng = np.random.default_rng(int(cx))
    w, h, nside, k, m = 600000, 40, 256, 6, 64
    scale = math.sqrt(4 * math.pi / (12.0 * (nside << k) ** 2))
    wcs = (0.9, 0.3, scale, 0.8, cx, 17.25)
    frame = np.full((h, w), 300.0, np.float32)
    x0 = int(cx) - 200
    frame[:, x0:x0 + 400] += rng.normal(0, 10, (h, 400)).astype(np.float32)
    fl = np.zeros((h, w), np.uint8)
    fl[:, x0:x0 + 400] = rng.random((h, 400)) < 0.01
    p = np.arange(12 * nside * nside)
    ix, iy, f = hp.nest2xyf(p, nside)
    x, y = hp.gnomonic(hp.xyf2vec(ix, iy, f, nside), *wcs)
    d = np.where(np.isfinite(x), (x - cx) ** 2 + (y - h / 2) ** 2, np.inf)
    segs = p[np.argsort(d)[:3]].astype(np.int64)
    out = torch.full((segs.size, m, m), -7.0, device="cuda")
    cov = torch.full((segs.size, m, m), 7, dtype=torch.uint8, device="cuda")
    B.argus_healpix_resample(dev_pitched(frame), dev_pitched(fl), B.argus_shape(w, h, pitch_for(w)), wcs, nside, k,
                             torch.from_numpy(segs).cuda(), segs.size, out, cov)
    torch.cuda.synchronize()
    out, cov = out.cpu().numpy(), cov.cpu().numpy()
    assert cov.any()
    for i, s in enumerate(segs):
        o, oc = hp.resample_segment(frame, fl, int(s), nside, k, wcs)
        np.testing.assert_array_equal(cov[i], oc)
        assert np.abs(out[i] - o).max() <= 4 * F32_EPS * float(frame.max())


@pytest.mark.parametrize("nside_seg,k,delta0", [(64, 10, 0.85),       # caps only, images wider than a row piece
                                               (256, 6, 0.7297),     # the belt's edge inside the frame
                                               (512, 7, -0.735),
                                               (256, 6, 0.69),       # a frame inside the belt, segments beyond it
                                               (128, 8, 1.52)])      # next to the pole
def test_healpix_halves_out_of_the_belt(ora, nside_seg, k, delta0):
    """Each half patch is taken by exactly one kernel, whatever part of the frame and of the segments
    lies in the belt, at the bars of the parity test."""
    from oracle import healpix as hp
    rng = np.random.default_rng(nside_seg + k)
    w, h = 700, 500
    scale = math.sqrt(4 * math.pi / (12.0 * (nside_seg << k) ** 2))
    wcs = (2.1, delta0, scale, -0.4, (w - 1) / 2, (h - 1) / 2)
    frame = (300 + rng.normal(0, 10, (h, w))).astype(np.float32)
    frame.flat[11::701] = np.nan
    fl = (rng.random((h, w)) < 0.01).astype(np.uint8)
    p = np.arange(12 * nside_seg * nside_seg)
    ix, iy, f = hp.nest2xyf(p, nside_seg)
    x, y = hp.gnomonic(hp.xyf2vec(ix, iy, f, nside_seg), *wcs)
    d = np.where(np.isfinite(x), (x - w / 2) ** 2 + (y - h / 2) ** 2, np.inf)
    near = p[np.argsort(d)[:1 if k == 10 else 60]]
    segs = np.concatenate([near[:1], rng.choice(near, size=min(7, near.size - 1), replace=False), [-1]]).astype(np.int64)
    m = 1 << k
    out = torch.full((segs.size, m, m), -7.0, device="cuda")
    cov = torch.full((segs.size, m, m), 7, dtype=torch.uint8, device="cuda")
    B.argus_healpix_resample(dev_pitched(frame), dev_pitched(fl), B.argus_shape(w, h, pitch_for(w)), wcs,
                             nside_seg, k, torch.from_numpy(segs).cuda(), segs.size, out, cov)
    torch.cuda.synchronize()
    out, cov = out.cpu().numpy(), cov.cpu().numpy()
    assert cov[0].any()
    for i, s in enumerate(segs[:-1]):
        o, oc = hp.resample_segment(frame, fl, int(s), nside_seg, k, wcs)
        np.testing.assert_array_equal(cov[i], oc)
        assert np.abs(out[i] - o).max() <= 4 * F32_EPS * float(np.nanmax(frame))
    assert not out[-1].any() and not cov[-1].any()


@pytest.mark.parametrize("radius,delta0", [(0.02, 0.3), (0.02, -1.1), (0.3, 0.7), (0.9, -0.2)])
def test_healpix_segments_of_the_whole_sky(ora, radius, delta0):
    """All segments of the sky on frames of 1 to 52 degrees' radius: those behind the tangent plane, off the
    frame, across its edge and on it.  An image pixel is 0.23 degrees (delta) here, and a cubic is off by up to
    21^4 / 24 times the fourth derivative: that of tan(theta) / scale is at most 24 sec^5, on theta up to a piece (0.25)
    past the frame's radius, and the HEALPix map's own curvature is given a factor of 4.  Coverage may differ
    from the oracle's only for pixels nearer than that to the frame's edge."""
    from oracle import healpix as hp
    nside, k, w, h = 4, 6, 300, 200
    scale = math.tan(radius) / math.hypot((w - 1) / 2, (h - 1) / 2)
    delta = math.sqrt(math.pi / 3) / (nside << k)
    near = 4 * 24 / math.cos(radius + 0.25) ** 5 * delta ** 4 * 21 ** 4 / 24 / scale
    assert near < 10
    wcs = (2.1, delta0, scale, -0.4, (w - 1) / 2, (h - 1) / 2)
    frame = np.full((h, w), 7.0, np.float32)
    segs = np.arange(12 * nside * nside, dtype=np.int64)
    m = 1 << k
    out = torch.full((segs.size, m, m), -7.0, device="cuda")
    cov = torch.full((segs.size, m, m), 7, dtype=torch.uint8, device="cuda")
    B.argus_healpix_resample(dev_pitched(frame), None, B.argus_shape(w, h, pitch_for(w)), wcs, nside, k,
                             torch.from_numpy(segs).cuda(), segs.size, out, cov)
    torch.cuda.synchronize()
    out, cov = out.cpu().numpy(), cov.cpu().numpy()
    assert cov.any() and (out == np.float32(7.0) * cov).all()
    for i, s in enumerate(segs):
        x, y = hp.gnomonic(hp.segment_vectors(int(s), nside, k), *wcs)
        inside = np.minimum(np.minimum(x, w - 1 - x), np.minimum(y, h - 1 - y))     # > 0: so far inside the frame
        inside = np.where(np.isfinite(inside), inside, -np.inf)
        assert cov[i][inside > near].all() and not cov[i][inside < -near].any()
