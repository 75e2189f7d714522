"""The index and shift arithmetic of the kernels on the CPU: host-callable functions of
the .cu files, compiled by nvcc as host code with a small driver each
(tests/host_drivers).  Needs nvcc, no GPU."""
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2207_14304_gb300", "csrc")
DRV = os.path.join(ROOT, "tests", "host_drivers")


@pytest.fixture(scope="module")
def driver(tmp_path_factory):
    """driver(name): the path of the compiled driver `name`; work files go beside it."""
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    d = tmp_path_factory.mktemp("host_lanes")

    def build(name):
        if not (d / name).exists():
            subprocess.check_call([nvcc, "-O2", "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-I", CSRC,
                                   "-I", os.path.join(ROOT, "include"), "-I", DRV, "-o", str(d / name),
                                   os.path.join(DRV, name + ".cu")])
        return d / name
    return build


def _run(exe, *args):
    subprocess.check_call([str(exe), *map(str, args)], cwd=exe.parent)


# --------------------------------------------------------------------------- clipped coadd
@pytest.mark.parametrize("size", [1, 31, 6388, 1 << 20])
def test_coadd_shifts_stay_in_range(driver, size):
    """Shifts inside the frame split exactly; any other, and any that is not finite, gives a
    window that no tile of the frame finds a pixel in, with coordinates and a union in range."""
    exe = driver("host_coadd_shift")
    v = np.array([0, -0.25, 0.5, 1, -1, 0.1, -0.3, 0.7123, -1e-9, size - 1, -size, size, size + 0.5, -size - 40, 46341, -46341, 65536, 1e9, -1e9, 2147483520,
                  -2147483648, 3e9, -3e9, 3e38, -3e38, np.inf, -np.inf, np.nan], np.float32)
    v.tofile(exe.parent / "shifts.bin")
    _run(exe, size, "shifts.bin", "shifts.out")
    raw = (exe.parent / "shifts.out").read_bytes()
    n = v.size
    whole, frac = np.frombuffer(raw, np.int32, n), np.frombuffer(raw, np.float32, n, 4 * n)
    weights = np.frombuffer(raw, np.float32, 2 * n, 8 * n).reshape(2, n)
    fits = np.frombuffer(raw, np.uint8, n * n, 16 * n).reshape(n, n)
    inside = np.abs(v) <= size
    d = v[np.isfinite(v)].astype(np.float64)
    np.testing.assert_array_equal(whole[inside], np.floor(v[inside]))
    np.testing.assert_array_equal(frac[np.isfinite(v)], (d - np.floor(d)).astype(np.float32))
    assert np.isnan(frac[~np.isfinite(v)]).all()
    f = frac[np.isfinite(v)].astype(np.float64)             # the variances' weights: squares rounded once
    np.testing.assert_array_equal(weights[:, np.isfinite(v)], np.stack([(1 - f) ** 2, f ** 2]).astype(np.float32))
    # a tile starts in [0, size); its window reaches 32 pixels on
    first, last = whole.astype(np.int64), whole.astype(np.int64) + size - 1 + 31
    assert ((first[~inside] >= size) | (last[~inside] < 0)).all()
    assert (np.abs(first) <= size + 32).all()
    span = np.abs(first[:, None] - first[None, :])
    np.testing.assert_array_equal(fits, ((span + 32) * 9 <= 512) & ((span + 9) * 32 <= 512))


# --------------------------------------------------------------------------- subtraction
def test_subtraction_bands(driver):
    """Bands start on block boundaries (whole blocks of 4 and 8 source rows), a variance band divides a
    128-row tile, and the choice is that of tests/gpu_helpers.band_rows."""
    from tests.gpu_helpers import band_rows
    exe = driver("host_bands")
    rng = np.random.default_rng(3)
    w = np.exp(rng.uniform(0, np.log(20000), 400)).astype(np.int32)
    h = np.exp(rng.uniform(0, np.log(20000), 400)).astype(np.int32)
    c = np.stack([w, h, rng.choice([5, 10], 400), rng.choice([1, 16, 148, 152, 160], 400)], 1).astype(np.int32)
    c.tofile(exe.parent / "bands.bin")
    _run(exe, "bands.bin", "bands.out")
    rows = np.fromfile(exe.parent / "bands.out", np.int32).reshape(-1, 2)
    assert (rows > 0).all() and (rows[:, 0] % 4 == 0).all() and np.isin(rows[:, 1], [16, 32, 64, 128]).all()
    want = [[band_rows(*map(int, q), v) for v in (False, True)] for q in c]
    np.testing.assert_array_equal(rows, want)


# --------------------------------------------------------------------------- background map
def test_background_scratch_holds_every_part(driver):
    """The parts of a call's scratch lie apart and aligned, and a frame's own pixels (an int each, a pitch
    of a multiple of 16) leave room for them at the smallest box and the most ragged sizes."""
    sizes = [(w, h) for w in (1, 7, 8, 9, 16, 17, 130, 9576) for h in (1, 8, 9, 65, 6388)]
    cells = [-(-w // 8) * -(-h // 8) for w, h in sizes]
    out = subprocess.check_output([str(driver("host_bg_scratch")), *map(str, cells)]).decode().split("\n")
    for (w, h), n, line in zip(sizes, cells, out):
        fill, meshf, missing, size = map(int, line.split())
        parts = [(0, 8 * n, 8), (fill, 8, 8), (meshf, 4 * n, 4), (missing, 4, 4)]     # start, bytes, alignment
        assert all(a + b <= c for (a, b, _), (c, _, _) in zip(parts, parts[1:]))
        assert all(a % k == 0 for a, _, k in parts) and missing + 4 <= size <= 4 * h * (-(-w // 16) * 16)


# --------------------------------------------------------------------------- transforms
@pytest.mark.parametrize("T", [256, 512, 1024])
@pytest.mark.parametrize("dbl", [0, 1])
def test_register_transforms_match_numpy(driver, T, dbl):
    """The register passes, lane by lane, against numpy, at the bar of the whole transforms' test (a few
    ulps times log2 of the points), and unit impulses at every position of a lane's eight values."""
    exe = driver("host_fft_lanes")
    rng = np.random.default_rng(T + dbl)
    x = rng.normal(size=(40, T)) + 1j * rng.normal(size=(40, T))
    x[8:] = np.eye(T)[(np.arange(32) * (T // 32) + np.arange(32) % 7) % T]
    x = x.astype(np.complex128 if dbl else np.complex64)
    x.tofile(exe.parent / "seq.bin")
    for sign in (-1, 1):
        _run(exe, "full", T, dbl, sign, "seq.bin", "seq.out")
        y = np.fromfile(exe.parent / "seq.out", x.dtype).reshape(x.shape)
        x64 = x.astype(np.complex128)
        ref = np.fft.fft(x64) if sign < 0 else np.fft.ifft(x64) * T
        err = (np.abs(y - ref).max(1) / np.abs(ref).max(1)).max()
        assert err < 8 * (2.0 ** -53 if dbl else 2.0 ** -24) * np.log2(T), (sign, err)


@pytest.mark.parametrize("T", [256, 512, 1024])
@pytest.mark.parametrize("ps", [1, 3, 13, 15, 17, 31, 33, 63])
def test_psf_transforms_leave_out_only_zeros(driver, T, ps):
    """A stamp's sequence with its centre at position 0: the passes that leave out zeros against numpy, and
    equal to the passes that don't (a value that is left out is NaN in the driver)."""
    exe = driver("host_fft_lanes")
    rng = np.random.default_rng(T + ps)
    p = rng.normal(size=(5, ps))
    p.tofile(exe.parent / "psf.bin")
    _run(exe, "psf", T, ps, "psf.bin", "psf.out")
    y, whole = np.fromfile(exe.parent / "psf.out", np.complex128).reshape(2, 5, T)
    x = np.zeros((5, T))
    x[:, (np.arange(ps) - ps // 2) % T] = p
    ref = np.fft.fft(x)
    assert np.abs(y - ref).max() < 8 * 2.0 ** -53 * np.log2(T) * np.abs(ref).max()
    np.testing.assert_array_equal(y, whole)


def test_coadd_cuts_fit_the_pool(driver):
    """Every cut holds at least a pair of a tile, all pairs where a chunk has several tiles, no more than was
    asked for, and stays inside the plan's pool."""
    exe = driver("host_cut")
    rng = np.random.default_rng(8)
    n = 4000
    most = np.exp(rng.uniform(0, np.log(400), n)).astype(np.int32)
    c = np.stack([rng.choice([256, 512, 1024], n), most, 1 + (rng.random(n) * most).astype(np.int32), rng.integers(1, 33, n),
                  rng.choice([1, 3, 31, 63], n), rng.integers(0, 2, n), rng.integers(0, 2, n)], 1).astype(np.int32)
    c.tofile(exe.parent / "cuts.bin")
    _run(exe, "cuts.bin", "cuts.out")
    tiles, group, used, pool = np.fromfile(exe.parent / "cuts.out", np.int64).reshape(-1, 4).T
    assert (group >= 1).all() and (tiles >= 1).all() and (tiles <= c[:, 2]).all() and (group <= c[:, 3]).all()
    assert (group[tiles > 1] == c[tiles > 1, 3]).all()
    assert (used <= pool).all()


@pytest.mark.parametrize("n", [1, 2, 33, 64, 2304, 4096])
def test_box_selection_ends_at_the_median(driver, n):
    """The bracketing selection's median equals numpy's exactly, on noise, ties, wide ranges, two values,
    extremes of the type, denormals, signed zeros and boxes with invalid pixels, within the interpolated passes plus one
    per bit of a key."""
    exe = driver("host_box_median")
    rng = np.random.default_rng(n)
    big = np.finfo(np.float32).max
    x = [rng.normal(300, 15, n), np.rint(rng.normal(5, 2, n)), np.full(n, 7.5), np.exp(rng.normal(0, 40, n)),
         rng.choice([-1.0, 1.0], n), rng.choice([-big, big], n), rng.choice([0.0, -0.0, 1e-45, -1e-45], n), rng.choice([1e-40, -3.0], n),
         np.where(rng.random(n) < 0.5, big, rng.normal(0, 1, n)), np.sort(rng.normal(0, 1, n)), -np.sort(-rng.normal(0, 1, n)),
         np.r_[np.full(n // 2, -big), rng.normal(1e30, 1e28, n - n // 2)]]
    x += [np.where(rng.random(n) < p, np.nan, rng.normal(300, 15, n)) for p in (0.01, 0.5, 0.97)]
    with np.errstate(over="ignore"):
        x = np.stack(x).astype(np.float32)                  # (the wide range reaches infinity, which is no valid pixel)
    x[:, 0] = np.where(np.isnan(x[:, 0]), 1.0, x[:, 0])     # a valid pixel at least
    x.tofile(exe.parent / "boxes.bin")
    _run(exe, n, "boxes.bin", "boxes.out")
    raw = (exe.parent / "boxes.out").read_bytes()
    med, passes = np.frombuffer(raw, np.float64, len(x)), np.frombuffer(raw, np.int32, len(x), 8 * len(x))
    np.testing.assert_array_equal(med, np.nanmedian(np.where(np.isfinite(x), x, np.nan).astype(np.float64), axis=1))
    assert passes.max() <= 11 + 32


# --------------------------------------------------------------------------- HEALPix patches
@pytest.mark.parametrize("nside_seg,k,delta0,rot", [(256, 6, 0.3, 0.8), (256, 9, -0.2, -2.0), (64, 7, 0.0, 0.0), (128, 8, 0.7, 0.3)])
def test_patch_positions_follow_the_exact_ones(driver, nside_seg, k, delta0, rot):
    """The fixed-point positions of halves in the belt against the exact path's.  A cubic through the
    columns 0, 21, 42, 63 is off by at most 21^4 / 24 times the fourth derivative, which for a map of
    one frame pixel per image pixel is F delta^3 (delta the pixel's angle, F <= 20 within 10 degrees of the tangent
    point); the rows' nodes are half as far apart; the differences and the fixed point add less than 1e-9."""
    from oracle import healpix as hp
    exe = driver("host_hp_patch")
    delta = np.sqrt(4 * np.pi / (12.0 * (nside_seg << k) ** 2))
    wcs = np.array([0.9, delta0, delta, rot, 400.0, 300.0])
    p = np.arange(12 * nside_seg * nside_seg)
    ix, iy, f = hp.nest2xyf(p, nside_seg)
    x, y = hp.gnomonic(hp.xyf2vec(ix, iy, f, nside_seg), *wcs)
    near = p[np.argsort(np.where(np.isfinite(x), np.hypot(x - 400, y - 300), np.inf))[:3]]
    wcs.tofile(exe.parent / "wcs.bin")
    near.astype(np.int64).tofile(exe.parent / "segs.bin")
    _run(exe, "pos", nside_seg, k, "wcs.bin", "segs.bin", "pos.out")
    o = np.fromfile(exe.parent / "pos.out").reshape(-1, 4)
    assert len(o) >= 2 * 64 * 32
    assert np.abs(o[:, :2] - o[:, 2:]).max() <= 20 * delta ** 3 * 21 ** 4 / 24 * (1 + 1 / 16) + 1e-9


def test_fixed_point_interpolation(driver):
    """Four values and fractions of 2^-44 against FP64: one rounding (half an ulp of the result) and the pairs'
    2^-44 of the largest value, over ten decades, of either sign, ties of values and the ends of a pixel."""
    exe = driver("host_hp_patch")
    rng = np.random.default_rng(1)
    n = 200000
    q = (rng.normal(size=(n, 4)) * 10.0 ** rng.uniform(-5, 5, (n, 1))).astype(np.float32)
    q[::5] = (300 + rng.normal(size=(len(q[::5]), 4))).astype(np.float32)
    q[::7, 1] = q[::7, 0]
    t = np.floor(rng.random((n, 2)) * 2.0 ** 44) / 2.0 ** 44
    t[::11, 0], t[::13, 1], t[::17] = 0.0, 0.0, (2.0 ** 44 - 1) / 2.0 ** 44
    (exe.parent / "lerp.bin").write_bytes(q.tobytes() + t.tobytes())
    _run(exe, "lerp", "lerp.bin", "lerp.out")
    v = np.fromfile(exe.parent / "lerp.out", np.float32).astype(np.float64)
    d = q.astype(np.float64)
    top, bot = d[:, 0] + t[:, 0] * (d[:, 1] - d[:, 0]), d[:, 2] + t[:, 0] * (d[:, 3] - d[:, 2])
    ref = top + t[:, 1] * (bot - top)
    assert (np.abs(v - ref) <= 2.0 ** -24 * np.abs(ref) * 1.0001 + 16 * 2.0 ** -44 * np.abs(d).max(1)).all()
