"""ZOGY (Sec. 4.2) and the proper coadd (Sec. 4.1.3) on the GPU against the FP64
oracle, tile by tile.

Tolerances, from the FP32 rounding of the image transforms (the PSF
transforms are FP64): with u = 2^-24 and the unit
  e = u log2(T^2) (||N||_2 / s_n + ||R||_2 / s_r) / T
(the rms rounding of a T^2-point FP32 FFT carried through the quotient, whose
gain is at most 1/s_n and 1/s_r), |dD| <= 8 e and |dS| <= 8 (e F_D ||P_D||_1 +
u log2(T^2) ||D||_2 / T) (S filters D with F_D P_D and shares D's inverse
transform); an FP32 emulation of the same algorithm (numpy's
single-precision FFT) stays within 1.4 e and 3.1 e F_D ||P_D||_1 on these
tiles.  P_D within 64 u max|P_D|, sigma_S within 1e-6 relative.

The kernels have not run on a GPU yet, so the file is skipped until they have.
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


def _gauss(sig, half=15):
    u = np.arange(-half, half + 1)
    g = np.exp(-(u[None, :] ** 2 + u[:, None] ** 2) / (2 * sig * sig))
    return (g / g.sum()).astype(np.float32)


def _frame(w, h, seed, sn, sr, psf_n, psf_r, Fn, Fr):
    from oracle import proper
    rng = np.random.default_rng(seed)
    sky = np.zeros((h, w))
    n = w * h // 130
    np.add.at(sky, (rng.integers(0, h, n), rng.integers(0, w, n)), 1e2 * 1e4 ** rng.random(n))
    conv = lambda img, P: np.fft.ifft2(np.fft.fft2(img) * np.fft.fft2(proper.psf_on_tile(P, img.shape))).real
    N = (Fn * conv(sky, psf_n) + rng.normal(0, sn, (h, w))).astype(np.float32)
    R = (Fr * conv(sky, psf_r) + rng.normal(0, sr, (h, w))).astype(np.float32)
    return N, R


@pytest.mark.parametrize("T,origins", [(256, [(0, 0), (300, 100), (520, 260)]), (512, [(64, 32)]),
                                       (1024, [(0, 0)])])
def test_zogy_parity(ora, T, origins):
    from oracle import proper
    w, h = 800, 600 if T < 1024 else 1024
    w = max(w, T)
    specs = [(1.05, 1.0, 18.0, 3.3, 2.0, 1.2), (0.9, 1.1, 10.0, 4.0, 1.3, 1.6), (1.0, 1.0, 7.0, 7.0, 2.2, 2.2)]
    N, R = _frame(w, h, seed=T, sn=12.0, sr=3.0, psf_n=_gauss(1.8), psf_r=_gauss(1.3), Fn=1.0, Fr=1.0)
    rec = np.zeros(len(origins), B.ZOGY_TILE_DTYPE)
    pn = np.zeros((len(origins), 31, 31), np.float32)
    pr = np.zeros_like(pn)
    for i, (x0, y0) in enumerate(origins):
        Fn, Fr, sn, sr, gn, gr = specs[i % len(specs)]
        rec[i] = (x0, y0, Fn, Fr, sn, sr)
        pn[i], pr[i] = _gauss(gn), _gauss(gr)
    nt = len(origins)
    plan = B.proper_plan_create(0, T, 4)
    try:
        pitch = pitch_for(w)
        dN, dR = dev_pitched(N), dev_pitched(R)
        d_rec = torch.from_numpy(rec.view(np.uint8).copy()).cuda()
        D = torch.full((nt, T, T), -7.0, device="cuda")
        S = torch.full((nt, T, T), -7.0, device="cuda")
        PD = torch.full((nt, T, T), -7.0, device="cuda")
        sig = torch.zeros(nt, dtype=torch.float64, device="cuda")
        B.argus_zogy(plan, dN, dR, B.argus_shape(w, h, pitch), d_rec, nt, torch.from_numpy(pn).cuda(),
                     torch.from_numpy(pr).cuda(), 31, 1e-8, D, S, PD, sig)
        torch.cuda.synchronize()
        D, S, PD, sig = D.cpu().numpy(), S.cpu().numpy(), PD.cpu().numpy(), sig.cpu().numpy()
    finally:
        B.proper_plan_destroy(plan)
    for i, (x0, y0) in enumerate(origins):
        Fn, Fr, sn, sr = (float(rec[i][k]) for k in ("Fn", "Fr", "sn", "sr"))
        tN = np.zeros((T, T), np.float32)
        tR = np.zeros((T, T), np.float32)
        ys, xs = slice(y0, min(y0 + T, h)), slice(x0, min(x0 + T, w))
        tN[: ys.stop - y0, : xs.stop - x0] = N[ys, xs]
        tR[: ys.stop - y0, : xs.stop - x0] = R[ys, xs]
        o = proper.zogy(tN, tR, pn[i].astype(np.float64), pr[i].astype(np.float64), Fn, Fr, sn, sr)
        e = F32_EPS * math.log2(T * T) * (np.linalg.norm(tN) / sn + np.linalg.norm(tR) / sr) / T
        dD = np.abs(D[i] - o["D"]).max()
        # S filters D with F_D P_D and shares D's inverse transform
        sS = e * o["F_D"] * np.abs(o["P_D"]).sum() + F32_EPS * math.log2(T * T) * np.linalg.norm(o["D"]) / T
        dS = np.abs(S[i] - o["S"]).max()
        print(f"\n[zogy T={T} tile {i}] |dD| {dD:.2e} = {dD / e:.2f} e   |dS| = {dS / sS:.2f} e F_D |P_D|_1")
        assert dD <= 8 * e
        assert dS <= 8 * sS
        assert np.abs(PD[i] - o["P_D"]).max() <= 64 * F32_EPS * np.abs(o["P_D"]).max()
        assert abs(sig[i] / o["sigma_S"] - 1) < 1e-6


@pytest.mark.parametrize("T,J", [(256, 3), (512, 2)])
def test_proper_coadd_parity(ora, T, J):
    """Proper coadd (Sec. 4.1.3) through the entry point against the oracle per tile:
    R within 8 e_R, S within 8 e_S (the units of tests/test_host_kernels.py), P_R
    within 64 ulps of its maximum, F_R and sigma_S within 1e-6."""
    from oracle import proper
    w, h = 700, 600
    rng = np.random.default_rng(T + J)
    sky = np.zeros((h, w))
    n = w * h // 150
    np.add.at(sky, (rng.integers(0, h, n), rng.integers(0, w, n)), 1e2 * 1e4 ** rng.random(n))
    conv = lambda img, P: np.fft.ifft2(np.fft.fft2(img) * np.fft.fft2(proper.psf_on_tile(P, img.shape))).real
    origins = [(0, 0), (400, 300)] if T == 256 else [(100, 50)]
    nt = len(origins)
    gs = [1.2, 1.9, 1.5][:J]
    F = np.array([1.0, 0.8, 1.2][:J], np.float32)
    sg = np.array([5.0, 9.0, 4.0][:J], np.float32)
    frames = [(f * conv(sky, _gauss(g)) + rng.normal(0, s, (h, w))).astype(np.float32) for g, f, s in zip(gs, F, sg)]
    psfs = np.stack([np.stack([_gauss(g + 0.1 * t) for g in gs]) for t in range(nt)])     # [nt][J][31][31]
    pitch = pitch_for(w)
    plan = B.proper_plan_create(0, T, 4)
    try:
        stack = torch.zeros((J, h, pitch), device="cuda")
        for j in range(J):
            stack[j, :, :w] = torch.from_numpy(frames[j]).cuda()
        d_org = torch.tensor(origins, dtype=torch.int32, device="cuda")
        S = torch.full((nt, T, T), -7.0, device="cuda")
        R = torch.full((nt, T, T), -7.0, device="cuda")
        PR = torch.full((nt, T, T), -7.0, device="cuda")
        FR = torch.zeros(1, dtype=torch.float64, device="cuda")
        sig = torch.zeros(nt, dtype=torch.float64, device="cuda")
        B.argus_proper_coadd(plan, stack, J, B.argus_shape(w, h, pitch), d_org, nt, torch.from_numpy(F).cuda(),
                             torch.from_numpy(sg).cuda(), torch.from_numpy(psfs).cuda(), 31, 1e-8, S, R, PR, FR, sig)
        torch.cuda.synchronize()
        S, R, PR, FR, sig = (t.cpu().numpy() for t in (S, R, PR, FR, sig))
    finally:
        B.proper_plan_destroy(plan)
    for i, (x0, y0) in enumerate(origins):
        Ms = [np.ascontiguousarray(f[y0:y0 + T, x0:x0 + T]) for f in frames]
        Ps = [psfs[i, j].astype(np.float64) for j in range(J)]
        o = proper.proper_coadd(Ms, Ps, [float(f) for f in F], [float(s) for s in sg])
        lg = F32_EPS * math.log2(T * T) / T
        eR = lg * sum(np.linalg.norm(M) / s for M, s in zip(Ms, sg))
        eS = lg * (sum(f / s ** 2 * np.abs(P).sum() * np.linalg.norm(M) for M, P, f, s in zip(Ms, Ps, F, sg))
                   + np.linalg.norm(o["R"]))
        assert np.abs(R[i] - o["R"]).max() <= 8 * eR
        assert np.abs(S[i] - o["S"]).max() <= 8 * eS
        assert np.abs(PR[i] - o["P_R"]).max() <= 64 * F32_EPS * np.abs(o["P_R"]).max()
        assert abs(FR[0] / o["F_R"] - 1) < 1e-6 and abs(sig[i] / o["sigma_S"] - 1) < 1e-6


def test_zogy_reuses_psf_transforms_and_coadd_discards_them(ora):
    """A call without PSFs gives the outputs of the call that supplied them, bit for bit;
    after a proper-coadd call on the plan it is refused."""
    T, w, h = 256, 600, 400
    N, R = _frame(w, h, seed=5, sn=12.0, sr=3.0, psf_n=_gauss(1.8), psf_r=_gauss(1.3), Fn=1.0, Fr=1.0)
    rec = np.zeros(2, B.ZOGY_TILE_DTYPE)
    rec[0] = (0, 0, 1.0, 1.0, 12.0, 3.0)
    rec[1] = (300, 100, 1.0, 1.0, 12.0, 3.0)
    pn = np.stack([_gauss(1.8), _gauss(1.9)])
    pr = np.stack([_gauss(1.3), _gauss(1.3)])
    pitch = pitch_for(w)
    plan = B.proper_plan_create(0, T, 2)
    try:
        dN, dR = dev_pitched(N), dev_pitched(R)
        d_rec = torch.from_numpy(rec.view(np.uint8).copy()).cuda()
        sh = B.argus_shape(w, h, pitch)
        D1 = torch.empty((2, T, T), device="cuda")
        S1 = torch.empty((2, T, T), device="cuda")
        D2 = torch.empty((2, T, T), device="cuda")
        S2 = torch.empty((2, T, T), device="cuda")
        B.argus_zogy(plan, dN, dR, sh, d_rec, 2, torch.from_numpy(pn).cuda(), torch.from_numpy(pr).cuda(), 31, 1e-8,
                     D1, S1)
        B.argus_zogy(plan, dN, dR, sh, d_rec, 2, None, None, 31, 1e-8, D2, S2)
        torch.cuda.synchronize()
        assert torch.equal(D1, D2) and torch.equal(S1, S2)
        stack = dN.unsqueeze(0).contiguous()
        org = torch.zeros((1, 2), dtype=torch.int32, device="cuda")
        one = torch.ones(1, device="cuda")
        B.argus_proper_coadd(plan, stack, 1, sh, org, 1, one, one, torch.from_numpy(pn[:1]).cuda(), 31, 1e-8,
                             torch.empty((1, T, T), device="cuda"), torch.empty((1, T, T), device="cuda"))
        with pytest.raises(B.ArgusError):
            B.argus_zogy(plan, dN, dR, sh, d_rec, 2, None, None, 31, 1e-8, D2, S2)
    finally:
        B.proper_plan_destroy(plan)


def test_shared_psfs_match_per_tile_copies(ora):
    """One PSF (pair) shared by every tile gives, bit for bit, what the same PSF copied
    into every tile gives, for ZOGY (also when reused) and for the proper coadd."""
    T, w, h, nt = 256, 700, 500, 3
    N, R = _frame(w, h, seed=6, sn=12.0, sr=3.0, psf_n=_gauss(1.8), psf_r=_gauss(1.3), Fn=1.0, Fr=1.0)
    rec = np.zeros(nt, B.ZOGY_TILE_DTYPE)
    for i, (x0, y0) in enumerate([(0, 0), (300, 100), (420, 240)]):
        rec[i] = (x0, y0, 1.0, 1.0, 12.0, 3.0)
    pn, pr = _gauss(1.8), _gauss(1.3)
    pitch = pitch_for(w)
    sh = B.argus_shape(w, h, pitch)
    plan = B.proper_plan_create(0, T, nt)
    try:
        dN, dR = dev_pitched(N), dev_pitched(R)
        d_rec = torch.from_numpy(rec.view(np.uint8).copy()).cuda()
        out = [torch.empty((nt, T, T), device="cuda") for _ in range(6)]
        B.argus_zogy(plan, dN, dR, sh, d_rec, nt, torch.from_numpy(np.stack([pn] * nt)).cuda(),
                     torch.from_numpy(np.stack([pr] * nt)).cuda(), 31, 1e-8, out[0], out[1])
        B.argus_zogy(plan, dN, dR, sh, d_rec, nt, torch.from_numpy(pn).cuda(), torch.from_numpy(pr).cuda(), 31, 1e-8,
                     out[2], out[3], psf_per_tile=False)
        B.argus_zogy(plan, dN, dR, sh, d_rec, nt, None, None, 31, 1e-8, out[4], out[5], psf_per_tile=False)
        torch.cuda.synchronize()
        for a, b in ((0, 2), (1, 3), (0, 4), (1, 5)):
            assert torch.equal(out[a], out[b]), (a, b)
        with pytest.raises(B.ArgusError):       # per-tile reuse after a shared call: nothing to reuse
            B.argus_zogy(plan, dN, dR, sh, d_rec, nt, None, None, 31, 1e-8, out[4], out[5])
        J = 3
        stack = torch.stack([dN, dR, dN]).contiguous()
        org = torch.tensor([(0, 0), (300, 100), (420, 240)], dtype=torch.int32, device="cuda")
        F = torch.ones(J, device="cuda")
        sg = torch.tensor([12.0, 3.0, 12.0], device="cuda")
        ps = np.stack([_gauss(g) for g in (1.8, 1.3, 1.6)])
        S1, R1, S2, R2 = (torch.empty((nt, T, T), device="cuda") for _ in range(4))
        B.argus_proper_coadd(plan, stack, J, sh, org, nt, F, sg, torch.from_numpy(np.stack([ps] * nt)).cuda(), 31, 1e-8,
                             S1, R1)
        B.argus_proper_coadd(plan, stack, J, sh, org, nt, F, sg, torch.from_numpy(ps).cuda(), 31, 1e-8, S2, R2,
                             psf_per_tile=False)
        torch.cuda.synchronize()
        assert torch.equal(S1, S2) and torch.equal(R1, R2)
    finally:
        B.proper_plan_destroy(plan)


@pytest.mark.parametrize("T,nt,J,ps,per_tile", [(256, 1, 41, 63, True),     # pairs in groups, the score carried; odd
                                                (256, 3, 64, 63, True),     # groups within chunks of one tile
                                                (256, 3, 64, 31, False),    # the same with shared PSFs
                                                (256, 8, 5, 31, True)])     # chunks of several tiles
def test_proper_coadd_cuts(ora, T, nt, J, ps, per_tile):
    """Every way a coadd is cut into chunks of tiles and groups of pairs, with tiles hanging
    off the frame and a frame left out (sigma 0), at the bars of test_proper_coadd_parity."""
    from oracle import proper
    w, h = T + 90, T + 40
    rng = np.random.default_rng(T + J)
    origins = [(-20 + 17 * i, 31 - 13 * i) for i in range(nt)]
    F = rng.uniform(0.8, 1.2, J).astype(np.float32)
    sg = rng.uniform(4, 9, J).astype(np.float32)
    if J > 3:
        sg[2] = 0.0
    frames = rng.normal(0, 6, (J, h, w)).astype(np.float32)
    frames[:, rng.integers(0, h, 40), rng.integers(0, w, 40)] += 3e3
    half = ps // 2
    psfs = np.stack([np.stack([_gauss(1.2 + 0.02 * j + 0.05 * t, half) for j in range(J)])
                     for t in range(nt if per_tile else 1)])
    pitch = pitch_for(w)
    stack = torch.zeros((J, h, pitch), device="cuda")
    stack[:, :, :w] = torch.from_numpy(frames).cuda()
    S, R, PR = (torch.full((nt, T, T), -7.0, device="cuda") for _ in range(3))
    FR = torch.zeros(1, dtype=torch.float64, device="cuda")
    sig = torch.zeros(nt, dtype=torch.float64, device="cuda")
    plan = B.proper_plan_create(0, T, nt)
    try:
        B.argus_proper_coadd(plan, stack, J, B.argus_shape(w, h, pitch),
                             torch.tensor(origins, dtype=torch.int32, device="cuda"), nt, torch.from_numpy(F).cuda(),
                             torch.from_numpy(sg).cuda(), torch.from_numpy(psfs).cuda(), ps, 1e-8, S, R, PR, FR, sig,
                             psf_per_tile=per_tile)
        torch.cuda.synchronize()
        S, R, PR, FR, sig = (t.cpu().numpy() for t in (S, R, PR, FR, sig))
    finally:
        B.proper_plan_destroy(plan)
    use = [j for j in range(J) if sg[j] > 0]
    for i, (x0, y0) in enumerate(origins):
        Ms = []
        for j in use:
            M = np.zeros((T, T), np.float32)
            xs, ys = slice(max(x0, 0), min(x0 + T, w)), slice(max(y0, 0), min(y0 + T, h))
            M[ys.start - y0:ys.stop - y0, xs.start - x0:xs.stop - x0] = frames[j, ys, xs]
            Ms.append(M)
        Ps = [psfs[i if per_tile else 0, j].astype(np.float64) for j in use]
        o = proper.proper_coadd(Ms, Ps, [float(F[j]) for j in use], [float(sg[j]) for j in use])
        lg = F32_EPS * math.log2(T * T) / T
        eR = lg * sum(np.linalg.norm(M) / sg[j] for M, j in zip(Ms, use))
        eS = lg * (sum(F[j] / sg[j] ** 2 * np.abs(P).sum() * np.linalg.norm(M) for M, P, j in zip(Ms, Ps, use))
                   + np.linalg.norm(o["R"]))
        assert np.abs(R[i] - o["R"]).max() <= 8 * eR
        assert np.abs(S[i] - o["S"]).max() <= 8 * eS
        assert np.abs(PR[i] - o["P_R"]).max() <= 64 * F32_EPS * np.abs(o["P_R"]).max()
        assert abs(FR[0] / o["F_R"] - 1) < 1e-6 and abs(sig[i] / o["sigma_S"] - 1) < 1e-6


def test_proper_coadd_1024(ora):
    """A 1024 tile of five noise frames at the bars of test_proper_coadd_parity."""
    from oracle import proper
    T, J = 1024, 5
    rng = np.random.default_rng(9)
    F, sg = np.array([1.0, 0.8, 1.2, 0.9, 1.1], np.float32), np.array([5.0, 9.0, 4.0, 7.0, 6.0], np.float32)
    frames = (rng.normal(0, 1, (J, T, T)) * sg[:, None, None]).astype(np.float32)
    psfs = np.stack([_gauss(1.2 + 0.2 * j) for j in range(J)])
    S, R = (torch.empty((1, T, T), device="cuda") for _ in range(2))
    plan = B.proper_plan_create(0, T, 1)
    try:
        B.argus_proper_coadd(plan, torch.from_numpy(frames).cuda(), J, B.argus_shape(T, T, T),
                             torch.zeros((1, 2), dtype=torch.int32, device="cuda"), 1, torch.from_numpy(F).cuda(),
                             torch.from_numpy(sg).cuda(), torch.from_numpy(psfs).cuda(), 31, 1e-8, S, R)
        torch.cuda.synchronize()
        S, R = S[0].cpu().numpy(), R[0].cpu().numpy()
    finally:
        B.proper_plan_destroy(plan)
    o = proper.proper_coadd(list(frames), [p.astype(np.float64) for p in psfs], [float(f) for f in F],
                            [float(s) for s in sg])
    lg = F32_EPS * math.log2(T * T) / T
    eR = lg * sum(np.linalg.norm(M) / s for M, s in zip(frames, sg))
    eS = lg * (sum(f / s ** 2 * np.abs(P).sum() * np.linalg.norm(M) for M, P, f, s in zip(frames, psfs, F, sg))
               + np.linalg.norm(o["R"]))
    assert np.abs(R - o["R"]).max() <= 8 * eR
    assert np.abs(S - o["S"]).max() <= 8 * eS


@pytest.mark.parametrize("T,ps", [(256, 15), (256, 3), (512, 31), (512, 29)])
def test_zero_rim_of_a_stamp_changes_nothing(T, ps):
    """PSF stamps up to the side whose transforms leave out zeros, and the same stamps inside a rim
    of zeros that takes them past it: the same bits."""
    rng = np.random.default_rng(T + ps)
    rim = max((T // 16 - ps) // 2 + 1, 1)
    small = rng.normal(0, 0.1, (2, ps, ps)).astype(np.float32)
    small[:, ps // 2, ps // 2] = 1.0
    large = np.pad(small, ((0, 0), (rim, rim), (rim, rim)))
    assert ps // 2 < T // 32 <= large.shape[1] // 2
    img = [torch.from_numpy(rng.normal(0, 5, (T, T)).astype(np.float32)).cuda() for _ in range(2)]
    rec = np.zeros(1, B.ZOGY_TILE_DTYPE)
    rec[0] = (0, 0, 1.05, 1.0, 5.0, 4.0)
    d_rec, shape = torch.from_numpy(rec.view(np.uint8).copy()).cuda(), B.argus_shape(T, T, T)
    org, F, sg = torch.zeros((1, 2), dtype=torch.int32, device="cuda"), torch.ones(2, device="cuda"), torch.full((2,), 5.0, device="cuda")
    stack = torch.stack(img)
    plan = B.proper_plan_create(0, T, 1)
    try:
        out = []
        for p in (small, large):
            D, S, PD, S2, R2, PR = (torch.full((1, T, T), -7.0, device="cuda") for _ in range(6))
            sig = torch.zeros(1, dtype=torch.float64, device="cuda")
            pn, pr = (torch.from_numpy(q[None].copy()).cuda() for q in p)
            B.argus_zogy(plan, *img, shape, d_rec, 1, pn, pr, p.shape[1], 1e-8, D, S, PD, sig)
            B.argus_proper_coadd(plan, stack, 2, shape, org, 1, F, sg, torch.from_numpy(p).cuda(), p.shape[1], 1e-8, S2,
                                 R2, PR, psf_per_tile=False)
            torch.cuda.synchronize()
            out.append((D, S, PD, sig, S2, R2, PR))
        for a, b in zip(*out):
            assert torch.equal(a, b)
    finally:
        B.proper_plan_destroy(plan)


@pytest.fixture(scope="module")
def host_zogy(tmp_path_factory):
    """The CPU driver of the separated form (one frequency pair at a time, whole transforms)."""
    import os
    import shutil
    import subprocess
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    d = tmp_path_factory.mktemp("host_zogy")
    subprocess.check_call([nvcc, "-O2", "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-I",
                           os.path.join(root, "paper_2207_14304_gb300", "csrc"), "-I", os.path.join(root, "include"),
                           "-o", str(d / "host_zogy"), os.path.join(root, "tests", "host_drivers", "host_zogy.cu")])

    def run(T, **arrays):
        for name, a in arrays.items():
            a.tofile(d / f"{name}.bin")
        np.array([arrays["pn"].shape[0], 0], np.int32).tofile(d / "hdr.bin")
        subprocess.check_call([str(d / "host_zogy"), str(T), str(d)])
        return (np.fromfile(d / f"{k}.bin", np.float32).reshape(T, T) for k in ("D", "S"))
    return run


@pytest.mark.parametrize("T", [256, 512])
def test_zogy_error_is_that_of_separated_images(ora, host_zogy, T):
    """Where N and R agree D is far smaller than either, so an image that stays in D's transforms
    costs precision: the rms errors of D and S are at most 1.1 times those of the form that
    separates the images before the quotient, run on the CPU (the same butterflies; over T^2 pixels
    the two rms figures scatter by less than a per cent, the fused multiply-adds apart)."""
    from oracle import proper
    rng = np.random.default_rng(T + 5)
    Fn, Fr, sn, sr = 1.05, 0.95, 18.0, 3.0
    pn, pr = _gauss(1.8), _gauss(1.2)
    N, R = _frame(T, T, seed=T + 6, sn=sn, sr=sr, psf_n=pn, psf_r=pr, Fn=Fn, Fr=Fr)
    N[rng.integers(0, T, 20), rng.integers(0, T, 20)] += 500.0
    rec = np.zeros(1, B.ZOGY_TILE_DTYPE)
    rec[0] = (0, 0, Fn, Fr, sn, sr)
    o = proper.zogy(N, R, pn.astype(np.float64), pr.astype(np.float64), *(float(rec[0][k]) for k in ("Fn", "Fr", "sn", "sr")))
    plan = B.proper_plan_create(0, T, 1)
    try:
        D, S = (torch.empty((1, T, T), device="cuda") for _ in range(2))
        B.argus_zogy(plan, torch.from_numpy(N).cuda(), torch.from_numpy(R).cuda(), B.argus_shape(T, T, T),
                     torch.from_numpy(rec.view(np.uint8).copy()).cuda(), 1, torch.from_numpy(pn[None].copy()).cuda(),
                     torch.from_numpy(pr[None].copy()).cuda(), 31, 1e-8, D, S)
        torch.cuda.synchronize()
    finally:
        B.proper_plan_destroy(plan)
    rms = lambda a, b: float(np.sqrt(np.mean((a.astype(np.float64) - b) ** 2)))  # noqa: E731
    for name, gpu, cpu in zip("DS", (D, S), host_zogy(T, N=N, R=R, pn=pn, pr=pr, tile=rec)):
        e, bar = rms(gpu[0].cpu().numpy(), o[name]), rms(cpu, o[name])
        print(f"\n[zogy T={T}] rms error of {name}: {e:.3e}, separated on the CPU {bar:.3e}, ratio {e / bar:.3f}")
        assert e <= 1.1 * bar
