"""The V_px DP's packed keys at and beyond the energies they hold, and its layouts at their edges, against the oracle with
every stage bit-exact.

Keys hold 16 E down to -(2^30 - 2^20) at an exchange; a frame whose path gathers more is done again with plain energies.
The radial frames put up to a sixth of all votes into the vanishing point's columns, which is what that takes."""
import numpy as np
import pytest

import oracle
from gpu_util import compare_frame, oracle_params
from paper_1807_02752_gb300 import ld, scenes

LIMIT = 2 ** 26 - 2 ** 16      # energy of a path at which the packed rows end


def _radial(period, w=120, h=1088, d=256, h0=30):
    """A flat road to row h0 whose texture is constant along the lines through one point on the horizon."""
    v, u = np.arange(h)[:, None], np.arange(w)[None, :]
    disp = np.where(v > h0, np.broadcast_to((d - 6) * (v - h0) / (h - 1 - h0), (h, w)), 0).astype(np.float32)
    angle = 600 * (u - (w // 2 + 0.25)) / np.maximum(v - h0, 1)
    img = np.round(510 * np.abs((angle / period) % 1 - 0.5)).astype(np.uint8)
    return disp, np.ascontiguousarray(img)


def _params(**kw):
    return ld.default_params(n_disp=256, bilateral=0, vote_rho=16, chi=256, lambda_x=0, **kw)


def _path_energy(ref, h):
    return -sum(int(ref["m_x"][v, ref["path_x"][v]]) for v in range(ref["v_top"], h))


RADIAL = [(4.0, {"tau_x": 2}), (6.0, {"tau_x": 5}), (14.0, {"tau_x": 0}), (14.0, {"tau_x": 2}), (9.0, {"tau_x": 7}),
          (14.0, {"tau_x": 3, "band_literal_bottom": 1})]


@pytest.mark.gpu
@pytest.mark.parametrize("period,kw", RADIAL)
def test_large_energies(torch_cuda, period, kw):
    torch = torch_cuda
    p = _params(**kw)
    big, small = _radial(period), scenes.make_tiny_frame(120, 1088, 256, 5)
    disp, img = np.stack([big[0], small[0], big[0]]), np.stack([big[1], small[1], big[1]])
    det = ld.Detector(120, 1088, 3, p)
    det.capture(True)
    res = ld.Detector.lanes(det.detect(torch.from_numpy(disp).cuda(), torch.from_numpy(img).cuda()))
    for k in range(3):
        compare_frame(det, res[k], k, disp[k], img[k], p)
    det.close()


def test_radial_frames_lie_on_both_sides_of_the_limit(oracle_mod):
    for period, beyond in ((4.0, False), (6.0, True), (9.0, True), (14.0, True)):
        disp, img = _radial(period)
        ref = oracle.detect(disp, img, oracle_params(_params(tau_x=2)), dumps=True)
        e = _path_energy(ref, 1088)
        assert e > LIMIT if beyond else LIMIT // 2 < e < LIMIT, (period, e)


LAYOUTS = [(w, 44, {}) for w in (704, 705, 768, 769, 832, 833, 1152, 1153, 1248, 1249, 2240, 2241, 2400)] + [
    (2401, 60, {}), (3333, 97, {}), (4096, 64, {"tau_x": 1}), (4096, 64, {"tau_x": 7}), (2401, 60, {"tau_x": 7, "lambda_x": 0}),
    (3333, 50, {"tau_x": 0}), (2560, 40, {"tau_x": 0}), (2561, 40, {"tau_x": 0}),
    (1242, 64, {"vote_rho": 16, "chi": 256}), (1300, 64, {"vote_rho": 16, "chi": 256, "tau_x": 7})]


@pytest.mark.gpu
@pytest.mark.parametrize("w,h,kw", LAYOUTS)
def test_layout_edges_with_texture(torch_cuda, w, h, kw):
    """The widths at which cells per lane, warps or rows per exchange change, with votes all over the road."""
    torch = torch_cuda
    p = ld.default_params(n_disp=32, bilateral=0, **kw)
    disp, _ = scenes.make_tiny_frame(w, h, 32, 1000 * w + h)
    img = np.random.default_rng([w, h]).integers(0, 256, (h, w), dtype=np.uint8)
    det = ld.Detector(w, h, 1, p)
    det.capture(True)
    res = ld.Detector.lanes(det.detect(torch.from_numpy(disp[None].copy()).cuda(), torch.from_numpy(img[None]).cuda()))
    ref = compare_frame(det, res[0], 0, disp, img, p)
    assert ref["votes"].sum() > 20 * (h - ref["v_top"])
    det.close()


def _slanted(w, h, centre, slope, seed):
    """A road whose only texture is a band of vertical stripes that moves `slope` columns a row: its votes stay in it, so
    the path follows it."""
    disp, img = scenes.make_tiny_frame(w, h, 32, seed)
    img[:] = 90
    u = np.arange(w)
    for v in range(h):
        at = centre + slope * (v - 3 * h // 4)
        inside = np.abs(u - at) < 14
        img[v, inside] = np.where((u[inside] // 2) % 2 == 0, 20, 235)
    return disp, img


# (width, rows, a column where one DP warp's cells end and the next one's begin, tau_x)
CROSSINGS = [(1242, 120, 312, 5), (1242, 120, 624, 5), (704, 100, 352, 5), (1152, 100, 864, 5), (1920, 120, 1120, 5),
             (2401, 120, 1120, 5), (2401, 120, 1680, 5), (4096, 100, 3360, 5), (4096, 100, 2080, 7), (1249, 100, 672, 7)]


@pytest.mark.parametrize("w,h,column,tau", CROSSINGS)
def test_slanted_paths_cross(w, h, column, tau, oracle_mod):
    for slope in (3, -3):
        disp, img = _slanted(w, h, column, slope, 7)
        p = ld.default_params(n_disp=32, bilateral=0, chi=2, lambda_x=0, tau_x=tau)
        ref = oracle.detect(disp, img, oracle_params(p), dumps=True)
        path = ref["path_x"][ref["v_top"]:]
        assert path.min() < column - 20 and path.max() > column + 20, (slope, path.min(), path.max())


@pytest.mark.gpu
@pytest.mark.parametrize("w,h,column,tau", CROSSINGS)
def test_paths_across_warps(torch_cuda, w, h, column, tau):
    torch = torch_cuda
    p = ld.default_params(n_disp=32, bilateral=0, chi=2, lambda_x=0, tau_x=tau)
    frames = [_slanted(w, h, column, slope, 7) for slope in (3, -3)]
    disp, img = np.stack([f[0] for f in frames]), np.stack([f[1] for f in frames])
    det = ld.Detector(w, h, 2, p)
    det.capture(True)
    res = ld.Detector.lanes(det.detect(torch.from_numpy(disp).cuda(), torch.from_numpy(img).cuda()))
    for k in range(2):
        compare_frame(det, res[k], k, disp[k], img[k], p)
    det.close()
