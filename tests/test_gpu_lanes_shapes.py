"""The energy and selection kernels against the oracle, bit-exact: road heights around the energy kernel's
batches of eight rows, frames whose starts just fit the selection's shared-memory copy of the energies and the
next wider ones, many candidates (several warps' worth) with and without suppression, and both lambda_g.
The energy kernel's quotient (two corrections by the exact remainder) is checked on the CPU in exact
arithmetic."""
from fractions import Fraction

import numpy as np
import pytest

from gpu_util import compare_frame
from paper_1807_02752_gb300 import ld, scenes


@pytest.fixture(scope="module")
def torch_cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1807_02752_gb300 import build
    build.build()
    return torch


CASES = [  # w, h, parameters
    (333, 24, {}), (333, 31, {}), (333, 32, {}), (333, 33, {}), (333, 47, {"lambda_g": 0}), (320, 120, {"lambda_g": 0}),
    (640, 60, {"thr_abs": -1, "near_px": 0, "max_lanes": 8}), (640, 60, {"thr_abs": -1, "near_px": 3}),
    (640, 61, {"thr_abs": -1, "near_px": 700, "max_lanes": 8}), (901, 60, {"thr_abs": -1, "max_lanes": 1}),
    (2726, 40, {"thr_abs": -1}), (2727, 40, {"thr_abs": -1}), (2900, 40, {"thr_abs": -1, "near_px": 1}),
]


@pytest.mark.gpu
@pytest.mark.parametrize("w,h,kw", CASES)
def test_lane_selection(torch_cuda, w, h, kw):
    torch = torch_cuda
    d = 32
    p = ld.default_params(n_disp=d, **kw)
    frames = [scenes.make_tiny_frame(w, h, d, 77 * w + h + k) for k in range(2)]
    disp = np.stack([f[0] for f in frames])
    img = np.stack([frames[0][1], np.random.default_rng(w + h).integers(0, 256, (h, w), dtype=np.uint8)])
    det = ld.Detector(w, h, 2, p)
    res = ld.Detector.lanes(det.detect(torch.from_numpy(disp).cuda(), torch.from_numpy(img).cuda()))
    for k in range(2):
        compare_frame(det, res[k], k, disp[k], img[k], p)
    det.close()


def _round32(x: Fraction) -> Fraction:
    """x to the nearest 24-bit binary fraction, ties to even (no exponent limits)."""
    if x == 0:
        return x
    s, a = (1, x) if x > 0 else (-1, -x)
    e = a.numerator.bit_length() - a.denominator.bit_length()
    if a < Fraction(2) ** e:
        e -= 1
    unit = Fraction(2) ** (e - 23)
    return s * unit * round(a / unit)   # round() takes ties to even


def test_quotient_by_reciprocal_is_correctly_rounded():
    rng = np.random.default_rng(5)
    edge = [1 << 23, (1 << 23) + 1, (1 << 24) - 1, (1 << 24) - 2, 3 << 22, (3 << 22) + 1, (3 << 22) - 1]
    pairs = [(n, d) for n in edge for d in edge]
    pairs += [tuple(int(v) for v in rng.integers(1 << 23, 1 << 24, 2)) for _ in range(20000)]
    for ni, di in pairs:
        n, d = Fraction(ni), Fraction(di)
        y = _round32(1 / d)
        q0 = _round32(n * y)
        q1 = _round32(q0 + _round32(n - q0 * d) * y)
        q2 = _round32(q1 + _round32(n - q1 * d) * y)
        assert q2 == _round32(n / d), (ni, di)
