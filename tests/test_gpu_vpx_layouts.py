"""The V_px DP kernel's layouts against the oracle, every stage bit-exact: each number of cells per lane and its
edges (a row that just fits one layout, one column more), eight DP warps, rows spoiled and exchanged at every
tau_x, frames shorter than one exchange, bands that reach every row, the literal bottom band, and energies too
large for packed keys."""
import numpy as np
import pytest

import oracle
from gpu_util import compare_frame, oracle_params
from paper_1807_02752_gb300 import ld, scenes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch_cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1807_02752_gb300 import build
    build.build()
    return torch


def _frame(w, h, d, seed, texture):
    disp, img = scenes.make_tiny_frame(w, h, d, seed)
    if texture:   # edges, and so votes, all over the road
        img = np.random.default_rng(seed).integers(0, 256, (h, w), dtype=np.uint8)
    return disp, img


CASES = [  # w, h, texture, parameters
    (16, 40, True, {}), (255, 40, True, {}), (704, 60, False, {}), (896, 48, True, {}), (897, 48, True, {}),
    (1344, 40, False, {}), (1345, 40, True, {}), (1921, 40, False, {}), (2400, 36, True, {}), (4096, 24, False, {}),
    (320, 20, False, {"chi": 0}), (640, 60, True, {"chi": 100}), (333, 97, True, {"band_literal_bottom": 1}),
    (1242, 60, True, {"tau_x": 0}), (1242, 60, True, {"tau_x": 1}), (700, 60, True, {"tau_x": 2}),
    (1242, 60, True, {"tau_x": 3}), (900, 60, True, {"tau_x": 4}), (1242, 60, True, {"tau_x": 6}),
    (1242, 60, True, {"tau_x": 7, "lambda_x": 0}), (320, 60, True, {"tau_x": 7, "lambda_x": 1000}),
    (1242, 64, True, {"vote_rho": 16, "chi": 256, "bilateral": 0}),              # energies beyond packed keys
    (1300, 64, True, {"vote_rho": 16, "chi": 256, "bilateral": 0, "tau_x": 7, "band_literal_bottom": 1}),
]


@pytest.mark.parametrize("w,h,texture,kw", CASES)
def test_vpx_layouts(torch_cuda, w, h, texture, kw):
    torch = torch_cuda
    d = 32
    p = ld.default_params(n_disp=d, **kw)
    frames = [_frame(w, h, d, 1000 * w + 10 * h + k, texture) for k in range(2)]
    disp, img = np.stack([f[0] for f in frames]), np.stack([f[1] for f in frames])
    det = ld.Detector(w, h, 2, p)
    det.capture(True)
    out = det.detect(torch.from_numpy(disp).cuda(), torch.from_numpy(img).cuda())
    res = ld.Detector.lanes(out)
    for k in range(2):
        compare_frame(det, res[k], k, disp[k], img[k], p)
    det.close()


def test_wide_energies_are_reached():
    """The last two cases above hold enough votes that a key would pass 2^29 (no GPU result needed)."""
    w, h, d = 1242, 64, 32
    p = ld.default_params(n_disp=d, vote_rho=16, chi=256, bilateral=0)
    disp, img = _frame(w, h, d, 1000 * w + 10 * h, True)
    ref = oracle.detect(disp, img, oracle_params(p), dumps=True)
    votes = int(ref["votes"].sum())
    assert (16 * 513 * votes + 5 * h) * 16 >= 2 ** 29
