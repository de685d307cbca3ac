"""The RANSAC kernels' thread layouts against the oracle: hypothesis counts that divide the CTA, leave threads
idle or need several groups per point list, and paths of more points than threads (tall frames)."""
import numpy as np
import pytest

from gpu_util import compare_frame
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


@pytest.mark.parametrize("w,h,d,kw", [
    (320, 120, 48, {"ransac_hyps": 2}), (320, 120, 48, {"ransac_hyps": 7, "seed": 3}), (320, 120, 48, {"ransac_hyps": 33}),
    (320, 120, 48, {"ransac_hyps": 100}), (320, 120, 48, {"ransac_hyps": 129, "seed": 11}),
    (320, 120, 48, {"ransac_hyps": 255, "tr_x": 0.25}), (640, 1088, 256, {}), (400, 1087, 256, {"ransac_hyps": 9, "tr_x": 1.0}),
])
def test_fit_layouts(torch_cuda, w, h, d, kw):
    torch = torch_cuda
    base = scenes.SMALL_320x120 if h == 120 else scenes.HD_1920x1080
    cfg = scenes.with_size(base, width=w, height=h, n_disp=d, stripe_px=(4.0, 8.0))
    p = ld.default_params(n_disp=d, **kw)
    disp, img, _ = scenes.make_batch(cfg, 2, first_frame=41)
    det = ld.Detector(w, h, 2, p)
    res = ld.Detector.lanes(det.detect(torch.from_numpy(disp).cuda(), torch.from_numpy(img).cuda()))
    for f in range(2):
        compare_frame(det, res[f], f, disp[f], img[f], p)
    det.close()
