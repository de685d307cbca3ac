"""The gradient kernel against the oracle, every stage and the captured filter output bit-exact: every window radius,
images that start at any byte, widths around a tile's 256 columns and its pixel pairs, heights around its 16 rows,
with and without the flatness test's pixels (flat images, textures) and the filter."""
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


CASES = [  # w, h, first byte of the image, texture (0 scene, 1 noise, 2 sparse dots), parameters
    (255, 33, 1, 0, {}), (256, 32, 2, 1, {}), (257, 31, 3, 2, {}), (259, 48, 1, 2, {}), (514, 47, 0, 2, {}),
    (17, 40, 3, 1, {}), (18, 24, 1, 2, {}), (300, 40, 2, 2, {"bilateral": 0}), (301, 40, 1, 1, {"bilateral": 2}),
    (258, 40, 1, 2, {"bf_rho": 1}), (258, 40, 3, 1, {"bf_rho": 2}), (262, 40, 1, 2, {"bf_rho": 3}), (262, 40, 2, 1, {"bf_rho": 4}),
    (261, 40, 0, 2, {"bf_rho": 5, "edge_thresh": 1}), (261, 40, 3, 2, {"bf_rho": 2, "edge_thresh": 200}),
]


@pytest.mark.parametrize("w,h,first,texture,kw", CASES)
def test_grad_tiles(torch_cuda, w, h, first, texture, kw):
    torch = torch_cuda
    d, n = 32, 2
    p = ld.default_params(n_disp=d, **kw)
    frames = [scenes.make_tiny_frame(w, h, d, 31 * w + h + k) for k in range(n)]
    disp, img = np.stack([f[0] for f in frames]), np.stack([f[1] for f in frames])
    rng = np.random.default_rng(w * h + first)
    if texture == 1:
        img = rng.integers(0, 256, (n, h, w), dtype=np.uint8)
    elif texture == 2:
        img = np.where(rng.random((n, h, w)) < 0.004, 255, 100).astype(np.uint8)
    buf = torch.zeros(n * h * w + 8, dtype=torch.uint8, device="cuda")
    dimg = buf[first:first + n * h * w].view(n, h, w)
    dimg.copy_(torch.from_numpy(img))
    det = ld.Detector(w, h, n, p)
    det.capture(True)
    res = ld.Detector.lanes(det.detect(torch.from_numpy(disp).cuda(), dimg))
    for k in range(n):
        compare_frame(det, res[k], k, disp[k], img[k], p)
    det.close()
