"""The V_px backtrack rows lie in the frame's part of M_1: narrow frames, whose part is small and starts at any multiple of
four bytes, alone and in one launch with wide ones."""
import numpy as np
import pytest

from gpu_util import compare_frame
from paper_1807_02752_gb300 import ld, scenes

pytestmark = pytest.mark.gpu


def _frame(w, h, seed):
    disp, _ = scenes.make_tiny_frame(w, h, 16, seed)
    return disp, np.random.default_rng([w, h, seed]).integers(0, 256, (h, w), dtype=np.uint8)


@pytest.mark.parametrize("w,h", [(16, 16), (17, 33), (23, 47), (28, 61), (31, 45), (33, 39), (97, 51), (241, 75)])
def test_narrow_frames(torch_cuda, w, h):
    torch = torch_cuda
    p = ld.default_params(n_disp=16, bilateral=0)
    frames = [_frame(w, h, k) for k in range(5)]
    disp, img = np.stack([f[0] for f in frames]), np.stack([f[1] for f in frames])
    det = ld.Detector(w, h, 5, p)
    res = ld.Detector.lanes(det.detect(torch.from_numpy(disp).cuda(), torch.from_numpy(img).cuda()))
    for k in range(5):
        compare_frame(det, res[k], k, disp[k], img[k], p)
    det.close()


def test_narrow_frames_among_wide_ones(torch_cuda):
    torch = torch_cuda
    p = ld.default_params(n_disp=16, bilateral=0)
    sizes = [(2401, 40, 2), (16, 16, 3), (19, 39, 3), (1345, 33, 1), (22, 17, 5)]
    det = ld.Detector(2401, 40, sum(s[2] for s in sizes), p)
    groups = []
    for w, h, n in sizes:
        frames = [_frame(w, h, k) for k in range(n)]
        groups.append(tuple(torch.from_numpy(np.stack([f[q] for f in frames])).cuda() for q in (0, 1)))
    got = [ld.Detector.lanes(o) for o in det.detect_groups(groups, mixed=True)]
    for (w, h, n), (d, i), res in zip(sizes, groups, got):
        alone = ld.Detector(w, h, n, p)
        assert res.tobytes() == ld.Detector.lanes(alone.detect(d, i)).tobytes(), (w, h)
        alone.close()
    det.close()
