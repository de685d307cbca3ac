"""The proposal's top-k against the oracle, bit-exact scores and candidate sets: one start, one more than a warp's
bins, all but one, and more than there are; scores that are all equal, equal in all but few, negative, and that
differ only in the last bits of the order key."""
import numpy as np
import pytest

import oracle
from oracle import proposal as P
from paper_1807_02752_gb300 import ld, scenes
from test_gpu_net import _frames, _oracle_frames, _oracle_learned, torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("top_k", [1, 33, 159, 160, 256])
def test_topk_sets(torch_cuda, top_k):  # noqa: F811
    torch = torch_cuda
    cfg, _ = scenes.WORKLOADS["small_320x120"]
    n = 2
    disp, img, _ = _frames(cfg, n, first=31)
    p, op = ld.default_params(n_disp=cfg.n_disp), oracle.default_params(n_disp=cfg.n_disp)
    det = ld.Detector(cfg.width, cfg.height, n, p)
    net = ld.Net(det)
    mh, mw = P.map_shape(cfg.height, cfg.width)
    rng = np.random.default_rng(top_k)
    flat = np.full((n, mh, mw), 0.5, np.float32)
    dots = np.where(rng.random(flat.shape) < 0.01, np.float32(1), np.float32(0))
    near = (np.float32(1) + rng.integers(0, 3, flat.shape) * np.float32(2.0 ** -23)).astype(np.float32)
    d, i = torch.from_numpy(disp).cuda(), torch.from_numpy(img).cuda()
    rs = _oracle_frames(disp, img, op)
    for z in (flat, dots, near, -near, 0.0 * flat):
        got = ld.Detector.lanes(net.detect(d, i, top_k=top_k, heatmap=torch.from_numpy(z).cuda()))
        for f, r in enumerate(rs):
            starts, energies, flags, sc, cf = _oracle_learned(r, z[f], cfg, op, top_k)
            assert list(got[f]["start_u"][:got[f]["n_lanes"]]) == list(starts), f
            if sc is not None:
                assert np.array_equal(net.debug(f, ld.NET_STAGE_SCORES), sc)
                assert np.array_equal(net.debug(f, ld.NET_STAGE_CFLAG), cf)
    net.close()
    det.close()
