"""GPU parity of the stereo kernel's launch shapes: a whole map per CTA, maps split over clusters of 2, 4 and 8
CTAs (by the number of pairs and the width), one and two search warps per strip, the scattered-search path and
the exact comparison of near-equal scores.  Integer decisions: every map equals the oracle's."""
import numpy as np
import pytest

import oracle
from paper_1807_02752_gb300 import ld

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch_cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1807_02752_gb300 import build
    build.build()
    return torch


def _pair(rng, w, h, kind):
    if kind == "noise":          # no match anywhere: scattered estimates
        return rng.integers(0, 256, (h, w), dtype=np.uint8), rng.integers(0, 256, (h, w), dtype=np.uint8)
    if kind == "periodic":       # equal scores at every period, and a constant band (NCC 0)
        row = np.tile(np.array([10, 200, 90, 30], np.uint8), w // 4 + 2)
        left = np.stack([row[v % 2:v % 2 + w] for v in range(h)])
        left[h // 3:h // 2] = 77
        return left, np.roll(left, -4, axis=1)
    left = np.clip(100 + rng.normal(0, 25, (h, w)), 0, 255).astype(np.uint8)   # shifted texture, a step in depth
    right = np.roll(left, -9, axis=1)
    right[:, w // 2:] = np.roll(left, -21, axis=1)[:, w // 2:]
    right = np.clip(right + rng.integers(-4, 5, right.shape), 0, 255).astype(np.uint8)
    return left, right


@pytest.mark.parametrize("w,h,n,kind,kw", [
    (1242, 40, 1, "shift", {}), (1242, 40, 1, "noise", {}), (1242, 40, 1, "periodic", {}),
    (1241, 24, 10, "shift", {}), (1243, 24, 30, "noise", {}), (1242, 24, 40, "shift", {}),
    (1242, 24, 40, "noise", {}), (774, 40, 1, "shift", {"rho": 1}), (1411, 40, 2, "noise", {"rho": 2, "tau": 2}),
    (4096, 20, 1, "shift", {"d_max": 1023}), (4095, 18, 40, "shift", {"tau": 5}), (1242, 20, 1, "noise", {"tau": 64}),
    (197, 33, 1, "shift", {"tau": 0}), (198, 33, 1, "noise", {"d_max": 1023}), (1920, 24, 3, "shift", {"d_max": 255}),
    (16, 16, 1, "noise", {}), (1242, 20, 40, "periodic", {"rho": 2}),
])
def test_stereo_launch_shapes(torch_cuda, w, h, n, kind, kw):
    torch = torch_cuda
    rng = np.random.default_rng([w, h, n])
    pairs = [_pair(rng, w, h, kind) for _ in range(n)]
    left, right = np.stack([p[0] for p in pairs]), np.stack([p[1] for p in pairs])
    det = ld.Detector(w, h, n, ld.default_params(n_disp=128))
    sp = ld.stereo_params(**kw)
    st = ld.Stereo(det, sp)
    disp = st.run(torch.from_numpy(left).cuda(), torch.from_numpy(right).cuda()).cpu().numpy()
    dmax = sp.d_max if sp.d_max >= 0 else 127
    for f in sorted({0, n // 2, n - 1}):
        lf, rt, d = oracle.stereo(left[f], right[f], sp.rho, dmax, sp.tau, sp.tr_lrc)
        glf, grt, _ = st.maps(f, w, h)
        assert np.array_equal(glf, lf), (f, "left map")
        assert np.array_equal(grt, rt), (f, "right map")
        assert np.array_equal(disp[f], d.astype(np.float32)), (f, "checked disparity")
    st.close()
    det.close()
