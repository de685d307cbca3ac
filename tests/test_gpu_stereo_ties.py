"""Stereo maps where many candidates have the same score, against the oracle: images constant along their rows or
repeating within a search range, near ties, and such regions next to texture.  Ties go to the smaller disparity and
everything closer than the float scores can tell is compared in integers."""
import numpy as np
import pytest

import oracle
from paper_1807_02752_gb300 import ld

pytestmark = pytest.mark.gpu


def _pair(rng, w, h, kind):
    rows = (np.arange(h) * 7 % 251).astype(np.uint8)[:, None]
    if kind == "rows":            # every candidate of a pixel has the same N and D
        left = np.repeat(rows, w, axis=1)
        return left, left.copy()
    if kind == "period":          # ties at every period of 2, 3 and 5 columns
        u = np.arange(w)
        left = np.stack([(37 * ((u + v) % (2, 3, 5)[v // 8 % 3]) + v) % 256 for v in range(h)]).astype(np.uint8)
        return left, np.roll(left, -3, axis=1)
    if kind == "near":            # rows but for a few pixels: scores that differ in their last bits
        left = np.repeat(rows, w, axis=1)
        left[rng.random((h, w)) < 0.02] += 1
        right = np.repeat(rows, w, axis=1)
        right[rng.random((h, w)) < 0.02] += 1
        return left, right
    left = rng.integers(0, 256, (h, w), dtype=np.uint8)      # "mixed": flat, constant rows and texture side by side
    right = np.roll(left, -6, axis=1)
    for x in (left, right):
        x[:, w // 4:w // 2] = rows
        x[h // 3:h // 2] = 131
    return left, right


@pytest.mark.parametrize("w,h,n,kind,kw", [
    (1242, 40, 1, "rows", {}), (1242, 40, 44, "rows", {}), (1242, 40, 1, "near", {}), (1242, 40, 44, "near", {}),
    (1242, 48, 1, "period", {}), (1241, 48, 40, "period", {"tau": 4}), (777, 48, 2, "mixed", {"rho": 1}),
    (1242, 48, 44, "mixed", {"rho": 2}), (1920, 32, 3, "near", {"rho": 2, "tau": 3}), (320, 64, 1, "near", {"rho": 1, "tau": 2}),
    (333, 40, 80, "near", {"rho": 1}), (4096, 20, 2, "near", {"d_max": 300}), (64, 33, 1, "period", {"rho": 1}),
    (200, 33, 90, "mixed", {"tau": 0}),
])
def test_ties(torch_cuda, w, h, n, kind, kw):
    torch = torch_cuda
    rng = np.random.default_rng([w, h, n])
    pairs = [_pair(rng, w, h, kind) for _ in range(min(n, 3))]
    pairs = [pairs[k % len(pairs)] for k in range(n)]
    left, right = np.stack([p[0] for p in pairs]), np.stack([p[1] for p in pairs])
    det = ld.Detector(w, h, n, ld.default_params(n_disp=64))
    sp = ld.stereo_params(**kw)
    st = ld.Stereo(det, sp)
    disp = st.run(torch.from_numpy(left).cuda(), torch.from_numpy(right).cuda()).cpu().numpy()
    dmax = sp.d_max if sp.d_max >= 0 else 63
    for f in sorted({0, min(n - 1, 1), n - 1}):
        lf, rt, d = oracle.stereo(left[f], right[f], sp.rho, dmax, sp.tau, sp.tr_lrc)
        glf, grt, _ = st.maps(f, w, h)
        assert np.array_equal(glf, lf), (f, "left map")
        assert np.array_equal(grt, rt), (f, "right map")
        assert np.array_equal(disp[f], d.astype(np.float32)), (f, "checked disparity")
    st.close()
    det.close()
