"""Warp-wide and cluster-wide instructions that follow code only some lanes execute.  Such code has to bring the
warp together again; what follows is compared where every exchange has storing and silent lanes in one warp."""
import numpy as np
import pytest

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


@pytest.mark.parametrize("w,h,rho", [(1242, 121, 3), (777, 97, 1), (1613, 64, 2)])
def test_cluster_exchange_equals_whole_maps(torch_cuda, w, h, rho):
    """One pair, whose maps are split over clusters that exchange their edge estimates every eight rows (a store per
    edge lane, then the cluster barrier), gives the maps of the same pair in a batch
    that takes as few CTAs a map as the width allows."""
    torch = torch_cuda
    rng = np.random.default_rng([w, h, rho])
    left = rng.integers(0, 256, (h, w), dtype=np.uint8)
    right = np.clip(np.roll(left, -11, axis=1).astype(int) + rng.integers(-6, 7, left.shape), 0, 255).astype(np.uint8)
    n = 96
    det = ld.Detector(w, h, n, ld.default_params(n_disp=64))
    st = ld.Stereo(det, ld.stereo_params(rho=rho))
    many = [torch.from_numpy(np.repeat(x[None], n, 0)).cuda() for x in (left, right)]
    one = [x[:1].contiguous() for x in many]
    st.run(*many)
    want = [st.maps(f, w, h) for f in (0, n - 1)]
    for _ in range(3):
        st.run(*one)
        got = st.maps(0, w, h)
        for ref in want:
            assert np.array_equal(got[0], ref[0]) and np.array_equal(got[1], ref[1])
    st.close()
    det.close()
