"""Warp-wide and cluster-wide instructions that follow code only some lanes execute.  Such code has to bring the
warp together again; what follows is compared where every exchange has storing and silent lanes in one warp."""
import numpy as np
import pytest

from gpu_util import compare_frame
from paper_1807_02752_gb300 import ld, scenes

pytestmark = pytest.mark.gpu


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


@pytest.mark.parametrize("w,h", [(1242, 90), (705, 75)])
def test_uneven_vote_rows(torch_cuda, w, h):
    """V_px producers clear their rows of the ring and add votes in loops that end per lane, then meet at a barrier of
    their own: rows of very uneven vote counts, every stage against the oracle."""
    torch = torch_cuda
    disp, img = scenes.make_tiny_frame(w, h, 32, 11)
    rng = np.random.default_rng([w, h])
    for v in range(h // 2, h, 3):                    # texture on every third road row, of growing width
        n = 16 + (v - h // 2) * w // h
        img[v, :n] = rng.integers(0, 256, n, dtype=np.uint8)
    p = ld.default_params(n_disp=32, bilateral=0)
    det = ld.Detector(w, h, 1, p)
    det.capture(True)
    res = ld.Detector.lanes(det.detect(torch.from_numpy(disp[None].copy()).cuda(), torch.from_numpy(img[None]).cuda()))
    ref = compare_frame(det, res[0], 0, disp, img, p)
    counts = ref["votes"].sum(axis=1)
    assert counts.max() > 64 and (counts[counts > 0] % 32 != 0).any()
    det.close()


@pytest.mark.parametrize("w,h,n", [(264, 130, 3), (1000, 68, 2)])
def test_network_maps_of_partial_tiles(torch_cuda, w, h, n):
    """k_conv_tc copies halos and stores cells in loops that end per lane, then reads tensor memory with warp-wide
    loads: the per-layer forward is the fused one's, bit for bit, over several tiles per block."""
    torch = torch_cuda
    rng = np.random.default_rng([w, h, n])
    det = ld.Detector(w, h, n, ld.default_params(n_disp=32))
    net = ld.Net(det)
    net.set_params(torch.from_numpy((rng.standard_normal(ld.NET_PARAMS) * 0.1).astype(np.float32)).cuda())
    mh, mw = ld.Net.map_shape(w, h)
    x = torch.from_numpy(rng.integers(0, 1 << 22, (n, mh, mw), dtype=np.int32)).cuda()
    per_layer = net.forward(x, w, h).cpu().numpy()
    net.set_fused(True)
    assert np.array_equal(net.forward(x, w, h).cpu().numpy(), per_layer)
    net.close()
    det.close()
