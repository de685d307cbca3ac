"""GPU parity of the network's gradient on maps around the kernels' tile sizes (16 x 8 and 8 x 16 cells) and on
enough tiles that every CTA works through several (its buffers wrap around).

Tolerance: the one of the gradient's parity on whole frames: activations are bf16, so about one stored value
in a hundred rounds to the neighbouring bf16 value (0.4 % of itself), and a parameter group's gradient stays
within 1 % (relative norm) of the float64 oracle's; the loss within 1e-4.
"""
import numpy as np
import pytest

from oracle import proposal as P
from paper_1807_02752_gb300 import ld
from test_gpu_net import init_params

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mw,mh,n", [(8, 16, 2), (9, 17, 2), (16, 8, 1), (17, 9, 3), (10, 33, 1), (31, 7, 2), (33, 17, 300)])
def test_gradient_on_ragged_maps(mw, mh, n):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1807_02752_gb300 import build
    build.build()
    rng = np.random.default_rng(1000 * mw + mh)
    W, H = 4 * mw - 1, 4 * mh - 2          # the last cells of a row and column are partly outside the frame
    det = ld.Detector(W, H, n, ld.default_params(n_disp=16))
    net = ld.Net(det, training=True)
    theta = init_params(9)
    net.set_params(torch.from_numpy(theta).cuda())
    xs = rng.integers(-1 << 22, 1 << 23, (n, mh, mw)).astype(np.int32)
    labels = (rng.random((n, mh, mw)) < 0.05).astype(np.uint8)
    g, loss = net.grad(torch.from_numpy(xs).cuda(), torch.from_numpy(labels).cuda(), W, H)
    net.status()
    g, loss = g.cpu().numpy().astype(np.float64), float(loss.cpu().numpy()[0])
    X = np.stack([P.xmap_input(x) for x in xs])
    want_loss, want = P.loss_and_grad(P.unpack(theta.astype(np.float64)), X, labels)
    assert abs(loss - want_loss) <= 1e-4 * abs(want_loss)
    gd = P.unpack(g)
    for name, _ in P.param_shapes():
        a, b = gd[name].ravel(), want[name].ravel()
        assert np.linalg.norm(a - b) <= 1e-2 * np.linalg.norm(b) + 1e-12, (name, np.linalg.norm(a - b), np.linalg.norm(b))
    net.close()
    det.close()
