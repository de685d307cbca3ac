"""The bounds-checked build on frames without a road, in a workspace of stale values: the stages after the road fit leave
such a frame alone, so nothing they would have written may be tested against a bound."""
import os
import subprocess

import numpy as np
import pytest

from paper_1807_02752_gb300 import ld, scenes

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture
def poisoned(tmp_path, monkeypatch):
    """The bounds-checked library whose fresh device memory holds large numbers (tests/fake/poison.cpp)."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1807_02752_gb300 import build
    build.build(checked=True)
    objs = [os.path.join(build.OBJ_DIR_CHECKED, os.path.basename(s)[:-3] + ".o") for s in build.sources()]
    out = str(tmp_path / "libld_poisoned.so")
    subprocess.check_call([build.nvcc(), *build.ARCH, "-shared", "-Xcompiler", "-fPIC", "-Xlinker", "--wrap=cudaMalloc", "-o",
                           out, os.path.join(HERE, "fake", "poison.cpp"), *objs, "-lcudart_static", "-lrt", "-lpthread",
                           "-ldl"])
    monkeypatch.setattr(ld, "LIB_CHECKED_PATH", out)
    yield torch, ld.load(checked=True)
    ld._libs.pop(out, None)


def test_roadless_frames_in_a_stale_workspace(poisoned):
    torch, L = poisoned
    w, h, n = 320, 120, 8
    disp, img = (np.repeat(x[None], n, 0) for x in scenes.make_tiny_frame(w, h, 32, 3))
    disp[1::2] = 0.0                                     # every other frame has no valid disparity
    det = ld.Detector(w, h, n, ld.default_params(n_disp=32), lib=L)
    assert L.ld_check_reset() == ld.OK
    res = ld.Detector.lanes(det.detect(torch.from_numpy(disp).cuda(), torch.from_numpy(img).cuda()))
    torch.cuda.synchronize()
    assert (res["flags"][1::2] & (ld.F_NO_ROAD | ld.F_DEGEN_Y)).all() and not (res["flags"][::2] & ld.F_NO_ROAD).any()
    st = ld.check_status(L)
    assert st["failures"] == 0, st
    det.close()
