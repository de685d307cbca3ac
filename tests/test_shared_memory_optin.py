"""A kernel's dynamic shared memory beyond 48 KB needs an opt-in, which the CUDA runtime keeps per kernel and device.
Here the library's own host code runs against a stand-in runtime with two devices (tests/fake/cudart.cpp): every
call that one device serves is served by the other, and no call takes back what another one needs."""
import ctypes as C
import os
import shutil
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CUDA_INCLUDE = "/usr/local/cuda/include"


@pytest.fixture(scope="module")
def built(tmp_path_factory):
    if not shutil.which("g++") or not os.path.exists(os.path.join(CUDA_INCLUDE, "cuda_runtime_api.h")):
        pytest.skip("no host compiler or CUDA headers")
    from paper_1807_02752_gb300 import build
    build.build()
    objs = [os.path.join(build.OBJ_DIR, os.path.basename(s)[:-3] + ".o") for s in build.sources()]
    out = str(tmp_path_factory.mktemp("fake") / "libld_fake.so")
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-I", CUDA_INCLUDE, "-o",
                           out, os.path.join(HERE, "fake", "cudart.cpp"), *objs, "-lpthread", "-ldl", "-lrt"])
    return out


@pytest.fixture
def fake(built, tmp_path, monkeypatch):
    """The library on a fresh stand-in runtime: a copy of its own, as the counters and opt-ins are the process's."""
    from paper_1807_02752_gb300 import ld
    path = str(tmp_path / "libld_fake.so")
    shutil.copy(built, path)
    monkeypatch.setattr(ld, "LIB_PATH", path)
    L = ld.load()
    for name in ("fake_launches", "fake_refused", "fake_lowered"):
        getattr(L, name).restype = C.c_longlong
    for name in ("fake_first_refused", "fake_first_lowered"):
        getattr(L, name).restype = C.c_char_p
    yield ld, L
    ld._libs.pop(path, None)


def _detector(ld, L, w, h, n, **kw):
    p = ld.Params()
    L.ld_params_default(C.byref(p))
    for k, v in kw.items():
        setattr(p, k, v)
    det = C.c_void_p()
    assert L.ld_create(C.byref(p), w, h, n, None, C.byref(det)) == ld.OK
    return det


def test_network_calls_on_a_second_device(fake):
    ld, L = fake
    w, h, n = 320, 120, 2
    mw, mh = (w + 3) // 4, (h + 3) // 4
    xs, lb = np.zeros((n, mh, mw), np.int32), np.zeros((n, mh, mw), np.uint8)
    z, g, loss = np.zeros((n, mh, mw), np.float32), np.zeros(ld.NET_PARAMS, np.float32), np.zeros(1, np.float32)
    disp, img, lanes = np.zeros((n, h, w), np.float32), np.zeros((n, h, w), np.uint8), np.zeros(n, ld.LANES_DTYPE)
    at = lambda a: a.ctypes.data  # noqa: E731
    for device in (0, 1):
        L.fake_set_device(device)
        det, net = _detector(ld, L, w, h, n), C.c_void_p()
        assert L.ld_net_create(det, 1, C.byref(net)) == ld.OK
        for call in (lambda: L.ld_net_forward(net, at(xs), w, h, n, at(z)),
                     lambda: L.ld_net_grad(net, at(xs), at(lb), w, h, n, at(g), at(loss)),
                     lambda: L.ld_net_train_step(net, at(xs), at(lb), w, h, n, 1e-3, at(loss)),
                     lambda: L.ld_detect_learned(net, None, at(disp), at(img), w, h, n, 32, at(lanes)),
                     lambda: L.ld_net_set_fused(net, 1),
                     lambda: L.ld_net_forward(net, at(xs), w, h, n, at(z))):
            assert call() == ld.OK, (device, L.fake_first_refused())
        L.ld_net_destroy(net)
        L.ld_destroy(det)
    assert L.fake_launches() > 40 and L.fake_refused() == 0


def test_stereo_calls_keep_what_other_handles_need(fake):
    """The kernel instances are shared by all handles of a device, also by handles on other threads: a call on narrow
    frames must not lower the allowance that a call on wide ones has made sure of and is about to launch with."""
    ld, L = fake
    for rho in (1, 2, 3):
        sp = ld.StereoParams()
        L.ld_stereo_params_default(C.byref(sp))
        sp.rho = rho
        for w, n in ((1242, 64), (640, 64), (1242, 1), (320, 1), (4096, 2), (64, 80)):
            h = 24
            det, st = _detector(ld, L, w, h, n), C.c_void_p()
            assert L.ld_stereo_create(det, C.byref(sp), C.byref(st)) == ld.OK
            left, out = np.zeros((n, h, w), np.uint8), np.zeros((n, h, w), np.float32)
            assert L.ld_stereo_run(st, left.ctypes.data, left.ctypes.data, w, h, n, out.ctypes.data) == ld.OK
            L.ld_stereo_destroy(st)
            L.ld_destroy(det)
    assert L.fake_launches() > 0 and L.fake_refused() == 0
    assert L.fake_lowered() == 0, L.fake_first_lowered()
