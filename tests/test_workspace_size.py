"""Device memory of a handle, counted by the stand-in runtime: a server's memory budget buys a number of them, so they may
not grow."""
import ctypes as C

import pytest

from test_shared_memory_optin import _detector, built, fake  # noqa: F401  (fixtures)

# bytes of a handle with default parameters while the V_px backtrack kept a buffer of half a byte a pixel
BYTES = {(16, 16, 1): 113920, (320, 120, 8): 6679040, (1242, 375, 64): 596044288, (1241, 376, 8): 74728960,
         (1920, 1080, 16): 657056256, (4096, 1088, 2): 175223808}


@pytest.mark.parametrize("w,h,n", sorted(BYTES))
def test_handles_do_not_grow(fake, w, h, n):  # noqa: F811
    ld, L = fake
    L.fake_allocated.restype = C.c_longlong
    det = _detector(ld, L, w, h, n)
    assert L.fake_allocated() <= BYTES[w, h, n]
    L.ld_destroy(det)
