"""What a batch refuses before it reaches the device."""
import ctypes

import pytest

from paper_2201_05058_gb300 import _lib


def create(nz, z0, z1):
    lib = _lib.load()
    caps = (ctypes.c_int32 * 7)(100, 100, 16 * z0 + 8, 120, 100, 16 * z1 + 8, 4)
    env = _lib.PcdfEnv()
    env.grid = _lib.PcdfGrid(16, 16, nz, 0.05, (ctypes.c_float * 3)(0, 0, 0))
    env.T = env.H = 1
    env.caps = ctypes.cast(caps, ctypes.c_void_p)
    env.occ = env.comp_sq = 1 << 20  # never read here
    h = ctypes.c_void_p()
    rc = lib.pcdf_batch_create(ctypes.byref(env), 1, None, ctypes.byref(h))
    msg = lib.pcdf_last_error().decode() if rc else ""
    if h:
        lib.pcdf_batch_destroy(h)
    return rc, msg


@pytest.mark.parametrize("slices,refused", [(500, True), (439, True), (438, False), (45, False)])
def test_tall_slabs_are_refused(slices, refused):
    rc, msg = create(512, 2, 2 + slices - 1)
    assert (rc == -1 and "shared memory" in msg) == refused, (rc, msg)
