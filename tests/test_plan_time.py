"""Planning a composite takes time in proportion to the slab's slices, also
where every slice has cross-sections of its own (tilted humans in a tall slab)."""
import ctypes
import time

import numpy as np

from paper_2201_05058_gb300 import _lib


def us_per_slice(nz, T):
    lib = _lib.load()
    rng = np.random.default_rng(2)
    grid = _lib.PcdfGrid(256, 256, nz, 0.05, (ctypes.c_float * 3)(0, 0, 0))
    caps = np.zeros((T, 3, 7), np.int32)
    caps[..., :2] = rng.integers(300, 3700, (T, 3, 2))
    caps[..., 3:5] = caps[..., :2] + rng.integers(-900, 900, (T, 3, 2))
    caps[..., 2], caps[..., 5], caps[..., 6] = 100, 16 * nz - 100, 60
    need = ctypes.c_size_t(0)
    ptr = caps.ctypes.data_as(ctypes.c_void_p)
    best = float("inf")
    for _ in range(40):
        t0 = time.perf_counter()
        assert lib.pcdf_composite_workspace_bytes(ctypes.byref(grid), T, 3, ptr, ctypes.byref(need)) == 0
        best = min(best, time.perf_counter() - t0)
    return best / (nz * T) * 1e6


def test_tall_slabs_take_no_longer_per_slice():
    """255 slices that all differ took 3.3 times as long per slice as 60 when
    each was compared with all before it."""
    assert us_per_slice(255, 16) < 2 * us_per_slice(60, 64)
