"""The z pass's root of squared distances below 177^2, for every value that a
field can hold there (the sums of three squares) from 148 on, where one of the
three is 8 or more: each as the largest one of a block of free voxels, which
takes that root and not the general one."""
import math

import numpy as np
import pytest
import torch

import oracle
import scenes

pytestmark = pytest.mark.gpu

pcdf = pytest.importorskip("paper_2201_05058_gb300")

FAR = 177 ** 2
LEAST = 3 * 7 ** 2 + 1


def corners():
    """{z^2 + y^2 + x^2: (z, y, x)} with z >= 8 (another block of 8 slices than
    the site's) and y, x as small as can be."""
    two = {}
    for y in range(177):
        for x in range(y + 1):
            two.setdefault(y * y + x * x, (y, x))
    out = {}
    for v in range(LEAST, FAR):
        for z in range(math.isqrt(v), 7, -1):
            if v - z * z in two:
                out[v] = (z,) + two[v - z * z]
                break
    return out


def test_every_root():
    at = corners()
    sums = {z * z + y * y + x * x for z in range(177) for y in range(z + 1) for x in range(y + 1)}
    assert {v for v in sums if LEAST <= v < FAR} == set(at)
    got_sq, got_sdf = [], []
    occ = torch.zeros(256 * 256 * 256, dtype=torch.uint8, device="cuda")
    for z, y, x in at.values():
        nz = (z + 8) // 8 * 8  # the corner (nz - 1, y, x) ends a whole block, the site lies z slices before it
        shape = (nz, y + 1, x + 1)
        o = occ[: math.prod(shape)].view(shape)
        o[nz - 1 - z, 0, 0] = 1
        sq, sdf = pcdf.build_static_sdf(o, scenes.Grid(x + 1, y + 1, nz, 0.05))
        o[nz - 1 - z, 0, 0] = 0
        got_sq.append(sq[-1, -1, -1])
        got_sdf.append(sdf[-1, -1, -1])
    want = np.array(list(at), np.int32)
    assert np.array_equal(torch.stack(got_sq).cpu().numpy(), want)
    assert np.array_equal(torch.stack(got_sdf).cpu().numpy().view(np.int32), oracle.sdf_from_sq(want, 0.05).view(np.int32))
