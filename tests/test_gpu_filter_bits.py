"""The voxel filter in bit planes and the collapsed map: widths of 16- and 4-byte
rows around the tile of 256 voxels, remainders of its 8 rows and 8 slices, any
non-zero byte as occupied, every threshold, and unaligned maps."""
import numpy as np
import pytest
import torch

import oracle
import scenes

pytestmark = pytest.mark.gpu

pcdf = pytest.importorskip("paper_2201_05058_gb300")


@pytest.mark.parametrize("nx,ny,nz", [(4, 1, 1), (16, 9, 8), (28, 7, 17), (256, 8, 9), (260, 3, 5), (272, 17, 3), (512, 2, 10), (37, 10, 9)])
def test_filter_and_collapse(nx, ny, nz):
    rng = np.random.default_rng(nx + ny)
    grid = scenes.Grid(nx, ny, nz, 0.05)
    for density in (0.05, 0.4, 1.0):
        occ = (rng.random((nz, ny, nx)) < density).astype(np.uint8)
        raw = occ * rng.integers(1, 256, occ.shape).astype(np.uint8)
        aligned = torch.from_numpy(raw).to("cuda")
        shifted = torch.empty(raw.size + 1, dtype=torch.uint8, device="cuda")[1:].view(raw.shape).copy_(aligned)
        want = oracle.collapse(occ, 1 if nz > 2 else 0, nz)
        for dev in (aligned, shifted):
            for least in (0, 1, 5, 13, 26, 27):
                got = pcdf.filter_voxels(dev, grid, least).cpu().numpy()
                assert np.array_equal(got, oracle.voxel_filter(occ, least)), (density, least)
            assert np.array_equal(pcdf.collapse_2d(dev, grid, 1 if nz > 2 else 0, nz).cpu().numpy(), want)
