"""The composite items of a batch are whole runs of the time steps that a CTA
takes together, one per column block and run."""
import numpy as np
import pytest
import torch

import oracle
import scenes

pytestmark = pytest.mark.gpu

pcdf = pytest.importorskip("paper_2201_05058_gb300")


def test_plan_grows_by_one_item_per_run_of_steps():
    """64 column blocks, no human in the map: 8 more time steps are two more
    items per block (16 bytes each), not eight."""
    grid = scenes.Grid(64, 64, 16, 0.05)
    occ = torch.zeros(grid.shape, dtype=torch.uint8, device="cuda")
    size = {}
    for T in (8, 16):
        caps = np.full((T, 1, 7), -900, np.int32)
        caps[..., 6] = 20
        size[T] = pcdf.Batch([(grid, occ, caps)]).workspace.numel()
    assert size[16] - size[8] < 64 * 3 * 16 + 2048, size


@pytest.mark.parametrize("tiles", [None, (32, 1, 1), (8, 4, 2), (32, 1, 3), (64, 2, 4), (32, 1, 7), (32, 1, 100)])
@pytest.mark.parametrize("T", [1, 4, 5, 9, 14])
def test_every_step_is_computed(tiles, T):
    rng = np.random.default_rng(T)
    envs, want = [], []
    for nx, ny, nz in ((65, 20, 33), (31, 17, 80)):
        grid = scenes.Grid(nx, ny, nz, 0.05)
        occ, _ = scenes.boxes_occupancy(grid, 4, rng)
        c = 16 * np.array([nx, ny, nz])
        caps = np.array([[[30 + 20 * t, c[1] // 2, 20, 30 + 20 * t, c[1] // 2, c[2] - 20, 40]] for t in range(T)], np.int32)
        envs.append((grid, torch.from_numpy(occ).to("cuda"), caps))
        want.append(oracle.predicted_composite(oracle.edt(occ), caps))
    batch = pcdf.Batch(envs, tiles=tiles)
    for f in batch.comp_sq:
        f.fill_(7)
    batch.run()
    assert batch.error() == 0
    for got, w in zip(batch.comp_sq, want):
        assert np.array_equal(got.cpu().numpy(), w)
