"""Batches take their device in every form that PyTorch takes it."""
import numpy as np
import pytest
import torch

import oracle
import scenes

pytestmark = pytest.mark.gpu

pcdf = pytest.importorskip("paper_2201_05058_gb300")


@pytest.mark.parametrize("device", ["cuda", "cuda:0", 0, torch.device("cuda"), None])
def test_device_forms(device):
    rng = np.random.default_rng(7)
    grid = scenes.Grid(33, 20, 17, 0.05)
    occ, _ = scenes.boxes_occupancy(grid, 4, rng)
    caps = scenes.walking_capsules(grid, 1, 3, rng)
    envs = [(grid, torch.from_numpy(occ).to("cuda"), caps)]
    batch = pcdf.Batch(envs, device=device)
    batch.run()
    assert batch.error() == 0
    assert np.array_equal(batch.comp_sq[0].cpu().numpy(), oracle.predicted_composite(oracle.edt(occ), caps))
    tiles, ms = pcdf.batch_autotune(envs, reps=1, device=device)
    assert len(tiles) == 3 and ms > 0
