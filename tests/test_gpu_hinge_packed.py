"""HingeCost packs its spheres in the query's own launch when centres and radii
are contiguous float32, and by concatenation otherwise: both give the plain
query's values and gradients, also when the inputs change before the backward
pass, and what was refused stays refused."""
import numpy as np
import pytest
import torch

import scenes

pytestmark = pytest.mark.gpu

pcdf = pytest.importorskip("paper_2201_05058_gb300")


@pytest.mark.parametrize("shape", [(1,), (257,), (3, 5, 7), (0,)])
def test_packed_equals_plain(shape):
    sc = scenes.scene_small_walking(seed=3, T=4, H=1)
    grid = sc["grid"]
    sdf = pcdf.predicted_fields(torch.from_numpy(sc["occ"]).to("cuda"), grid, sc["caps"])[3]
    rng = np.random.default_rng(5)
    sph = torch.from_numpy(rng.uniform(0.1, 3.0, shape + (4,)).astype(np.float32)).to("cuda")
    sph[..., 3] *= 0.05
    tidx = torch.from_numpy(rng.integers(0, 6, shape).astype(np.int32)).to("cuda")
    up = torch.from_numpy(rng.uniform(0.5, 1.5, shape).astype(np.float32)).to("cuda")
    want = pcdf.query_cost(sdf, grid, sph, tidx, 0.2)
    want_c, want_r = pcdf.query_cost_backward(sdf, grid, sph, tidx, 0.2, up)
    for packed in (True, False):
        c = sph[..., :3].clone() if packed else sph[..., :3]  # a slice of the spheres is not contiguous
        r = sph[..., 3].clone() if packed else sph[..., 3]
        c, r = c.detach().requires_grad_(True), r.detach().requires_grad_(True)
        h = pcdf.hinge_cost(c, r, sdf, tidx, 0.2, grid)
        if packed:
            with torch.no_grad():
                c.add_(0.5)  # the spheres of the forward pass are kept
        gc, gr = torch.autograd.grad(h, (c, r), up)
        assert torch.equal(h, want) and torch.equal(gc, want_c) and torch.equal(gr, want_r)
    with pytest.raises((ValueError, RuntimeError)):
        pcdf.hinge_cost(sph[..., :3].double().contiguous(), sph[..., 3].contiguous(), sdf, tidx, 0.2, grid)
