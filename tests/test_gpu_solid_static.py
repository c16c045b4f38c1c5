"""Composite fields where the static map is solid over whole blocks of the z
stage (64 columns, 8 slices): a wall, a floor, a ceiling slice alone in the
last block, a grid one slice thick, a nearly solid map and a solid tail of
columns, with humans inside and beside.  The composite is the least of the two
signed fields, so a voxel inside a human and a wall takes the deeper value."""
import numpy as np
import pytest
import torch

import oracle
import scenes

pytestmark = pytest.mark.gpu

pcdf = pytest.importorskip("paper_2201_05058_gb300")


def solid_map(kind, nx, ny, nz):
    occ = np.zeros((nz, ny, nx), np.uint8)
    if kind == "wall":          # one voxel thick, along x over the whole height
        occ[:, ny // 2] = 1
    elif kind == "floor":       # fills the first block of slices
        occ[:8] = 1
    elif kind == "floor16":
        occ[:min(16, nz)] = 1
    elif kind == "ceiling":     # the last slice
        occ[-1] = 1
    elif kind == "free voxel":  # solid but for one voxel in a corner
        occ[:] = 1
        occ[-1, -1, -1] = 0
    elif kind == "tail":        # the last rows: the last, short tile of columns is solid
        occ[:, ny - 2:] = 1
    return occ


# humans through the middle, at the floor, at the ceiling and the far corner,
# and one some voxels away from the wall
def humans(nx, ny, nz, T):
    r = 16 * min(5, max(nx, ny, nz))
    cx, cy = 8 * nx, 8 * (ny // 2 * 2 + 1)
    out = []
    for t in range(T):
        x = cx + 21 * t
        out.append([[x, cy, 0, x, cy, 16 * nz, r],
                    [x - 200, cy + 16 * 8, 40, x - 200, cy + 16 * 8, 90, r],
                    [16 * nx - 10, 16 * ny - 20, 16 * nz - 30, 16 * nx - 60, 16 * ny - 20, 16 * nz + 20, r + 16]])
    return np.array(out, np.int32)


def same(got, want, vox):
    sq, sdf = got
    if sq is not None:
        assert np.array_equal(sq.cpu().numpy(), want)
    if sdf is not None:
        assert np.array_equal(sdf.cpu().numpy().view(np.int32), oracle.sdf_from_sq(want, vox).view(np.int32))


@pytest.mark.parametrize("kind", ["wall", "floor", "floor16", "ceiling", "free voxel", "tail"])
@pytest.mark.parametrize("nx,ny,nz,T", [(64, 40, 41, 5), (128, 24, 48, 3), (97, 33, 25, 6), (130, 21, 1, 2)])
def test_humans_in_solid_blocks(kind, nx, ny, nz, T):
    grid = scenes.Grid(nx, ny, nz, 0.05)
    occ, caps = solid_map(kind, nx, ny, nz), humans(nx, ny, nz, T)
    static = oracle.edt(occ)
    sdf = oracle.sdf_from_sq(static, grid.vox)
    want = oracle.predicted_composite(static, caps)
    if not occ.all():
        assert (want < static)[:, occ != 0].any()  # some human is deeper in the solid part than its own depth
    st, sf, oc = (torch.from_numpy(a).to("cuda") for a in (static, sdf, occ))
    for want_sq, want_f, given in ((True, True, sf), (True, True, None), (True, False, None), (False, True, sf), (False, True, None)):
        same(pcdf.build_predicted_composite(st, grid, caps, want_sq=want_sq, want_sdf=want_f, static_sdf=given), want, grid.vox)
    fields = pcdf.predicted_fields(oc, grid, caps)
    same(fields[2:], want, grid.vox)
    ws = pcdf.composite_workspace(grid, caps, st.device)
    pcdf.composite_prepare(grid, caps, ws)
    sq = torch.zeros((T,) + grid.shape, dtype=torch.int32, device="cuda")
    f = torch.zeros((T,) + grid.shape, device="cuda")
    for t0, nt in ((0, 1), (1, T - 1)):
        pcdf.composite_finish(st, grid, caps, ws, sq, f, static_sdf=sf, t_range=(t0, nt))
    same((sq, f), want, grid.vox)
    ctx = pcdf.Context("cuda")
    same(ctx.build_predicted_composite(st, grid, caps, static_sdf=sf), want, grid.vox)
    ctx.close()
    batch = pcdf.Batch([(grid, oc, caps)] * 2)
    batch.run()
    assert batch.error() == 0
    for got in batch.comp_sq:
        same((got, None), want, grid.vox)
