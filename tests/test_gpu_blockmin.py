"""The block search of the y and z passes (csrc/blockmin.cuh) where it can go
wrong: tiles of 64 columns and blocks of 8 elements with remainders, sides from
1 to 512, distances on both sides of the 16-bit range (177 voxels), solid maps
(the other site set), and the float field's root over every squared distance
of that range."""
import numpy as np
import pytest
import torch

import oracle
import scenes

pytestmark = pytest.mark.gpu

pcdf = pytest.importorskip("paper_2201_05058_gb300")


def run(occ, vox=0.05):
    nz, ny, nx = occ.shape
    sq, sdf = pcdf.build_static_sdf(torch.from_numpy(np.ascontiguousarray(occ)).to("cuda"), scenes.Grid(nx, ny, nz, vox))
    return sq.cpu().numpy(), sdf.cpu().numpy()


def squares(shape, at):
    z, y, x = np.ogrid[:shape[0], :shape[1], :shape[2]]
    return ((z - at[0]) ** 2 + (y - at[1]) ** 2 + (x - at[2]) ** 2).astype(np.int32)


def check(occ, want):
    sq, sdf = run(occ)
    assert np.array_equal(sq, want)
    assert np.array_equal(sdf.view(np.int32), oracle.sdf_from_sq(want, 0.05).view(np.int32))


# one occupied (or, solid, one free) voxel: the answer in closed form, with
# every sum of three squares up to 177^2 and beyond
@pytest.mark.parametrize("solid", [False, True])
@pytest.mark.parametrize("shape,at", [((180, 178, 179), (0, 0, 0)), ((9, 8, 512), (8, 0, 511)), ((512, 7, 65), (0, 3, 64)),
                                      ((16, 512, 63), (15, 511, 1)), ((1, 300, 300), (0, 299, 0)), ((177, 1, 178), (176, 0, 0))])
def test_one_voxel(shape, at, solid):
    occ = np.full(shape, int(solid), np.uint8)
    occ[at] = 1 - int(solid)
    want = squares(shape, at)
    if solid:
        want = -want
        want[at] = 1  # the free voxel: its nearest occupied neighbour
    else:
        want[at] = -1
    check(occ, want)


@pytest.mark.parametrize("density", [0.0, 0.0005, 0.03, 0.6, 1.0])
@pytest.mark.parametrize("shape", [(1, 1, 1), (8, 8, 64), (7, 9, 63), (17, 15, 65), (41, 23, 130), (33, 64, 127), (3, 200, 257)])
def test_random_maps(shape, density):
    rng = np.random.default_rng(sum(shape) + int(1e4 * density))
    occ = (rng.random(shape) < density).astype(np.uint8)
    check(occ, oracle.edt(occ))


# far blocks next to near ones: a few voxels in long grids, a thick slab
@pytest.mark.parametrize("shape", [(24, 400, 66), (400, 24, 66), (20, 30, 470)])
def test_sparse_and_thick(shape):
    rng = np.random.default_rng(shape[0])
    occ = np.zeros(shape, np.uint8)
    for _ in range(3):
        occ[tuple(int(rng.integers(0, n)) for n in shape)] = 1
    check(occ, oracle.edt(occ))
    occ[:, : shape[1] // 2] = 1
    check(occ, oracle.edt(occ))


# capsule slices (the same search behind runs instead of row words): runs over
# several words, to both walls, over whole rows and slices, overlapping humans,
# rows that end inside a word, far columns
@pytest.mark.parametrize("nx,ny,nz", [(65, 23, 17), (97, 40, 33), (200, 9, 21), (31, 64, 9), (400, 30, 12)])
def test_capsule_slices(nx, ny, nz):
    c = 16 * np.array([nx, ny, nz])
    caps = [[[8, c[1] // 2, c[2] // 2, c[0] - 8, c[1] // 2, c[2] // 2, 40], [0, 0, 0, 0, 0, 0, 200]],   # wall to wall, and a corner
            [[c[0] // 2, c[1] // 2, 0, c[0] // 2, c[1] // 2, c[2], 130], [c[0] // 2 + 60, c[1] // 2 + 30, 40, c[0] // 2 + 60, c[1] // 2 + 30, 90, 130]],
            [[-200, c[1] // 2, c[2] // 2, 700, c[1] // 2, c[2] // 2, 16 * max(ny, nz)], [30, 30, 30, 30, 30, 30, 17]],   # whole slices
            [[c[0] - 20, 20, 20, c[0] - 20, 20, 20, 30], [-900, -900, -900, -900, -900, -900, 10]]]                     # one small, one outside
    caps = np.array(caps, np.int32)
    static = oracle.edt(scenes.random_occupancy((nz, ny, nx), 0.002, np.random.default_rng(nx)))
    grid = scenes.Grid(nx, ny, nz, 0.05)
    sq, sdf = pcdf.build_predicted_composite(torch.from_numpy(static).to("cuda"), grid, caps)
    want = oracle.predicted_composite(static, caps)
    assert np.array_equal(sq.cpu().numpy(), want)
    assert np.array_equal(sdf.cpu().numpy().view(np.int32), oracle.sdf_from_sq(want, 0.05).view(np.int32))


# the composite's z pass: groups of time steps with a remainder, blocks that are
# copies, near a human, inside one, and out of the 16-bit range (an empty or
# nearly empty map, humans more than 177 voxels away), every output variant
@pytest.mark.parametrize("nx,ny,nz,T,boxes", [(64, 9, 70, 5, 4), (33, 31, 41, 9, 6), (430, 6, 40, 3, 0), (7, 240, 96, 6, 1), (65, 33, 9, 1, 3)])
def test_composite_blocks(nx, ny, nz, T, boxes):
    rng = np.random.default_rng(nx + T)
    grid = scenes.Grid(nx, ny, nz, 0.05)
    occ, _ = scenes.boxes_occupancy(grid, boxes, rng)
    static = oracle.edt(occ)
    sdf = oracle.sdf_from_sq(static, 0.05)
    r = 16 * min(nx, ny, nz) // 3
    top = 16 * nz - 20
    caps = np.array([[[40 + 9 * t, 16 * ny // 2, r, 40 + 9 * t, 16 * ny // 2, max(top - r, r), r],
                      [60, 30 + 5 * t, 30, 60 + 3 * t, 30, top // 2, 25]] for t in range(T)], np.int32)
    want = oracle.predicted_composite(static, caps)
    want_sdf = oracle.sdf_from_sq(want, 0.05).view(np.int32)
    st, sf = torch.from_numpy(static).to("cuda"), torch.from_numpy(sdf).to("cuda")
    for want_sq, want_f, given in ((True, True, sf), (True, True, None), (True, False, None), (False, True, sf), (False, True, None)):
        sq, f = pcdf.build_predicted_composite(st, grid, caps, want_sq=want_sq, want_sdf=want_f, static_sdf=given)
        if want_sq:
            assert np.array_equal(sq.cpu().numpy(), want)
        if want_f:
            assert np.array_equal(f.cpu().numpy().view(np.int32), want_sdf)
    batch = pcdf.Batch([(grid, torch.from_numpy(occ).to("cuda"), caps)])
    batch.run()
    assert batch.error() == 0
    assert np.array_equal(batch.comp_sq[0].cpu().numpy(), want)


# rows read in 16-byte pieces, several to a warp, the last warp not full
@pytest.mark.parametrize("shape", [(3, 11, 32), (5, 7, 64), (7, 3, 128), (5, 5, 256), (1, 1, 512), (1, 3, 512), (2, 9, 96), (3, 3, 100)])
def test_row_words(shape):
    rng = np.random.default_rng(shape[2])
    for density in (0.0, 0.02, 0.5, 0.98):
        occ = (rng.random(shape) < density).astype(np.uint8) * rng.integers(1, 256, shape).astype(np.uint8)
        check(occ, oracle.edt((occ != 0).astype(np.uint8)))


def test_batches_of_different_sizes_side_by_side():
    """A smaller batch planned later does not lower the shared memory that an
    earlier, larger one may launch with."""
    rng = np.random.default_rng(3)
    made = []
    for n in (320, 96, 40):
        grid = scenes.Grid(48, n, 40, 0.05)
        occ, _ = scenes.boxes_occupancy(grid, 5, rng)
        caps = scenes.walking_capsules(grid, 1, 2, rng)
        made.append((pcdf.Batch([(grid, torch.from_numpy(occ).to("cuda"), caps)]), occ, caps))
    for batch, occ, caps in made:
        batch.run()
        assert batch.error() == 0
        assert np.array_equal(batch.comp_sq[0].cpu().numpy(), oracle.predicted_composite(oracle.edt(occ), caps))
