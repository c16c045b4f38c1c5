"""The C struct of a grid is made from the grid's values at the time of the call,
of whatever number type they are."""
from types import SimpleNamespace

import numpy as np
import pytest
import torch

pcdf = pytest.importorskip("paper_2201_05058_gb300")

from paper_2201_05058_gb300 import api  # noqa: E402


def fields(grid):
    g = api._cgrid(grid)
    return g.nx, g.ny, g.nz, round(g.vox, 6), tuple(g.origin)


@pytest.mark.parametrize("number", [np.array, np.float32, torch.tensor, float])
def test_number_types(number):
    grid = SimpleNamespace(nx=number(5), ny=number(6), nz=number(7), vox=number(0.25), origin=tuple(number(v) for v in (1.0, 2.0, 3.0)))
    assert fields(grid) == (5, 6, 7, 0.25, (1.0, 2.0, 3.0))
    grid.origin = [number(4.0), 5, number(6.0)]
    assert fields(grid) == (5, 6, 7, 0.25, (4.0, 5.0, 6.0))


def test_values_changed_in_place():
    origin, vox = torch.zeros(3), torch.tensor(0.5)
    grid = SimpleNamespace(nx=4, ny=4, nz=4, vox=vox, origin=tuple(origin))
    assert fields(grid) == (4, 4, 4, 0.5, (0.0, 0.0, 0.0))
    for v in grid.origin:
        v += 1
    vox += 1
    assert fields(grid) == (4, 4, 4, 1.5, (1.0, 1.0, 1.0))
