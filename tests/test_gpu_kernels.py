"""Kernels and dispatch branches at the sizes and values where they can go wrong (edges of cells,
of tiles and of blocks), against the FP64 oracle."""
import math

import numpy as np
import pytest

from oracle import oracle as O
from paper_2103_10449_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def N():
    from paper_2103_10449_gb300 import nefe
    nefe.load()
    return nefe


def soa(x):
    return torch.tensor(np.ascontiguousarray(x.T).reshape(-1), dtype=torch.float64, device="cuda")


# ------------------------------------------------------------------ cells
def _edge_positions(box, rcs, far):
    """Coordinates on cell edges, one unit in the last place beside them and a 1e-6 cell beside
    them, in the box and `far` boxes away on either side."""
    nc = [int(np.floor(L / rcs)) for L in box]
    rng = np.random.default_rng(5)
    x = np.zeros((3000, 3))
    for k in range(3):
        cell = rng.integers(-2 * nc[k], 2 * nc[k], len(x)) * (box[k] / nc[k])
        cell = cell + rng.choice([0.0, far, -far], len(x)) * box[k]
        step = rng.choice([0, 1, -1, 2, -2], len(x))
        x[:, k] = np.where(step == 0, cell, cell + np.where(np.abs(step) == 1, np.sign(step) * np.spacing(np.abs(cell)),
                                                            np.sign(step) * 1e-6 * box[k] / nc[k]))
    x[:500] = rng.uniform(-3.0, 3.0, (500, 3)) * box
    return x


@pytest.mark.parametrize("far", [0.0, 7.0, 4.0e4, 3.0e7])
def test_cell_of_coordinates_at_cell_edges(N, far):
    """The integer cell path gives the definition's cell (x / L rounded correctly) everywhere, also
    where its own rounding could cross an edge and beyond its range."""
    box, rcs = np.array([17.3, 23.9, 31.1]), 2.1
    x = _edge_positions(box, rcs, far)
    n = len(x)
    nc_o, cell_o, start_o, perm_o = O.cell_bin(x, box, rcs)
    cap = int(np.prod(nc_o))
    cell, perm = (torch.zeros(n, dtype=torch.int32, device="cuda") for _ in range(2))
    start = torch.zeros(cap + 1, dtype=torch.int32, device="cuda")
    N.nefe_cell_bin(soa(x), n, box, rcs, cell, start, perm, cap)
    torch.cuda.synchronize()
    assert np.array_equal(cell.cpu().numpy(), cell_o)
    assert np.array_equal(start.cpu().numpy(), start_o)
    assert np.array_equal(perm.cpu().numpy(), perm_o)


@pytest.mark.parametrize("cells", [(2, 2, 2), (16, 16, 16), (16, 16, 17), (64, 64, 31), (160, 150, 110)])
def test_cell_scan_over_one_and_several_blocks(N, cells):
    """Grids below, at and above the one-block scan's limit, with a ragged last span."""
    rcs = 1.0
    box = np.array(cells) * (rcs * 1.004)
    x = np.random.default_rng(6).uniform(0.0, 1.0, (2777, 3)) * box
    n = len(x)
    nc_o, cell_o, start_o, perm_o = O.cell_bin(x, box, rcs)
    assert tuple(nc_o) == cells
    cap = int(np.prod(nc_o))
    cell, perm = (torch.zeros(n, dtype=torch.int32, device="cuda") for _ in range(2))
    start = torch.zeros(cap + 1, dtype=torch.int32, device="cuda")
    N.nefe_cell_bin(soa(x), n, box, rcs, cell, start, perm, cap)
    torch.cuda.synchronize()
    assert np.array_equal(cell.cpu().numpy(), cell_o)
    assert np.array_equal(start.cpu().numpy(), start_o)
    assert np.array_equal(perm.cpu().numpy(), perm_o)
