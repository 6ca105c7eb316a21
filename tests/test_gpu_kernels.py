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


# ------------------------------------------------------------------ dual-number evaluation
RC = O.SW_SI[6] * O.SW_SI[1]
THETA = np.array(O.SW_SI[2:9])


def _dual(N, x, box, w, skin=0.5, cap=48, dtheta=None, shift=0):
    """nefe_sw_dual on a list whose rows start `shift` entries past a 16-byte boundary."""
    n, rcs = len(x), RC + skin
    xd, wd = soa(x), soa(w)
    nbr = torch.zeros(n * cap + shift, dtype=torch.int32, device="cuda")[shift:]
    cnt = torch.zeros(n, dtype=torch.int32, device="cuda")
    N.nefe_neighbor_build(xd, n, box, rcs, cap, nbr, cnt)
    f, fd = (torch.zeros(3 * n, dtype=torch.float64, device="cuda") for _ in range(2))
    out = torch.zeros(16, dtype=torch.float64, device="cuda")
    N.nefe_sw_dual(xd, wd, n, box, rcs, nbr, cnt, cap, N.nefe_sw_params_silicon(), dtheta, f, fd, out)
    torch.cuda.synchronize()
    return f.cpu().numpy().reshape(3, n).T, fd.cpu().numpy().reshape(3, n).T, out.cpu().numpy()


@pytest.mark.parametrize("cap,shift", [(48, 0), (48, 1), (47, 0)])
@pytest.mark.parametrize("n", [64, 65, 127, 1001])
def test_dual_evaluation_at_ragged_sizes(N, n, cap, shift):
    """Groups with a ragged last atom, rows that cannot be read 16 bytes at a time.  Forces to the
    FP64 tolerance of the parity tests (1e-10 of the largest), E' = -F.w and F' symmetric."""
    x, box = I.liquid(max(n, 700), 0.05, seed=n)
    x = x[:n] + np.array([0.0, 300.0, -2.0e5])
    rng = np.random.default_rng(n)
    w, w2 = rng.standard_normal((2, n, 3))
    f, fd, out = _dual(N, x, box, w, cap=cap, shift=shift)
    e_o, f_o, _, _ = O.sw_energy(x, box)
    scale = np.abs(f_o).max()
    # coordinates of 2e5 A carry 3e-11 A: times a stiffness of some 1e2 eV/A^2
    assert np.abs(f - f_o).max() <= 1e-10 * scale + 1e-8
    assert out[1] == pytest.approx(-np.sum(f * w), rel=1e-9, abs=1e-9 * np.abs(f * w).sum())
    _, fd2, _ = _dual(N, x, box, w2, cap=cap, shift=shift)
    assert abs(np.sum(fd * w2) - np.sum(fd2 * w)) <= 1e-10 * np.abs(fd * w2).sum()


def test_dual_evaluation_with_more_edges_than_a_batch(N):
    """A crystal compressed until 28 neighbours lie inside the cutoff: a warp's 32 atoms hold 896
    edges, above the 512 of a batch."""
    x, box = I.diamond(19, 19, 19, a=4.4)
    x = I.rattle(x, 0.05, 3)
    n = len(x)
    f, _, _ = _dual(N, x, box, np.zeros_like(x), skin=0.3, cap=64)
    idx = np.random.default_rng(4).choice(n, 24, replace=False)
    f_o = O.sw_force_atoms(x, box, idx)
    assert np.abs(f[idx] - f_o).max() <= 1e-10 * np.abs(f_o).max()


@pytest.mark.parametrize("kind", ["FL", "RS"])
def test_adjoint_does_not_depend_on_when_lists_are_built(N, kind):
    """A skin so small that every step builds its lists (but above the 2e-5 A margin of the edges'
    filter, so that a row holds every candidate), and skins that keep them for a while: the same W
    and gradient, bit for bit."""
    x0, box = I.diamond(3, 3, 3)
    v0 = I.gaussian_velocities(len(x0), math.sqrt(O.KB * 900.0 / (O.M_SI * O.MVV2E)), 8)
    got = []
    for skin in (1e-3, 0.1, 0.9):
        kw = dict(T=900.0, tdamp=0.1, seed=4, nsched=60, checkpoint_every=7, skin=skin)
        adj = N.Adjoint(x0, v0, box, kind=N.NEFE_SCHED_FL, r0=x0, k_E=5.0, **kw) if kind == "FL" else \
            N.Adjoint(x0, v0, box, kind=N.NEFE_SCHED_RS, lambda_f=0.5, P_GPa=1.0, **kw)
        W = adj.forward(45)
        got.append((W, *adj.backward(initial_state=True)))
        adj.close()
    for g in got[1:]:
        assert g[0] == got[0][0]
        assert all(np.array_equal(a, b) for a, b in zip(g[1:], got[0][1:]))
