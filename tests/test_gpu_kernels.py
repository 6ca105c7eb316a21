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


# ------------------------------------------------------------------ scatter form
def _forces32(N, x, box, skin, cap, shift=0):
    n, rcs = len(x), RC + skin
    xd = soa(x)
    nbr = torch.zeros(n * cap + shift, dtype=torch.int32, device="cuda")[shift:]
    nbr.fill_(-1)                                       # what lies past a row's length is the caller's
    cnt = torch.zeros(n, dtype=torch.int32, device="cuda")
    N.nefe_neighbor_build(xd, n, box, rcs, cap, nbr, cnt)
    f = torch.zeros(3 * n, dtype=torch.float64, device="cuda")
    e = torch.zeros(n, dtype=torch.float64, device="cuda")
    ev = torch.zeros(7, dtype=torch.float64, device="cuda")
    N.nefe_sw_forces(xd, n, box, rcs, nbr, cnt, cap, N.nefe_sw_params_silicon(), N.NEFE_FP32, f, e, ev)
    torch.cuda.synchronize()
    return f.cpu().numpy().reshape(3, n).T, e.cpu().numpy(), ev.cpu().numpy()


def _close32(x, box, got):
    """The FP32 tolerance of the parity tests: 1e-5 of the largest force, energy and virial scale."""
    e_o, f_o, vir_o, ea_o = O.sw_energy(x, box)
    f, e, ev = got
    assert np.abs(f - f_o).max() <= 1e-5 * np.abs(f_o).max()
    assert np.abs(e - ea_o).max() <= 1e-5 * np.abs(ea_o).max()
    assert abs(ev[0] - e_o) <= 1e-5 * abs(e_o)
    assert np.abs(ev[1:] - vir_o).max() <= 1e-4 * np.abs(vir_o).max()


@pytest.mark.parametrize("cap,shift", [(48, 0), (48, 1), (47, 0), (64, 0)])
@pytest.mark.parametrize("n", [31, 33, 129, 1000])
def test_scatter_forces_at_ragged_sizes(N, n, cap, shift):
    """Ragged warps and tiles, rows that cannot be read 16 bytes at a time, rows above 32 entries
    (skin 1.4 A), coordinates many boxes away."""
    x, box = I.liquid(max(n, 700), 0.05, seed=100 + n)
    x = x[:n] + np.array([7.0 * box[0], -123.0, 0.0])
    _close32(x, box, _forces32(N, x, box, 1.4 if cap == 64 else 0.5, cap, shift))


def test_scatter_forces_with_more_edges_than_a_list(N):
    """28 neighbours inside the cutoff: a warp's edges take several batches (896 of 224)."""
    x, box = I.diamond(5, 5, 5, a=4.4)
    x = I.rattle(x, 0.05, 7)
    _close32(x, box, _forces32(N, x, box, 0.3, 64))


@pytest.mark.parametrize("r", [1.2, 0.8])
def test_scatter_forces_of_close_pairs(N, r):
    """Terms far above what the first accumulator holds (some 1e2 to 1e4 eV/A) are split and lose
    nothing: relative to the largest force as any other."""
    x, box = I.diamond(3, 3, 3)
    x = I.rattle(x, 0.1, 8)
    d = x[1] - x[0]
    d -= box * np.rint(d / box)
    x[1] = x[0] + d * (r / np.linalg.norm(d))
    _close32(x, box, _forces32(N, x, box, 0.5, 48))


def test_chosen_scatter_form_refuses_what_it_always_refused(N):
    """A context whose form was set by hand flags terms of 48 eV/A or more; the default takes them."""
    x, box = I.diamond(3, 3, 3)
    d = x[4] - x[0]
    x[4] = x[0] + d * (1.3 / np.linalg.norm(d))
    got = {}
    for chosen in (False, True):
        ctx = N.Context(precision=N.NEFE_FP32, skin=0.5, nbr_cap=48)
        s = ctx.add_system(x, box, v=np.zeros_like(x))
        if chosen:
            ctx.set_tuning(0)
        ctx.run(1)
        got[chosen] = ctx.results(s)["error"]
        ctx.close()
    assert got == {False: 0, True: 4}


@pytest.mark.parametrize("shape", [(2, 2, 2), (10, 10, 10), (16, 16, 16)])
def test_scatter_form_atoms_per_warp(N, shape):
    """Context sizes that take 8, 16 and 32 atoms to a warp, with different potentials in one context
    (constants from the table) and with one (constants as arguments): energy of the state read back
    against the FP64 kernel's, 1e-5 relative."""
    x0, box = I.diamond(*shape)
    n = len(x0)
    reps = 5 if shape == (10, 10, 10) else 1
    for scale in (1.0, 0.97):
        ctx = N.Context(precision=N.NEFE_FP32, skin=0.5, nbr_cap=48)
        for r in range(reps + 1):
            s = ctx.add_system(x0, box, v=I.gaussian_velocities(n, 5.0, 40 + r))
            ctx.set_thermostat(s, 900.0, 0.1, 50 + r)
        p = N.nefe_sw_params_silicon()
        p.lambda3 *= scale
        ctx.set_sw_params(0, p)
        ctx.run(40)
        for s in (0, reps):
            x, _, b = ctx.get_state(s)
            xd = soa(x)
            nbr = torch.zeros(n * 48, dtype=torch.int32, device="cuda")
            cnt = torch.zeros(n, dtype=torch.int32, device="cuda")
            N.nefe_neighbor_build(xd, n, b, RC + 0.5, 48, nbr, cnt)
            f, ev = torch.zeros(3 * n, dtype=torch.float64, device="cuda"), torch.zeros(7, dtype=torch.float64, device="cuda")
            N.nefe_sw_forces(xd, n, b, RC + 0.5, nbr, cnt, 48, p if s == 0 else N.nefe_sw_params_silicon(), N.NEFE_FP64, f,
                             None, ev)
            r = ctx.results(s)
            assert r["error"] == 0
            assert r["U"] == pytest.approx(float(ev[0]), rel=1e-5)
        ctx.close()


# ------------------------------------------------------------------ FP64 edge lists
@pytest.mark.parametrize("cap,shift", [(48, 0), (48, 1), (47, 0)])
@pytest.mark.parametrize("n", [31, 65, 130, 2433])
def test_fp64_forces_at_ragged_sizes(N, n, cap, shift):
    """Ragged warps and tiles of 4 and 8 atoms to a warp, rows that cannot be read 16 bytes at a time:
    forces, energies per atom, virial and dE/dtheta's energy to the FP64 tolerance (1e-10)."""
    x, box = I.liquid(max(n, 700), 0.05, seed=200 + n)
    x = x[:n]
    rcs = RC + 0.5
    xd = soa(x)
    nbr = torch.full((n * cap + shift,), -1, dtype=torch.int32, device="cuda")[shift:]
    cnt = torch.zeros(n, dtype=torch.int32, device="cuda")
    N.nefe_neighbor_build(xd, n, box, rcs, cap, nbr, cnt)
    f, f2 = (torch.zeros(3 * n, dtype=torch.float64, device="cuda") for _ in range(2))
    e = torch.zeros(n, dtype=torch.float64, device="cuda")
    ev, eg = torch.zeros(7, dtype=torch.float64, device="cuda"), torch.zeros(8, dtype=torch.float64, device="cuda")
    prm = N.nefe_sw_params_silicon()
    N.nefe_sw_forces(xd, n, box, rcs, nbr, cnt, cap, prm, N.NEFE_FP64, f, e, ev)
    N.nefe_sw_energy_grad(xd, n, box, rcs, nbr, cnt, cap, prm, N.NEFE_FP64, f2, eg)
    torch.cuda.synchronize()
    e_o, f_o, vir_o, ea_o = O.sw_energy(x, box)
    scale = np.abs(f_o).max()
    assert np.abs(f.cpu().numpy().reshape(3, n).T - f_o).max() <= 1e-10 * scale
    assert np.array_equal(f.cpu().numpy(), f2.cpu().numpy())
    assert np.abs(e.cpu().numpy() - ea_o).max() <= 1e-10 * np.abs(ea_o).max()
    assert abs(float(ev[0]) - e_o) <= 1e-10 * abs(e_o) and abs(float(eg[0]) - e_o) <= 1e-10 * abs(e_o)
    assert np.abs(ev.cpu().numpy()[1:] - vir_o).max() <= 1e-9 * np.abs(vir_o).max()


@pytest.mark.parametrize("lanes", [8, 16, 32])
def test_fp64_forces_with_more_edges_than_a_list(N, lanes):
    """28 neighbours inside the cutoff, 16 atoms to a warp (448 edges of 192), through the engine:
    its energy and one step's motion against the oracle."""
    x, box = I.diamond(4, 4, 4, a=4.4)
    x = I.rattle(x, 0.02, 9)
    ctx = N.Context(precision=N.NEFE_FP64, skin=0.3, nbr_cap=64)
    s = ctx.add_system(x, box, v=np.zeros_like(x))
    ctx.set_tuning(lanes)
    ctx.run(3)
    got, v, _ = ctx.get_state(s)
    r = ctx.results(s)
    ctx.close()
    orc = O.System(x=x.copy(), v=np.zeros_like(x), box=box.copy())
    orc.run(3)
    assert r["error"] == 0
    assert r["U"] == pytest.approx(orc.results()["U"], rel=1e-10)
    assert np.abs(got - orc.x).max() < 1e-10 and np.abs(v - orc.v).max() <= 1e-9 * np.abs(orc.v).max()


def test_block_sums_of_large_values(N):
    """Per-atom values beyond the integer sums' range (a pair at 0.05 A: some 1e7 eV) take the FP64
    sums: energy and virial still match the oracle."""
    x, box = I.diamond(3, 3, 3)
    d = x[4] - x[0]
    x[4] = x[0] + d * (0.05 / np.linalg.norm(d))
    n = len(x)
    xd = soa(x)
    nbr = torch.zeros(n * 48, dtype=torch.int32, device="cuda")
    cnt = torch.zeros(n, dtype=torch.int32, device="cuda")
    N.nefe_neighbor_build(xd, n, box, RC + 0.5, 48, nbr, cnt)
    f, ev = torch.zeros(3 * n, dtype=torch.float64, device="cuda"), torch.zeros(7, dtype=torch.float64, device="cuda")
    N.nefe_sw_forces(xd, n, box, RC + 0.5, nbr, cnt, 48, N.nefe_sw_params_silicon(), N.NEFE_FP64, f, None, ev)
    torch.cuda.synchronize()
    e_o, f_o, vir_o, _ = O.sw_energy(x, box)
    assert np.abs(vir_o).max() > 2 * 2 ** 22       # each end of the pair is above 2^22
    assert abs(float(ev[0]) - e_o) <= 1e-10 * abs(e_o)
    assert np.abs(ev.cpu().numpy()[1:] - vir_o).max() <= 1e-9 * np.abs(vir_o).max()


# ------------------------------------------------------------------ Uhlenbeck-Ford rows and pair sums
# Rows and sums by several lanes per atom: part-filled tiles, rows shorter than the lanes, runs of
# cells that wrap at either edge of the smallest grid (5 cells, all of an axis in one run) and of a
# wider one.  Energies and forces normwise within 1e-10 (FP64) and 1e-5 (FP32) of the oracle, as for
# the other force kernels; pairs a bit closer than sigma to a few sigma apart.
@pytest.mark.parametrize("precision,tol", [(1, 1e-10), (0, 1e-5)])
@pytest.mark.parametrize("n,cells", [(2, (5, 5, 5)), (17, (5, 5, 5)), (129, (5, 6, 5)), (700, (5, 5, 9)), (1299, (7, 5, 6))])
def test_uf_rows_and_sums_by_lanes(N, n, cells, precision, tol):
    uf = (25.0, 2.0, 2200.0, 8.0)
    skin = 0.5
    rcs = O.SW_SI[6] * O.SW_SI[1] + skin
    box = np.array(cells) * rcs * 1.001
    rng = np.random.default_rng(100 + n)
    x = rng.uniform(0.0, box, (n, 3))
    for _ in range(40):                          # away from contacts: resample what is closer than 1 A
        d = x[:, None] - x[None]
        d -= box * np.round(d / box)
        r2 = (d * d).sum(2) + 1e9 * np.eye(n)
        bad = np.unique(np.argwhere(r2 < 1.0)[:, 0])
        if not len(bad):
            break
        x[bad] = rng.uniform(0.0, box, (len(bad), 3))
    if n == 2:
        x = np.array([[0.2, 0.3, 0.1], box - 0.9])                       # a pair across three faces
    x = x + box * rng.integers(-3, 4, (n, 3))
    e_o, f_o, vir_o, ea_o = O.uf_energy(x, box, uf)
    f = torch.zeros(3 * n, dtype=torch.float64, device="cuda")
    ea = torch.zeros(n, dtype=torch.float64, device="cuda")
    ev = torch.zeros(7, dtype=torch.float64, device="cuda")
    N.nefe_uf_forces(soa(x), n, box, rcs, skin, N.uf_params(*uf), precision, f, ea, ev)
    f = f.cpu().numpy().reshape(3, n).T
    assert np.abs(f - f_o).max() <= tol * np.abs(f_o).max()
    assert np.abs(ea.cpu().numpy() - ea_o).max() <= tol * np.abs(ea_o).max()
    assert abs(float(ev[0]) - e_o) <= tol * np.abs(ea_o).sum()
    assert np.abs(ev[1:].cpu().numpy() - vir_o).max() <= 10 * tol * np.abs(vir_o).max()


# ------------------------------------------------------------------ noise drawn ahead, finer blocks at the end
@pytest.mark.parametrize("baro", [False, True])
@pytest.mark.parametrize("shapes", [((2, 2, 2), (3, 3, 3)), ((2, 2, 2), (12, 12, 11)), ((14, 14, 13),)])
def test_noise_drawn_by_the_previous_step(N, shapes, baro):
    """FP64 contexts below and above the size where pass A draws the next step's noise (152 tiles), of
    part-filled tiles, with a system without a thermostat and with a box that moves: 23 steps in one
    call, in calls of 1 to 7 steps (whose first step draws its own) and captured, bit for bit."""
    got = []
    for parts in ((23,), (1, 1, 5, 7, 2, 7), (16, 7)):
        ctx = N.Context(precision=N.NEFE_FP64, skin=0.6, nbr_cap=48)
        for r, shape in enumerate(shapes):
            x, box = I.diamond(*shape)
            s = ctx.add_system(x, box, v=I.gaussian_velocities(len(x), 4.0, 70 + r))
            ctx.set_thermostat(s, 800.0, 0.1, 80 + r)
            if baro:
                ctx.set_barostat(s, N.NEFE_BARO_ISO, 0.0, 0.5)
        x, box = I.diamond(2, 2, 2)
        ctx.add_system(x, box, v=I.gaussian_velocities(len(x), 4.0, 79))
        for k in parts:
            ctx.run(k)
        got.append([ctx.get_state(s) for s in range(len(shapes) + 1)])
        assert all(ctx.results(s)["error"] == 0 for s in range(len(shapes) + 1))
        ctx.close()
    for other in got[1:]:
        for a, b in zip(got[0], other):
            assert all(np.array_equal(u, v) for u, v in zip(a, b))


@pytest.mark.parametrize("precision,tol,copies", [(1, 1e-10, (2, 1, 1)), (1, 1e-10, (3, 2, 2)), (0, 1e-5, (5, 2, 4)),
                                                  (0, 1e-5, (4, 4, 3))])
def test_forces_where_the_last_blocks_are_cut_finer(N, precision, tol, copies):
    """Sizes below and above the ones from which the last tiles are cut finer: a rattled crystal repeated
    in space has the forces, energies and virial of one copy (the FP64 ones of 4096 atoms), normwise."""
    x1, box1 = I.diamond(8, 8, 8)
    x1 = I.rattle(x1, 0.1, 4)
    _, f1, v1, e1 = O.sw_energy(x1, box1)
    m = int(np.prod(copies))
    shift = np.stack(np.meshgrid(*[np.arange(c) for c in copies], indexing="ij"), -1).reshape(-1, 1, 3) * box1
    x, box, n = (x1[None] + shift).reshape(-1, 3), box1 * np.array(copies), m * len(x1)
    xd = soa(x)
    nbr = torch.zeros(n * 48, dtype=torch.int32, device="cuda")
    cnt = torch.zeros(n, dtype=torch.int32, device="cuda")
    N.nefe_neighbor_build(xd, n, box, RC + 0.5, 48, nbr, cnt)
    f, e = torch.zeros(3 * n, dtype=torch.float64, device="cuda"), torch.zeros(n, dtype=torch.float64, device="cuda")
    ev = torch.zeros(7, dtype=torch.float64, device="cuda")
    N.nefe_sw_forces(xd, n, box, RC + 0.5, nbr, cnt, 48, N.nefe_sw_params_silicon(), precision, f, e, ev)
    torch.cuda.synchronize()
    f, e, ev = f.cpu().numpy().reshape(3, n).T.reshape(m, -1, 3), e.cpu().numpy().reshape(m, -1), ev.cpu().numpy()
    assert np.abs(f - f1).max() <= tol * np.abs(f1).max()
    assert np.abs(e - e1).max() <= tol * np.abs(e1).max()
    assert abs(ev[0] / m - e1.sum()) <= tol * np.abs(e1).sum()
    assert np.abs(ev[1:] / m - v1).max() <= 10 * tol * np.abs(v1).max()


# ------------------------------------------------------------------ rebuild by clusters
@pytest.mark.parametrize("policy", [0, 1])
@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("shapes", [((2, 2, 2), (5, 5, 4)), ((16, 16, 7), (3, 3, 3)), ((16, 16, 10), (3, 3, 3))])
def test_rebuild_by_clusters_and_by_worklist(N, shapes, precision, policy):
    """The same systems in a context of at most 32 (cells by a cluster per system, up to 128 tiles in all) and of 35
    (worklist): hot enough that lists are rebuilt every few steps, the same motion bit for bit.  (The FP64
    passes' lanes are set: their sums' order, and so the last bits, go by the context's size otherwise.)"""
    got = []
    for extra in (0, 33):
        ctx = N.Context(precision=precision, skin=0.3, nbr_cap=48)
        for r, shape in enumerate(shapes):
            x, box = I.diamond(*shape)
            s = ctx.add_system(x, box, v=I.gaussian_velocities(len(x), 6.0, 90 + r))
            ctx.set_thermostat(s, 1500.0, 0.1, 30 + r)
        x, box = I.diamond(2, 2, 2)
        for r in range(extra):
            ctx.add_system(x, box, v=I.gaussian_velocities(len(x), 3.0, r))
        if precision == 1:
            ctx.set_tuning(8, 4)
        ctx.set_rebuild_policy(policy)
        ctx.run(60)
        got.append([ctx.get_state(s) for s in range(len(shapes))])
        assert all(ctx.results(s)["error"] == 0 for s in range(len(shapes)))
        ctx.close()
    for a, b in zip(*got):
        assert all(np.array_equal(u, v) for u, v in zip(a, b))


# ------------------------------------------------------------------ sums of a stateless FP64 call
@pytest.mark.parametrize("seed", [1, 2, 3])
def test_fp64_sums_keep_their_remainders(N, seed):
    """Energy, virial and dE/d(A) of 64 atoms in blocks of 8: block sums in 2^-40 eV units, so some 500
    conversions of at most 2^-41 eV each (1e-11 eV, 4e-14 of the energy), where one rounding to 2^-32 eV per
    block is 1e-10 eV and more."""
    x, box = I.diamond(2, 2, 2)
    x = I.rattle(x, 0.1, seed)
    n, cap = len(x), 48
    xd = soa(x)
    nbr, cnt = torch.zeros(n * cap, dtype=torch.int32, device="cuda"), torch.zeros(n, dtype=torch.int32, device="cuda")
    N.nefe_neighbor_build(xd, n, box, RC + 0.5, cap, nbr, cnt)
    f = torch.zeros(3 * n, dtype=torch.float64, device="cuda")
    ev, eg = torch.zeros(7, dtype=torch.float64, device="cuda"), torch.zeros(8, dtype=torch.float64, device="cuda")
    N.nefe_sw_forces(xd, n, box, RC + 0.5, nbr, cnt, cap, N.nefe_sw_params_silicon(), N.NEFE_FP64, f, None, ev)
    N.nefe_sw_energy_grad(xd, n, box, RC + 0.5, nbr, cnt, cap, N.nefe_sw_params_silicon(), N.NEFE_FP64, f, eg)
    torch.cuda.synchronize()
    e_o, _, vir_o, _ = O.sw_energy(x, box)
    assert abs(float(ev[0]) - e_o) <= 1e-13 * abs(e_o)
    assert abs(float(eg[0]) - e_o) <= 1e-13 * abs(e_o)
    assert np.abs(ev.cpu().numpy()[1:] - vir_o).max() <= 1e-13 * abs(e_o)


# ------------------------------------------------------------------ large sums
def _sw(N, x, box, prm, precision, skin=0.5, cap=48, grad=False):
    """Forces, energy and virial (or energy and dE/dtheta) of a stateless call, as numpy."""
    n, rcs = len(x), RC + skin
    xd = soa(x)
    nbr, cnt = torch.zeros(n * cap, dtype=torch.int32, device="cuda"), torch.zeros(n, dtype=torch.int32, device="cuda")
    N.nefe_neighbor_build(xd, n, box, rcs, cap, nbr, cnt)
    f = torch.zeros(3 * n, dtype=torch.float64, device="cuda")
    out = torch.zeros(8 if grad else 7, dtype=torch.float64, device="cuda")
    if grad:
        N.nefe_sw_energy_grad(xd, n, box, rcs, nbr, cnt, cap, prm, precision, f, out)
    else:
        N.nefe_sw_forces(xd, n, box, rcs, nbr, cnt, cap, prm, precision, f, None, out)
    torch.cuda.synchronize()
    return f.cpu().numpy().reshape(3, n).T, out.cpu().numpy()


def _silicon(N, **scale):
    p = N.nefe_sw_params_silicon()
    for k, v in scale.items():
        setattr(p, k, getattr(p, k) * v)
    return p


@pytest.mark.parametrize("power", [12, 16, 17, 18, 19, 20, 21])
def test_block_sums_whose_terms_are_in_range_but_not_their_total(N, power):
    """eps times 2^power: the sums are those of silicon times the same number.  A block (8 atoms, some 35 eV)
    crosses 2^22 eV at 2^17 and 2^23 at 2^18, a lane's term (some 2 eV) crosses 2^22 at 2^21 only.  Each of the
    500 conversions is within 2^-33 eV of its term, and the reference's (2^-40 units) within 2^power 2^-41."""
    x, box = I.diamond(2, 2, 2)
    x = I.rattle(x, 0.1, 21)
    k = 2.0 ** power
    _, ev1 = _sw(N, x, box, _silicon(N), N.NEFE_FP64)
    _, eg1 = _sw(N, x, box, _silicon(N), N.NEFE_FP64, grad=True)
    _, ev = _sw(N, x, box, _silicon(N, eps=k), N.NEFE_FP64)
    _, eg = _sw(N, x, box, _silicon(N, eps=k), N.NEFE_FP64, grad=True)
    tol = 1e-12 * abs(ev1[0])
    assert np.abs(ev / k - ev1).max() <= tol
    assert np.abs(eg / k - eg1).max() <= 1e-12 * np.abs(eg1).max()


def test_spring_energies_of_sites_in_other_images(N):
    """Springs take no nearest image: sites 20 boxes away hold 3.5e5 eV an atom, 1.1e7 eV in the 32 atoms of a
    block, in FP64 against the plain sum."""
    x, box = I.diamond(2, 2, 2)
    r0 = x + np.array([20.0, 20.0, 20.0]) * box
    ctx = N.Context(precision=N.NEFE_FP64, skin=0.5, nbr_cap=48)
    s = ctx.add_system(x, box, v=np.zeros_like(x), r0=r0)
    ctx.set_schedule(s, N.NEFE_SCHED_FL, 1, 1000, k_E=5.0)
    ctx.setup()
    r = ctx.results(s)
    ctx.close()
    assert r["error"] == 0
    assert r["U_E"] == pytest.approx(0.5 * 5.0 * float(((x - r0) ** 2).sum()), rel=1e-12)


@pytest.mark.parametrize("precision", [0, 1])
def test_coincident_atoms_give_nan_and_only_there(N, precision):
    """Two atoms at one place: NaN forces on them, energy and virial NaN (no finite sum stands for them),
    every atom further away than two cutoffs as without them."""
    x, box = I.diamond(4, 4, 4)
    x = I.rattle(x, 0.05, 5)
    x[9] = x[8]
    f, ev = _sw(N, x, box, _silicon(N), precision)
    assert np.isnan(f[8]).any() and np.isnan(f[9]).any()
    assert np.isnan(ev).any()
    d = x - x[8]
    d -= box * np.rint(d / box)
    far = np.flatnonzero((d * d).sum(1) > (2.0 * RC) ** 2)
    f_o = O.sw_force_atoms(x, box, far)
    assert len(far) > 100 and np.abs(f[far] - f_o).max() <= 1e-5 * np.abs(f_o).max()


@pytest.mark.parametrize("r", [0.06, 0.03, 0.012])
def test_scatter_forces_of_very_close_pairs(N, r):
    """Forces of some 5e8 to 1e12 eV/A: finite, relative to the largest as any other."""
    x, box = I.diamond(3, 3, 3)
    d = x[4] - x[0]
    x[4] = x[0] + d * (r / np.linalg.norm(d))
    f, _ = _sw(N, x, box, _silicon(N), N.NEFE_FP32)
    _, f_o, _, _ = O.sw_energy(x, box)
    # the pair's distance carries 2 units of 16 A 2^-32 (7.6e-9 A) and 2^-23 of itself; the force goes as r^-5
    assert np.abs(f - f_o).max() <= (1e-5 + 5 * 7.6e-9 / r) * np.abs(f_o).max()


def test_fp32_sums_out_of_range_for_a_block_but_not_for_its_warps(N):
    """39,304 atoms of some 690 eV each (eps times 160): 64 atoms of a block exceed the 32,768 eV that an FP32 block
    sum holds, the 32 of a warp do not (nor does dE/da, some 1500 eV an atom, the 65,536 of its own).  Energy against FP64,
    1e-5."""
    x, box = I.diamond(17, 17, 17)
    x = I.rattle(x, 0.05, 3)
    p = _silicon(N, eps=160.0)
    _, ev = _sw(N, x, box, p, N.NEFE_FP32)
    _, ev64 = _sw(N, x, box, p, N.NEFE_FP64)
    assert abs(ev[0] - ev64[0]) <= 1e-5 * abs(ev64[0])
    _, eg = _sw(N, x, box, p, N.NEFE_FP32, grad=True)
    assert abs(eg[0] - ev64[0]) <= 1e-5 * abs(ev64[0])


@pytest.mark.parametrize("scale", [1e-8, 1e-4, 1e-2, 0.5, 2.0, 100.0])
def test_scatter_forces_of_weak_and_strong_potentials(N, scale):
    """The FP32 tolerance is relative (1e-5 of the largest force) whatever the unit of energy, in a stateless call
    and in a context (velocity after one step from rest, FP64 against FP32)."""
    x, box = I.diamond(3, 3, 3)
    x = I.rattle(x, 0.1, 8)
    f, _ = _sw(N, x, box, _silicon(N, eps=scale), N.NEFE_FP32)
    _, f_o, _, _ = O.sw_energy(x, box)
    assert np.abs(f / scale - f_o).max() <= 1e-5 * np.abs(f_o).max()
    v = []
    for precision in (N.NEFE_FP32, N.NEFE_FP64):
        ctx = N.Context(precision=precision, skin=0.5, nbr_cap=48)
        for k in (scale, 1.0):                           # two potentials in one context
            s = ctx.add_system(x, box, v=np.zeros_like(x), mass=28.0855 * k)
            ctx.set_sw_params(s, _silicon(N, eps=k))
        ctx.run(1)
        assert all(ctx.results(s)["error"] == 0 for s in range(2))
        v.append([ctx.get_state(s)[1] for s in range(2)])
        ctx.close()
    for a, b in zip(*v):
        assert np.abs(a - b).max() <= 1e-5 * np.abs(b).max()


# ------------------------------------------------------------------ long boxes
@pytest.mark.parametrize("L", [1000.0, 2000.0, 2.0e4, 2.0e5])
def test_fp32_forces_in_long_boxes(N, L):
    """A slab in a box of up to 2e5 A: the FP32 tolerance of a short box, stateless and in a context (velocity after
    one step from rest), and for the Uhlenbeck-Ford term."""
    x, box = I.diamond(3, 2, 2)
    x = I.rattle(x, 0.1, 11) + np.array([0.61803 * L, 0.0, 0.0])
    box = np.array([L, box[1], box[2]])
    _close32(x, box, _forces32(N, x, box, 0.5, 48))
    v = []
    for precision in (N.NEFE_FP32, N.NEFE_FP64):
        ctx = N.Context(precision=precision, skin=0.5, nbr_cap=48)
        s = ctx.add_system(x, box, v=np.zeros_like(x))
        ctx.run(1)
        assert ctx.results(s)["error"] == 0
        v.append(ctx.get_state(s)[1])
        ctx.close()
    assert np.abs(v[0] - v[1]).max() <= 1e-5 * np.abs(v[1]).max()


@pytest.mark.parametrize("L", [1000.0, 2.0e4, 2.0e5])
def test_fp32_uf_forces_in_long_boxes(N, L):
    """1e-6 of the largest force: ten times the rounding of an FP32 distance."""
    uf, skin = (25.0, 2.0, 2200.0, 8.0), 0.5
    x, box = I.diamond(2, 4, 4)
    x = I.rattle(x, 0.1, 12) + np.array([0.61803 * L, 0.0, 0.0])
    box = np.array([L, 22.0, 22.0])
    n = len(x)
    e_o, f_o, vir_o, ea_o = O.uf_energy(x, box, uf)
    f = torch.zeros(3 * n, dtype=torch.float64, device="cuda")
    ea = torch.zeros(n, dtype=torch.float64, device="cuda")
    N.nefe_uf_forces(soa(x), n, box, RC + skin, skin, N.uf_params(*uf), N.NEFE_FP32, f, ea, None)
    f = f.cpu().numpy().reshape(3, n).T
    assert np.abs(f - f_o).max() <= 1e-6 * np.abs(f_o).max()


# ------------------------------------------------------------------ sums of the FP64 engine
@pytest.mark.parametrize("seed", [1, 2, 3, 4])
def test_fp64_engine_sums_keep_their_remainders(N, seed):
    """Energy and pressure of 64 atoms in blocks of 8, as test_fp64_sums_keep_their_remainders: 1e-13 of the
    energy (at rest the pressure is the virial's alone)."""
    x, box = I.diamond(2, 2, 2)
    x = I.rattle(x, 0.1, seed)
    ctx = N.Context(precision=N.NEFE_FP64, skin=0.5, nbr_cap=48)
    s = ctx.add_system(x, box, v=np.zeros_like(x))
    ctx.setup()
    r = ctx.results(s)
    ctx.close()
    e_o, _, vir_o, _ = O.sw_energy(x, box)
    V = float(np.prod(box))
    assert abs(r["U"] - e_o) <= 1e-13 * abs(e_o)
    assert np.abs(r["P"] * V / O.EV_A3_TO_GPA - vir_o).max() <= 2e-13 * abs(e_o)


# ------------------------------------------------------------------ shells of 32
def _ball(r_out):
    """An atom, 32 neighbours spread over a sphere inside the cutoff, one more at r_out."""
    k = np.arange(33) + 0.5
    z, t = 1.0 - 2.0 * k / 33, math.pi * (1.0 + 5.0 ** 0.5) * k
    u = np.stack([np.sqrt(1.0 - z * z) * np.cos(t), np.sqrt(1.0 - z * z) * np.sin(t), z], 1)
    r = np.full((33, 1), 3.55)
    r[16] = r_out
    return np.concatenate([[[0.0, 0.0, 0.0]], u * r])


def test_fp64_shell_of_32_with_one_more_just_outside(N):
    """The row filter's margin (1.4e-3 A in a box of 500 A) is not the cutoff: 32 neighbours and one 1e-4 A outside are
    a shell of 32, in the sums, the forces and the shell statistics."""
    box = np.array([500.0, 500.0, 500.0])
    x = _ball(RC + 1e-4) + 250.0
    f, ev = _sw(N, x, box, _silicon(N), N.NEFE_FP64, cap=64)
    e_o, f_o, vir_o, _ = O.sw_energy(x, box)
    assert np.abs(f - f_o).max() <= 1e-10 * np.abs(f_o).max()
    assert abs(ev[0] - e_o) <= 1e-10 * abs(e_o)
    ctx = N.Context(precision=N.NEFE_FP64, skin=0.5, nbr_cap=64)
    s = ctx.add_system(x, box, v=np.zeros_like(x))
    ctx.setup()
    r, st = ctx.results(s), ctx.shell_stats()
    ctx.close()
    assert r["error"] == 0 and r["U"] == pytest.approx(e_o, rel=1e-10)
    d = x[:, None] - x[None]
    m = ((d * d).sum(2) < RC * RC).sum(1) - 1
    assert m.max() == 32 and st == (m.mean(), 32)


def test_fp64_shell_of_33_is_refused(N):
    box = np.array([500.0, 500.0, 500.0])
    with pytest.raises(N.NefeError):
        _sw(N, _ball(RC - 1e-4) + 250.0, box, _silicon(N), N.NEFE_FP64, cap=64)


# ------------------------------------------------------------------ autotuner
def test_autotune_does_not_narrow_what_a_context_takes(N):
    """A pair at 1.3 A (terms above 48 eV/A) in an autotuned context, as in one left alone: no error, neither from the
    trial launches nor from the steps."""
    x, box = I.diamond(3, 3, 3)
    d = x[4] - x[0]
    x[4] = x[0] + d * (1.3 / np.linalg.norm(d))
    ctx = N.Context(precision=N.NEFE_FP32, skin=0.5, nbr_cap=48)
    s = ctx.add_system(x, box, v=np.zeros_like(x))
    ctx.autotune()
    assert ctx.results(s)["error"] == 0
    ctx.run(1)
    assert ctx.results(s)["error"] == 0
    ctx.close()


def test_autotune_of_shells_above_the_thread_form(N):
    """28 neighbours inside the cutoff: more than the one-thread form's 20, which flags its trial; the context takes
    another form and stays without error."""
    x, box = I.diamond(4, 4, 4, a=4.4)
    x = I.rattle(x, 0.02, 9)
    ctx = N.Context(precision=N.NEFE_FP32, skin=0.3, nbr_cap=64)
    s = ctx.add_system(x, box, v=np.zeros_like(x))
    lanes, _ = ctx.autotune()
    ctx.run(1)
    assert lanes != 1 and ctx.results(s)["error"] == 0
    ctx.close()


@pytest.mark.parametrize("kind,error", [("beta_tin", 0), ("diamond", 4)])
def test_autotuned_scatter_form_refuses_where_it_always_did(N, kind, error):
    """256,000 atoms, one of 32 systems with a pair at 1.3 A, in contexts whose fastest form is the scatter form: beta-tin
    (18 neighbours, once faster in the gather form, which takes any term) is not refused, diamond is, as before."""
    x, box = I.beta_tin(10, 10, 20) if kind == "beta_tin" else I.diamond(10, 10, 10)
    x = I.rattle(x, 0.02, 4)
    ctx = N.Context(precision=N.NEFE_FP32, skin=0.5, nbr_cap=48)
    for r in range(32):
        y = x.copy()
        if r == 3:
            d = y[1:] - y[0]
            d -= box * np.rint(d / box)
            k = np.argmin((d * d).sum(1))
            y[k + 1] = y[0] + d[k] * (1.3 / np.linalg.norm(d[k]))
        ctx.add_system(y, box, v=np.zeros_like(y))
    lanes, _ = ctx.autotune()
    assert all(r["error"] == 0 for r in ctx.results_all())
    ctx.run(1)
    assert lanes == 0
    assert [r["error"] for r in ctx.results_all()] == [error if r == 3 else 0 for r in range(32)]
    ctx.close()


# ------------------------------------------------------------------ scratch kept between calls
def test_scratch_is_given_back(N):
    """The stateless calls keep up to 256 MB mapped; nefe_release_scratch returns them (a call of 110,592 atoms in FP64
    wants some 150 MB, of which the list's and the force call's share is kept), twice in a row as well, and the
    next call finds its scratch again."""
    x, box = I.diamond(24, 24, 24)
    x = I.rattle(x, 0.05, 2)
    first = _sw(N, x, box, _silicon(N), N.NEFE_FP64)
    torch.cuda.empty_cache()
    kept = torch.cuda.mem_get_info()[0]
    N.nefe_release_scratch()
    assert torch.cuda.mem_get_info()[0] - kept >= 64 << 20
    N.nefe_release_scratch()
    again = _sw(N, x, box, _silicon(N), N.NEFE_FP64)
    assert np.array_equal(first[0], again[0]) and np.array_equal(first[1], again[1])
