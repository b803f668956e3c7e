"""Instances of the X-Y sweeps that ordinary solves are dispatched to, against the FP64 oracle:
the ring sweep (csrc/sweep2d_ring.cuh) with 8 cells per lane in every mode that takes them, its
linear mode with the step scheme and with an inflow, rows of 5 to 8 warps, and the row kernel
(csrc/sweep2d_row.cuh) that serves rows whose rings do not fit."""
import numpy as np
import pytest

import rom_workloads as W
from oracle import oracle as O

pytestmark = pytest.mark.gpu

TOL = 1e-5  # relative l2 of the flux, the bound of every FP32 path
BOUNDS = (0.0, 1.3, -0.2, 0.7)


@pytest.fixture(scope="module")
def rom():
    import torch
    assert torch.cuda.is_available()
    import __graft_entry__
    __graft_entry__.build()
    from paper_2407_12527_gb300 import rom as R
    return R


def medium_of(I, J, medium):
    st, ss, q = W.random_medium(I, J, seed=I + J, ratio_max=0.7)
    if medium == "uniform":
        st = np.full((J, I), 2.1)
        ss = np.minimum(ss, 1.4)
    return st, ss, q


def compare(rom, I, J, medium, sets, scheme="dd", kernel="iso", lit=False, some=None, iters=2,
            tol=TOL, **opts):
    """Solves and compares the samples `some` (all) with the oracle; returns the statistics."""
    st, ss, q = medium_of(I, J, medium)
    inflow = W.random_inflow(I, J, seed=7, scale=1.5) if lit else None
    g = 0.0 if kernel == "iso" else 0.4
    ctx = rom.RomContext(0)
    ctx.set_grid(I, J, BOUNDS, st, ss, q)
    ctx.set_ordinates([(o.c, o.s, o.zeta, o.w) for o in sets])
    if kernel != "iso":
        ctx.set_kernel(kernel, g)
    if lit:
        off = [0, J, 2 * J, 2 * J + I, 2 * J + 2 * I]
        for f in range(4):
            ctx.set_inflow_isotropic(f, inflow[off[f]:off[f + 1]])
    ctx.set_options(scheme=rom.SCHEME[scheme], fixed_iters=iters, **opts)
    stats = ctx.solve()
    some = list(range(len(sets))) if some is None else some
    phi = [ctx.scalar_flux(k) for k in some]
    leak, bal, _ = ctx.balance()
    ctx.close()
    ref = O.solve_xy(I, J, BOUNDS, st, ss, q, [sets[k] for k in some], inflow=inflow, kernel=kernel,
                     g=g, scheme=scheme, fixed_iters=iters)
    area = 1.3 * 0.9 / (I * J)
    for n, k in enumerate(some):
        assert np.linalg.norm(phi[n] - ref["phi"][n]) < tol * np.linalg.norm(ref["phi"][n]), k
        if kernel != "hg":
            scale = abs(ref["leak"][n]) + np.sum(st * ref["phi"][n]) * area
            assert abs(leak[k] - ref["leak"][n]) < tol * scale, k
    if kernel != "hg":
        assert np.all(bal < tol)
    return stats


def quadrant_sets(n, m):
    """n drawn sets of m ordinates per quadrant: 4 n work items of m ordinates."""
    nz, nt = W.partition(m)
    return [O.rom_ordinates_xy(11, k, nz, nt) for k in range(n)]


# 640 items and more: above every least number of items that the choice of 8 cells per lane has
# on 152 SMs (608 where 256-cell warps round up by more than 128-cell ones or with an inflow), and
# 614400 item rows where it takes 4000 per SM (varying sigma_T, four ordinates, above 256 columns).
@pytest.mark.parametrize("scheme", ["dd", "step"])
@pytest.mark.parametrize("I,J,S,medium,tile_g,lit,kernel", [
    (200, 17, 160, "uniform", 2, False, "iso"),
    (256, 18, 160, "uniform", 4, False, "iso"),
    (450, 17, 160, "uniform", 2, False, "iso"),
    (512, 18, 160, "uniform", 4, False, "iso"),
    (300, 17, 160, "uniform", 2, False, "iso"),
    (200, 19, 160, "uniform", 2, True, "iso"),
    (450, 17, 160, "uniform", 2, True, "iso"),
    (200, 19, 160, "uniform", 4, True, "iso"),
    (450, 17, 160, "uniform", 4, True, "iso"),
    (200, 17, 160, "varying", 2, False, "iso"),
    (450, 17, 160, "varying", 2, False, "iso"),
    (200, 17, 160, "varying", 2, True, "iso"),
    (450, 17, 160, "varying", 2, True, "iso"),
    (200, 17, 160, "varying", 4, False, "iso"),
    (390, 150, 1024, "varying", 4, False, "iso"),
    (200, 17, 160, "uniform", 2, False, "linear"),
    (200, 17, 160, "uniform", 4, False, "linear"),
    (200, 17, 160, "uniform", 2, True, "linear"),
    (200, 17, 160, "uniform", 4, True, "linear")])
def test_eight_cells(rom, I, J, S, medium, tile_g, lit, kernel, scheme):
    stats = compare(rom, I, J, medium, quadrant_sets(S, tile_g), scheme, kernel, lit,
                    some=[0, S // 2, S - 1], tile_g=tile_g, rows_per_step=1)
    assert stats["rows_per_step"] == 1 and stats["tile_g"] == tile_g


@pytest.mark.parametrize("scheme", ["dd", "step"])
@pytest.mark.parametrize("I", [200, 450])
@pytest.mark.parametrize("medium", ["uniform", "varying"])
@pytest.mark.parametrize("precision", [0, 1])
def test_eight_cells_dense_inflow(rom, scheme, I, medium, precision):
    stats = compare(rom, I, 17, medium, quadrant_sets(80, 2), scheme, "hg", True, some=[0, 41, 79],
                    dense_precision=precision)
    assert stats["rows_per_step"] == 1


@pytest.mark.parametrize("scheme", ["dd", "step"])
@pytest.mark.parametrize("n_samples", [2, 90])
def test_eight_cells_batch_of_grids(rom, scheme, n_samples):
    """Two grids, two and one warps wide (720 items of two ordinates with 90 samples a grid)."""
    grids, sets = [], []
    for I, J in ((430, 19), (201, 23)):
        grids.append((I, J, BOUNDS) + medium_of(I, J, "varying"))
        sets += quadrant_sets(n_samples, 2)
    ctx = rom.RomContext(0)
    ctx.set_grids(grids, [n_samples] * 2)
    ctx.set_ordinates([(o.c, o.s, o.zeta, o.w) for o in sets])
    ctx.set_options(scheme=rom.SCHEME[scheme], fixed_iters=2, tile_g=2, rows_per_step=1)
    ctx.solve()
    for p, (I, J, b, st, ss, q) in enumerate(grids):
        for k in (0, n_samples - 1):
            ref = O.solve_xy(I, J, b, st, ss, q, [sets[p * n_samples + k]], scheme=scheme,
                             fixed_iters=2)["phi"][0]
            phi = ctx.scalar_flux(p * n_samples + k)
            assert np.linalg.norm(phi - ref) < TOL * np.linalg.norm(ref), (p, k)
    ctx.close()


@pytest.mark.parametrize("grid", [(1, 1), (5, 8), (33, 16), (130, 18), (255, 40)])
@pytest.mark.parametrize("medium", ["uniform", "varying"])
@pytest.mark.parametrize("scheme", ["dd", "step"])
@pytest.mark.parametrize("lit", [False, True])
@pytest.mark.parametrize("tile_g", [2, 4])
def test_linear_kernel(rom, grid, medium, scheme, lit, tile_g):
    sets = [O.Ordinates(*W.random_directions(M, seed=M, weights="random")) for M in (7, 18)]
    stats = compare(rom, *grid, medium, sets, scheme, "linear", lit, iters=3, tile_g=tile_g,
                    rows_per_step=1)
    assert stats["rows_per_step"] == 1


@pytest.mark.parametrize("I", [769, 1024, 1025, 1536, 1537, 2041, 2048])
@pytest.mark.parametrize("medium", ["uniform", "varying"])
@pytest.mark.parametrize("kernel", ["iso", "linear", "hg"])
@pytest.mark.parametrize("scheme,lit", [("dd", False), ("dd", True), ("step", True)])
@pytest.mark.parametrize("rows", [0, 1])
def test_wide_rows(rom, I, medium, kernel, scheme, lit, rows):
    """Rows of 4 to 8 warps, the library's own choice of kernel and the one-row one: the ring
    sweep up to 768 (linear, varying sigma_T), 1024 (linear, uniform; dense, varying), 1536
    columns (isotropic, varying; dense, uniform) or all 2048 (isotropic, uniform), the row kernel
    (rows = 1) or the 4-row one above.

    An edge is multiplied by the same FP32 constant in each of a row's cells, (a - b - sigma_T) /
    (sigma_T + a + b) or a / (sigma_T + a + b), near 1 where cells are thin and narrow (here 1.3 /
    I by 0.04): six roundings, so that its error grows by up to 6 x 2^-24 a cell."""
    sets = [O.Ordinates(*W.random_directions(M, seed=M, weights="random")) for M in (5, 14)]
    ring = I <= {("iso", "uniform"): 2048, ("iso", "varying"): 1536, ("linear", "uniform"): 1024,
                 ("linear", "varying"): 768, ("hg", "uniform"): 1536,
                 ("hg", "varying"): 1024}[kernel, medium]
    for tile_g in (0, 4) if rows == 1 and kernel != "hg" else (0,):
        stats = compare(rom, I, 21, medium, sets, scheme, kernel, lit, rows_per_step=rows,
                        tile_g=tile_g, tol=TOL + 6 * I * 2.0 ** -24)
        assert stats["rows_per_step"] == (1 if ring or rows == 1 else 4)


@pytest.mark.parametrize("I,kernel", [(1536, "iso"), (1537, "iso"), (768, "linear"), (769, "linear")])
@pytest.mark.parametrize("scheme", ["dd", "step"])
@pytest.mark.parametrize("rows", [0, 1])
def test_wide_batch_of_grids(rom, I, kernel, scheme, rows):
    """The widest grid of a batch on either side of where the rings fit (bounds as above)."""
    grids, sets = [], []
    for w, J in ((I, 21), (130, 30)):
        grids.append((w, J, BOUNDS) + medium_of(w, J, "varying"))
        sets += [O.Ordinates(*W.random_directions(9, seed=w, weights="random"))]
    g = 0.4 if kernel == "linear" else 0.0
    ctx = rom.RomContext(0)
    ctx.set_grids(grids, [1, 1])
    ctx.set_ordinates([(o.c, o.s, o.zeta, o.w) for o in sets])
    ctx.set_kernel(kernel, g)
    ctx.set_options(scheme=rom.SCHEME[scheme], fixed_iters=2, rows_per_step=rows)
    stats = ctx.solve()
    assert stats["rows_per_step"] == (1 if I in (1536, 768) or rows == 1 else 4)
    for p, (w, J, b, st, ss, q) in enumerate(grids):
        ref = O.solve_xy(w, J, b, st, ss, q, [sets[p]], kernel=kernel, g=g, scheme=scheme,
                         fixed_iters=2)["phi"][0]
        phi = ctx.scalar_flux(p)
        assert np.linalg.norm(phi - ref) < (TOL + 6 * w * 2.0 ** -24) * np.linalg.norm(ref), p
    ctx.close()
