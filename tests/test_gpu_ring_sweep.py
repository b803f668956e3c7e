"""The ring-staged one-row X-Y sweep (csrc/sweep2d_ring.cuh) at the edges of its tiling
(lanes of 4 or 8 cells, 8-lane copy groups, 16-row rings, warps of 32 lanes, groups of 8
steps) against the FP64 oracle."""
import numpy as np
import pytest

import rom_workloads as W
from oracle import oracle as O

pytestmark = pytest.mark.gpu

TOL = 1e-5  # relative l2 of the flux, the bound of every FP32 path


@pytest.fixture(scope="module")
def rom():
    import torch
    assert torch.cuda.is_available()
    import __graft_entry__
    __graft_entry__.build()
    from paper_2407_12527_gb300 import rom as R
    return R


def solve(rom, I, J, st, ss, q, sets, inflow=None, kernel="iso", g=0.0, **opts):
    ctx = rom.RomContext(0)
    ctx.set_grid(I, J, (0.0, 1.3, -0.2, 0.7), st, ss, q)
    ctx.set_ordinates([(o.c, o.s, o.zeta, o.w) for o in sets])
    if kernel != "iso":
        ctx.set_kernel(kernel, g)
    off = [0, J, 2 * J, 2 * J + I, 2 * J + 2 * I]
    if inflow is not None:
        for f in range(4):
            v = np.ascontiguousarray(inflow[..., off[f]:off[f + 1]])
            if inflow.ndim == 1:
                ctx.set_inflow_isotropic(f, v)
            else:
                ctx.set_inflow_ordinates(f, v)
    ctx.set_options(**opts)
    stats = ctx.solve()
    phi = np.stack([ctx.scalar_flux(k) for k in range(len(sets))])
    leak, bal, _ = ctx.balance()
    ctx.close()
    return phi, leak, bal, stats


def oracle(I, J, st, ss, q, sets, inflow=None, **kw):
    per = inflow is not None and inflow.ndim == 2
    r = O.solve_xy(I, J, (0.0, 1.3, -0.2, 0.7), st, ss, q, sets, inflow=inflow,
                   inflow_per_ordinate=per, **kw)
    return r["phi"], r["leak"]


def rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


@pytest.mark.parametrize("grid", [(1, 1), (3, 2), (4, 7), (5, 8), (31, 15), (33, 16), (127, 17),
                                  (128, 9), (129, 33), (130, 3), (255, 40), (260, 12)])
@pytest.mark.parametrize("medium", ["uniform", "varying"])
@pytest.mark.parametrize("scheme", ["dd", "step"])
@pytest.mark.parametrize("inflow", ["vacuum", "ordinates"])
def test_tile_edges(rom, grid, medium, scheme, inflow):
    I, J = grid
    st, ss, q = W.random_medium(I, J, seed=I + 100 * J)
    if medium == "uniform":
        st = np.full((J, I), 1.7)
        ss = np.minimum(ss, 1.5)
    sets = [O.Ordinates(*W.random_directions(M, seed=M + I, weights="random")) for M in (7, 18)]
    inf = W.random_inflow(I, J, seed=3, per_ordinate_M=25) if inflow == "ordinates" else None
    for tile_g in (2, 4):
        phi, leak, bal, stats = solve(rom, I, J, st, ss, q, sets, inf, scheme=rom.SCHEME[scheme],
                                      fixed_iters=3, tile_g=tile_g, rows_per_step=1)
        ref, rleak = oracle(I, J, st, ss, q, sets, inf, scheme=scheme, fixed_iters=3)
        assert stats["rows_per_step"] == 1
        for k in range(2):
            assert rel(phi[k], ref[k]) < TOL, (tile_g, k)
            assert abs(leak[k] - rleak[k]) < 1e-5 * (abs(rleak[k]) + np.sum(q) * 1.17 / (I * J))
        assert np.all(bal < 1e-5)


@pytest.mark.parametrize("I", [129, 200, 256, 257, 300, 513])
@pytest.mark.parametrize("medium", ["uniform", "varying"])
@pytest.mark.parametrize("kernel", ["iso", "linear"])
def test_eight_cells_per_lane(rom, I, medium, kernel):
    """Enough items for the 8-cell lanes (two per SM), rows of one to three warps."""
    J, S = 21, 80
    st, ss, q = W.random_medium(I, J, seed=I)
    if medium == "uniform":
        st = np.full((J, I), 2.1)
        ss = np.minimum(ss, 1.8)
    sets = [O.Ordinates(*W.random_directions(9, seed=50 + k, weights="random")) for k in range(S)]
    phi, _, bal, stats = solve(rom, I, J, st, ss, q, sets, kernel=kernel, g=0.7, fixed_iters=2)
    ref, _ = oracle(I, J, st, ss, q, sets, kernel=kernel, g=0.7, fixed_iters=2)
    assert stats["rows_per_step"] == 1
    assert max(rel(phi[k], ref[k]) for k in range(S)) < TOL
    assert np.all(bal < 1e-5)


@pytest.mark.parametrize("widths", [(37, 64), (200, 256), (37, 130), (64, 3, 129)])
@pytest.mark.parametrize("n_samples", [2, 70])
def test_batch_of_narrower_grids(rom, widths, n_samples):
    """Grids narrower than the widest of the batch, whose lanes past their width idle (70
    samples a grid: enough items for the 8-cell lanes)."""
    grids, sets = [], []
    for p, I in enumerate(widths):
        J = 20 + 5 * p
        st, ss, q = W.random_medium(I, J, seed=I)
        grids.append((I, J, (0.0, 1.0, 0.0, 0.6), st, ss, q))
        sets.append([O.Ordinates(*W.random_directions(9, seed=10 * p + k, weights="random"))
                     for k in range(n_samples)])
    ctx = rom.RomContext(0)
    ctx.set_grids(grids, [n_samples] * len(grids))
    ctx.set_ordinates([(o.c, o.s, o.zeta, o.w) for s in sets for o in s])
    ctx.set_options(fixed_iters=2, rows_per_step=1)
    ctx.solve()
    for p, (I, J, b, st, ss, q) in enumerate(grids):
        ref = O.solve_xy(I, J, b, st, ss, q, sets[p], fixed_iters=2)["phi"]
        for k in range(n_samples):
            assert rel(ctx.scalar_flux(p * n_samples + k), ref[k]) < TOL, (p, k)
    ctx.close()


@pytest.mark.parametrize("grid", [(5, 8), (33, 16), (130, 18), (257, 40), (300, 12)])
@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("medium", ["uniform", "varying"])
@pytest.mark.parametrize("scheme", ["dd", "step"])
@pytest.mark.parametrize("n_samples", [2, 40])
def test_dense_mode(rom, grid, precision, medium, scheme, n_samples):
    """Per-ordinate sources in and psi out (FP32, split BF16), odd ordinate counts, an inflow
    with the fewer samples; 40 samples: enough items for the 8-cell lanes."""
    I, J = grid
    st, ss, q = W.random_medium(I, J, seed=I + J, ratio_max=0.7)
    if medium == "uniform":
        st = np.full((J, I), 1.9)
        ss = np.minimum(ss, 1.2)
    sets = [O.Ordinates(*W.random_directions(19, seed=70 + k, weights="random"))
            for k in range(n_samples)]
    inf = W.random_inflow(I, J, seed=5) if n_samples == 2 else None
    phi, _, _, stats = solve(rom, I, J, st, ss, q, sets, inf, kernel="hg", g=0.4, fixed_iters=3,
                             scheme=rom.SCHEME[scheme], dense_precision=precision)
    ref, _ = oracle(I, J, st, ss, q, sets, inf, kernel="hg", g=0.4, scheme=scheme, fixed_iters=3)
    assert stats["rows_per_step"] == 1
    assert max(rel(phi[k], ref[k]) for k in range(n_samples)) < TOL


@pytest.mark.parametrize("I,J,S,M,medium,tile_g,lit,kernel", [
    (385, 21, 160, 9, "uniform", 2, False, "iso"),
    (500, 13, 170, 9, "uniform", 4, False, "iso"),
    (448, 21, 160, 9, "varying", 2, False, "iso"),
    (391, 300, 512, 4, "varying", 4, False, "iso"),
    (300, 13, 160, 9, "uniform", 2, False, "iso"),
    (200, 21, 200, 9, "varying", 2, True, "iso"),
    (131, 21, 200, 9, "varying", 4, True, "iso"),
    (224, 17, 90, 9, "uniform", 2, False, "linear")])
def test_lane_widths_of_large_batches(rom, I, J, S, M, medium, tile_g, lit, kernel):
    """Batches on either side of the choice between 4 and 8 cells per lane (first, last and two
    other samples against the oracle)."""
    st, ss, q = W.random_medium(I, J, seed=I)
    if medium == "uniform":
        st = np.full((J, I), 2.1)
        ss = np.minimum(ss, 1.8)
    sets = [O.Ordinates(*W.random_directions(M, seed=50 + k, weights="random")) for k in range(S)]
    inflow = np.random.default_rng(I).uniform(0.0, 1.5, 2 * J + 2 * I) if lit else None
    phi, _, bal, stats = solve(rom, I, J, st, ss, q, sets, inflow, kernel=kernel, g=0.7,
                               fixed_iters=2, tile_g=tile_g, rows_per_step=1)
    some = [0, 1, S // 2, S - 1]
    ref, _ = oracle(I, J, st, ss, q, [sets[k] for k in some], inflow, kernel=kernel, g=0.7,
                    fixed_iters=2)
    assert stats["rows_per_step"] == 1
    for n, k in enumerate(some):
        assert rel(phi[k], ref[n]) < TOL, k
    assert np.all(bal < 1e-5)
