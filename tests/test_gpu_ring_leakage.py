"""The net leakage that the X-Y ring sweep (csrc/sweep2d_ring.cuh) keeps per sample."""
import numpy as np
import pytest

import rom_workloads as W
from oracle import oracle as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rom():
    import torch
    assert torch.cuda.is_available()
    import __graft_entry__
    __graft_entry__.build()
    from paper_2407_12527_gb300 import rom as R
    return R


@pytest.mark.parametrize("scheme", ["dd", "step"])
@pytest.mark.parametrize("medium", ["uniform", "varying"])
@pytest.mark.parametrize("kernel", ["iso", "linear"])
@pytest.mark.parametrize("inflow", ["vacuum", "isotropic"])
@pytest.mark.parametrize("tile_g", [2, 4])
@pytest.mark.parametrize("unit", [1e-30, 1e-18, 1e22])
def test_units_of_length(rom, scheme, medium, kernel, inflow, tile_g, unit):
    """Coefficients per length units other than the domain's own size.  1e-18: 1 / (sigma_T + a +
    b) is about 1e16, and a row that a lane computes past the grid's last one overflows if its
    source is the moments of another such row.  None of it reaches the leakage or the balance.
    1e-30 and 1e22: the area of a cell is outside the range of FP32, its edges are not."""
    I, J = 128, 21
    bounds = (0.0, 1.3 / unit, 0.0, 0.7 / unit)
    st, ss, q = (unit * a for a in W.random_medium(I, J, seed=5))
    if medium == "uniform":
        st = np.full((J, I), 1.7 * unit)
        ss = np.minimum(ss, 1.5 * unit)
    sets = [O.Ordinates(*W.random_directions(M, seed=M, weights="random")) for M in (7, 18)]
    inf = W.random_inflow(I, J, seed=3) if inflow == "isotropic" else None
    ctx = rom.RomContext(0)
    ctx.set_grid(I, J, bounds, st, ss, q)
    ctx.set_ordinates([(o.c, o.s, o.zeta, o.w) for o in sets])
    ctx.set_kernel(kernel, 0.6 if kernel == "linear" else 0.0)
    if inf is not None:
        off = [0, J, 2 * J, 2 * J + I, 2 * J + 2 * I]
        for f in range(4):
            ctx.set_inflow_isotropic(f, inf[off[f]:off[f + 1]])
    ctx.set_options(scheme=rom.SCHEME[scheme], fixed_iters=3, tile_g=tile_g, rows_per_step=1)
    stats = ctx.solve()
    leak, bal, _ = ctx.balance()
    phi = [ctx.scalar_flux(k) for k in range(2)]
    ctx.close()
    ref = O.solve_xy(I, J, bounds, st, ss, q, sets, inflow=inf, scheme=scheme, kernel=kernel,
                     g=0.6, fixed_iters=3)
    assert stats["rows_per_step"] == 1
    area = 1.3 * 0.7 / (I * J) / unit ** 2
    for k in range(2):
        assert np.linalg.norm(phi[k] - ref["phi"][k]) < 1e-5 * np.linalg.norm(ref["phi"][k])
        scale = abs(ref["leak"][k]) + np.sum(st * ref["phi"][k]) * area
        assert abs(leak[k] - ref["leak"][k]) < 1e-5 * scale
    assert np.all(bal < 1e-5) and np.isfinite(stats["balance_max"])


@pytest.mark.parametrize("scheme", ["dd", "step"])
@pytest.mark.parametrize("medium", ["uniform", "varying"])
@pytest.mark.parametrize("tile_g", [2, 4])
def test_rows_per_compensated_add(rom, scheme, medium, tile_g):
    """The x-face terms of the leakage go into the compensated sum at most four rows at a time.
    One ordinate along x, eight rows in one lane; the first carries 1, the others 2^-26, which
    an FP32 sum with the first's term drops (at most a quarter of its last place).  Of the seven,
    the four outside the first's sum stay: at least half of what they let out."""
    I, J, small = 4, 8, 2.0 ** -26
    st = np.full((J, I), 1e-3)
    if medium == "varying":
        st[0, 0] = 1.5e-3
    leak = []
    for rest in (0.0, small):
        ctx = rom.RomContext(0)
        ctx.set_grid(I, J, (0.0, 1.0, 0.0, float(J)), st, 0.0 * st, 0.0 * st)
        ctx.set_ordinates([(np.array([1.0]), np.array([0.0]), np.array([0.0]), np.array([1.0]))])
        ctx.set_inflow_isotropic(0, np.array([1.0] + [rest] * (J - 1)))
        ctx.set_options(scheme=rom.SCHEME[scheme], fixed_iters=1, tile_g=tile_g, rows_per_step=1)
        ctx.solve()
        leak.append(float(ctx.balance()[0][0]))
        ctx.close()
    # leakage = what goes out less what comes in; dy = 1, and e^-0.001 of the inflow passes
    out = (leak[1] - leak[0]) + 7 * small
    assert 0.5 * 7 * small * 0.99 < out < 1.01 * 7 * small
