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
