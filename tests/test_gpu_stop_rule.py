"""The stop rule of the source iteration (finalize_kernel, csrc/reduce.cu) where its samples
fill one warp, just more than one, and several: every sample stops by itself, on the device
loop as on the host's."""
import numpy as np
import pytest

import rom_workloads as W
from oracle import oracle as O

pytestmark = pytest.mark.gpu

I, J, BOUNDS, TOL = 12, 9, (0.0, 1.3, -0.2, 0.7), 1e-4


@pytest.fixture(scope="module")
def rom():
    import torch
    assert torch.cuda.is_available()
    import __graft_entry__
    __graft_entry__.build()
    from paper_2407_12527_gb300 import rom as R
    return R


def solve(rom, sets, **opts):
    st, ss, q = W.random_medium(I, J, seed=3)
    ctx = rom.RomContext(0)
    ctx.set_grid(I, J, BOUNDS, st, ss, q)
    ctx.set_ordinates([(o.c, o.s, o.zeta, o.w) for o in sets])
    ctx.set_options(**opts)
    ctx.solve()
    it, res = ctx.iterations()
    leak, bal, _ = ctx.balance()
    phi = np.stack([ctx.scalar_flux(k) for k in range(len(sets))])
    ctx.close()
    return np.asarray(it), np.asarray(res), leak, bal, phi


@pytest.mark.parametrize("S", [1, 31, 32, 33, 64, 70])
def test_each_sample_stops(rom, S):
    sets = [O.Ordinates(*W.random_directions(5, seed=100 + k, weights="random"))
            for k in range(S)]
    it, res, leak, bal, phi = solve(rom, sets, tol=TOL)
    assert np.all(res < TOL) and np.all(it > 1)
    # the particle balance is exact for the cell equations up to FP32 rounding
    assert np.all(bal < 1e-5)
    # the same rule on the host's loop; the residual sums are added in any order, so a sample
    # whose residual lies within their rounding of the tolerance may take one sweep more
    ih, rh, lh, bh, ph = solve(rom, sets, tol=TOL, check_every=1)
    assert np.max(np.abs(it - ih)) <= 1
    # the flux after one sweep more or less differs by at most the tolerance itself
    assert np.all(np.linalg.norm((phi - ph).reshape(S, -1), axis=1) <=
                  2 * TOL * np.linalg.norm(ph.reshape(S, -1), axis=1))
    i3 = solve(rom, sets, fixed_iters=3)[0]
    assert np.all(i3 == 3)
