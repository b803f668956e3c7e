"""Device memory of the linear kernel's per-sample state."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_linear_kernel_keeps_one_moment_of_phi():
    """The iterate's currents are kept only in the source they enter: one array of phi, three of
    sources and three of accumulators (64 samples of 512 x 512: 67 MB each), beside the grid and
    a few pages."""
    import torch
    import __graft_entry__
    __graft_entry__.build()
    from paper_2407_12527_gb300 import rom as R
    I = J = 512
    S = 64

    def context():
        ctx = R.RomContext(0)
        ctx.set_grid(I, J, (0.0, 1.0, 0.0, 1.0), 1.0, 0.5, 1.0)
        ctx.set_ordinates_seed(5, [1] * S, [1] * S)
        ctx.set_kernel("linear", 0.5)
        ctx.set_options(fixed_iters=2)
        return ctx

    warm = context()  # the library's modules are loaded at its first launches
    warm.solve()
    warm.close()
    torch.cuda.synchronize()
    ctx = context()
    before = torch.cuda.mem_get_info()[0]
    ctx.solve()
    used = before - torch.cuda.mem_get_info()[0]
    phi = ctx.scalar_flux(S - 1)
    ctx.close()
    assert used < 7.5 * S * I * J * 4
    assert np.all(np.isfinite(phi)) and phi.min() > 0.0
