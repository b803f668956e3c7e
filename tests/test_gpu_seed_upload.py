"""Seeded ordinate sets are drawn without waiting for the device: sets drawn one behind the
other each come from their own tables, and a stream under capture is refused."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rom():
    import torch
    assert torch.cuda.is_available()
    import __graft_entry__
    __graft_entry__.build()
    from paper_2407_12527_gb300 import rom as R
    return R


def context(rom):
    ctx = rom.RomContext(0)
    ctx.set_grid(9, 7, (0.0, 1.0, 0.0, 1.0), 1.0, 0.5, 1.0)
    return ctx


@pytest.mark.parametrize("n", [1, 40, 5000])
def test_sets_drawn_back_to_back(rom, n):
    a, b = context(rom), context(rom)
    rng = np.random.default_rng(n)
    for seed in range(20):
        nz, nt = rng.integers(1, 4, n).tolist(), rng.integers(1, 4, n).tolist()
        a.set_ordinates_seed(seed, nz, nt)
    b.set_ordinates_seed(19, nz, nt)
    m = 4 * sum(i * j for i, j in zip(nz, nt))
    for x, y in zip(a.get_ordinates(m), b.get_ordinates(m)):
        np.testing.assert_array_equal(x, y)
    a.close()
    b.close()


def test_capture_is_refused(rom):
    import torch
    ctx = context(rom)
    s = torch.cuda.Stream()
    ctx.set_stream(s.cuda_stream)
    g = torch.cuda.CUDAGraph()
    x = torch.zeros(4, device="cuda")
    torch.cuda.synchronize()
    with torch.cuda.graph(g, stream=s):
        x += 1
        with pytest.raises(rom.RomError):
            ctx.set_ordinates_seed(1, [2], [2])
    ctx.set_ordinates_seed(1, [2], [2])
    ctx.solve()
    assert np.all(np.isfinite(ctx.scalar_flux(0)))
    ctx.close()
