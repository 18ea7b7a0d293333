"""Flag-free two-grid steps run blocks of 256 threads where these tile every row
(nx a multiple of 512) and of 64 or 128 elsewhere. A box of two equal periods in x
takes the first and must hold, bit for bit, two copies of the box of one period."""
import pytest
import torch

from gpu_helpers import ensure_built

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage", ["f32", "f16s", "bf16s"])
@pytest.mark.parametrize("dims", [(256, 40, 30), (512, 23, 27)])  # rows of one and of two blocks
def test_two_periods(storage, dims):
    ensure_built()
    from paper_1112_0850_gb300.lattice import Lattice
    nx, ny, nz = dims
    g = torch.Generator(device="cuda").manual_seed(nx)
    u = 0.05 * (2 * torch.rand(3, nz, ny, nx, generator=g, device="cuda") - 1)
    res = []
    for copies in (1, 2):
        lat = Lattice(copies * nx, ny, nz, tau=0.7, storage=storage)
        assert (copies * nx * ny * nz // 2 > 300000) == (copies == 2)
        lat.init_equilibrium(u.repeat(1, 1, 1, copies).contiguous())
        lat.step(3)
        totals = lat.step_reduce(2)
        res.append((lat.macros(), totals))
        lat.close()
    (one, tot1), (two, tot2) = res
    for a, b in zip(one, two):
        assert torch.equal(b, torch.cat((a, a), dim=-1))
    # FP64 sums of at most 2500 exact partials: 2500 * 2^-53 of their magnitudes (< 3e4 for momentum)
    assert tot2 == pytest.approx(2 * tot1, rel=1e-12, abs=1e-8)
