"""The totals' integer sums (FP32 arithmetic): lattices below and above one warp,
one block and the two-stage final sum, values from 1e-12 to beyond the integer
range (which FP64 sums take over), against the FP64 sum of the fields."""
import numpy as np
import pytest
import torch

from gpu_helpers import ensure_built

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("amp,rho_max", [(1e-12, 0.0), (1e-3, 0.1), (0.1, 5.0), (0.1, 3000.0)])
@pytest.mark.parametrize("shape", [(1, 1, 1), (3, 5, 2), (64, 8, 1), (65, 33, 31), (128, 128, 140)])
@pytest.mark.parametrize("pattern", ["pull", "aa"])
def test_totals_match_fields(pattern, shape, amp, rho_max):
    from paper_1112_0850_gb300.lattice import Lattice
    ensure_built()
    nx, ny, nz = shape
    flags = None
    if nx > 3:
        flags = (np.random.default_rng(2).random((nz, ny, nx)) < 0.2).astype(np.uint8)
    lat = Lattice(nx, ny, nz, 0.7, flags=flags, storage="f32", pattern=pattern, model="incompressible")
    gen = torch.Generator(device="cuda").manual_seed(4)
    u = amp * torch.rand(3, nz, ny, nx, generator=gen, device="cuda")
    rho = 1 + rho_max * torch.rand(nz, ny, nx, generator=gen, device="cuda")
    lat.init_equilibrium(u, rho)
    r, v = lat.macros()  # (in this model v is the momentum)
    fluid = torch.ones_like(r, dtype=torch.bool) if flags is None else torch.tensor(flags == 0).cuda()
    want = np.array([r.double()[fluid].sum().item()] + [v[a].double()[fluid].sum().item() for a in range(3)])
    # macros round 1 + (rho - 1) to FP32: half an ulp of each density
    tol_rho = 2.0 ** -24 * r.abs().double()[fluid].sum().item()
    tol_j = 1e-13 * np.maximum(want[1:], 0) + 1e-30
    n = int(fluid.sum())
    for got in (lat.reduce(), lat.step_reduce(1)):
        assert abs(got[0] - want[0]) <= tol_rho
        # sums of n FP32 values: exact, against an FP64 sum of n terms, and the
        # integer grid's 2^-82 a value
        assert (np.abs(got[1:] - want[1:]) <= tol_j * max(1.0, n / 1000) + n * 2.0 ** -82).all(), (got, want)
    lat.close()


def test_totals_not_a_number():
    from paper_1112_0850_gb300.lattice import Lattice
    from paper_1112_0850_gb300.capi import LBMError
    ensure_built()
    lat = Lattice(40, 6, 5, 0.6, storage="f32")
    s = torch.zeros(19, 5, 6, 40, device="cuda")
    s[3, 2, 2, 2] = float("nan")
    lat.set_state(s)
    out = torch.zeros(4, dtype=torch.float64, device="cuda")
    try:
        lat.step_reduce(1, out)
        lat.synchronize()
    except LBMError:
        pass  # (the step reports the divergence)
    assert torch.isnan(out[0]) and torch.isnan(out[2])
    lat.close()
