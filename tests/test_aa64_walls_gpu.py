"""Solid cells of an FP64 AA lattice take no part in its arithmetic: their slots hold
NaN, which would send every warp with one of them through the FP64 form of the
collision. A walled channel's step then costs several times the two-grid one; it
stays within 3 times it (1.5 measured), and the two give the same fields."""
import pytest
import torch

import lbm_inputs
from gpu_helpers import ensure_built

pytestmark = pytest.mark.gpu


def test_walled_aa_step_stays_near_the_two_grid_one():
    from paper_1112_0850_gb300.lattice import Lattice
    ensure_built()
    nx, ny, nz = 128, 96, 96
    flags = lbm_inputs.channel_flags(nx, ny, nz, 0.1, lbm_inputs.seed_for(1))
    u0 = 0.03 * torch.randn(3, nz, ny, nx, generator=torch.Generator().manual_seed(2), dtype=torch.float64).cuda()
    ms, fields = {}, {}
    for pattern in ("pull", "aa"):
        lat = Lattice(nx, ny, nz, 0.55, flags=flags, force=(1e-6, 0.0, 0.0), storage="f64", pattern=pattern)
        lat.init_equilibrium(u0)
        lat.step(9)
        fields[pattern] = lat.macros()
        lat.prepare_steps(20)
        ms[pattern] = min(lat.step_timed(20) for _ in range(5))
        lat.close()
    for a, b in zip(fields["pull"], fields["aa"]):
        assert torch.allclose(a, b, rtol=0, atol=1e-14)
    assert ms["aa"] <= 3 * ms["pull"], ms
