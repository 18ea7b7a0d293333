"""States exchanged in FP64 with narrower storage, at sizes on both sides of the
lattice size and row length that choose their kernels: bit for bit the values of the
same state in the lattice's own format."""
import numpy as np
import pytest
import torch

from gpu_helpers import ensure_built

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("walls", [False, True])
@pytest.mark.parametrize("shape", [(33, 7, 5), (64, 6, 5), (127, 129, 65), (128, 129, 65)])
@pytest.mark.parametrize("pattern", ["pull", "aa"])
@pytest.mark.parametrize("storage", ["f32", "f16s", "bf16s"])
def test_fp64_states_carry_the_stored_values(storage, pattern, shape, walls):
    from paper_1112_0850_gb300.lattice import Lattice
    ensure_built()
    nx, ny, nz = shape
    flags = (np.random.default_rng(1).random((nz, ny, nx)) < 0.1).astype(np.uint8) if walls else None
    lat = Lattice(nx, ny, nz, 0.6, flags=flags, storage=storage, pattern=pattern)
    gen = torch.Generator(device="cuda").manual_seed(9)
    lat.init_equilibrium(0.03 * torch.randn(3, nz, ny, nx, generator=gen, device="cuda"))
    for step in range(2):  # (the AA pattern's two layouts)
        lat.step(step)
        own = lat.get_state()
        assert torch.equal(lat.get_state("f64"), own.double())
        # an output that starts on an odd element
        odd = torch.empty(own.numel() + 1, dtype=torch.float64, device="cuda")[1:].view(own.shape)
        lat.get_state("f64", out=odd)
        assert torch.equal(odd, own.double())
    lat.set_state(own.double())
    assert torch.equal(lat.get_state(), own)
    lat.close()
