"""The FP64 two-grid step and the odd AA step take 32-bit lattice offsets below
2^32 elements and 64-bit ones past that. Rows padded to 4096 bytes make lattices
beyond the limit from few cells; they must evolve bit for bit as the same cells
unpadded. Device memory: up to 70 GB (FP64, two lattices)."""
import numpy as np
import pytest
import torch

import lbm_inputs
from gpu_helpers import ensure_built

pytestmark = pytest.mark.gpu

PAD = 4096  # bytes per padded row


@pytest.mark.parametrize("storage,pattern,n", [("f64", "pull", 665), ("f32", "aa", 470), ("f16s", "aa", 333)])
def test_past_32bit_offsets_matches_unpadded_bit_for_bit(storage, pattern, n):
    from paper_1112_0850_gb300.lattice import Lattice
    ensure_built()
    pitch = PAD // {"f64": 8, "f32": 4, "f16s": 2}[storage]
    assert 19 * n * n * pitch >= 2 ** 32
    flags = lbm_inputs.channel_flags(8, n, n, 0.1, lbm_inputs.seed_for(1))
    rng = np.random.default_rng(5)
    u0 = 0.02 * rng.standard_normal((3, n, n, 8)) * (flags == 0)
    states = []
    for align in (PAD, 0):
        lat = Lattice(8, n, n, 0.55, flags=flags, force=(1e-5, -2e-6, 3e-6), storage=storage, pattern=pattern,
                      row_align=align)
        assert lat.info.pitch == (pitch if align else 8)
        lat.init_equilibrium(torch.tensor(u0, dtype=lat.real, device="cuda"))
        lat.step(1)
        lat.step(5)
        states.append(lat.get_state())
        assert lat.status_word() == 0
        lat.close()
    assert torch.count_nonzero(states[1]).item() > 0
    assert torch.equal(states[0], states[1])
