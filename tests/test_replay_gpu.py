"""LBMRollout keeps no copy of the final state where a segment recomputed from its
checkpoint ends on it bit for bit. That holds for every lattice and checkpoint
format it is claimed for: even and odd numbers of steps before the checkpoint and
after it, recorded steps against replayed graphs and single ones, walls, both
patterns, and checkpoints in a wider format than the lattice's."""
import numpy as np
import pytest
import torch

from gpu_helpers import ensure_built

pytestmark = pytest.mark.gpu

FORMATS = [("f64", "f64"), ("f32", "f32"), ("f32", "f64"), ("f16s", "f16s"), ("f16s", "f32"), ("bf16s", "bf16s"),
           ("bf16s", "f32"), ("bf16s", "f64")]


@pytest.mark.parametrize("nx", [37, 64])
@pytest.mark.parametrize("walls", [False, True])
@pytest.mark.parametrize("pattern", ["pull", "aa"])
@pytest.mark.parametrize("storage,ckpt", FORMATS)
def test_recorded_replay_ends_on_the_same_bits(storage, ckpt, pattern, walls, nx):
    from paper_1112_0850_gb300 import capi
    from paper_1112_0850_gb300.lattice import Lattice
    from paper_1112_0850_gb300.rollout import _replays_exactly
    ensure_built()
    ny, nz = 11, 9
    flags = None
    if walls:
        flags = (np.random.default_rng(2).random((nz, ny, nx)) < 0.2).astype(np.uint8)
        flags[:, 0] = 1
    lat = Lattice(nx, ny, nz, 0.55, flags=flags, storage=storage, pattern=pattern)
    assert _replays_exactly(lat, capi.STORAGE[storage], capi.STORAGE[ckpt])
    gen = torch.Generator(device="cuda").manual_seed(6)
    lat.set_force_field(1e-4 * torch.randn(3, nz, ny, nx, generator=gen, device="cuda", dtype=lat.real))
    u0 = 0.03 * torch.randn(3, nz, ny, nx, generator=gen, device="cuda", dtype=lat.real)
    for before in (0, 1, 4):
        for n in (1, 2, 5):
            lat.init_equilibrium(u0)
            lat.step(before)
            kept = lat.get_state(ckpt)
            lat.step(n)
            final, fields = lat.get_state(), lat.macros()
            lat.set_state(kept)
            lat.step_record(n, lat.new_tape(n))
            assert torch.equal(lat.get_state(), final), (before, n)
            for a, b in zip(lat.macros(), fields):
                assert torch.equal(a, b), (before, n)
    lat.close()
