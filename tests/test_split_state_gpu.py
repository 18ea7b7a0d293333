"""Setting the state of a moment-split lattice rounds its momentum words and its
remainders once, whatever format the state comes in: the values of a FP32 or 16-bit
state set as they are, and as the same numbers in FP64, give the same lattice bit
for bit (next to walls at rest and moving ones, in even and odd rows)."""
import numpy as np
import pytest
import torch

from gpu_helpers import ensure_built

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("walls", ["none", "rest", "moving"])
@pytest.mark.parametrize("shape", [(96, 40, 33), (95, 41, 32)])
@pytest.mark.parametrize("storage", ["f16m", "bf16m"])
def test_state_is_rounded_once(storage, shape, walls):
    from paper_1112_0850_gb300.lattice import Lattice
    ensure_built()
    nx, ny, nz = shape
    rng = np.random.default_rng(11)
    flags = None
    if walls != "none":
        flags = (rng.random((nz, ny, nx)) < 0.1).astype(np.uint8) * (2 if walls == "moving" else 1)
    # equilibrium-like values of many sizes, a momentum that nearly cancels in places
    w = np.array([1 / 3] + 6 * [1 / 18] + 12 * [1 / 36])[:, None, None, None]
    s = w * rng.standard_normal((19, nz, ny, nx)) * 10.0 ** rng.uniform(-6, -1, (1, nz, ny, nx))
    lats = [Lattice(nx, ny, nz, 0.6, flags=flags, storage=storage) for _ in range(2)]
    for fmt in (torch.float32, torch.float16, torch.bfloat16):
        x = torch.tensor(s).cuda().to(fmt)
        for lat, v in zip(lats, (x, x.double())):
            lat.set_wall_velocity((0.03, -0.02, 0.01))
            lat.set_state(v)
        assert torch.equal(lats[0].get_state("f32"), lats[1].get_state("f32")), fmt
    for lat in lats:
        lat.close()
