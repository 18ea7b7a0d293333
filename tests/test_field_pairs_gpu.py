"""The lattice readers and writers work on cell pairs and move canonical
arrays two elements at a time where these are aligned: odd and even rows, the
shortest rows, arrays that start on an odd element, walls that move and rest,
every layout (the AA pattern's two included), against the same call on aligned
arrays and against the input."""
import numpy as np
import pytest
import torch

from gpu_helpers import ensure_built

pytestmark = pytest.mark.gpu

CASES = [(s, "pull") for s in ("f64", "f32", "f16s", "bf16s", "f16m", "bf16m")] + [
    (s, "aa") for s in ("f64", "f32", "f16s", "bf16s")]
DTYPE = {"f64": torch.float64, "f32": torch.float32, "f16s": torch.float16, "bf16s": torch.bfloat16}


def _lattice(storage, pattern, nx, ny, nz, walls):
    from paper_1112_0850_gb300.lattice import Lattice
    ensure_built()
    flags = None
    if walls:
        rng = np.random.default_rng(5)
        flags = (rng.random((nz, ny, nx)) < 0.25).astype(np.uint8)
        flags[rng.random((nz, ny, nx)) < 0.1] = 2
        flags[0, 0, 0] = 0
    lat = Lattice(nx, ny, nz, 0.6, flags=flags, storage=storage, pattern=pattern)
    if walls:
        lat.set_wall_velocity((0.03, -0.02, 0.01))
    fluid = torch.ones(nz, ny, nx, dtype=torch.bool) if flags is None else torch.tensor(flags == 0)
    return lat, fluid.cuda()


def _odd(t):
    """The same values, contiguous, starting one element past an aligned address."""
    b = torch.empty(t.numel() + 1, dtype=t.dtype, device="cuda")
    b[1:] = t.reshape(-1)
    return b[1:].view(t.shape)


@pytest.mark.parametrize("walls", [False, True])
@pytest.mark.parametrize("shape", [(1, 3, 2), (2, 2, 3), (7, 5, 4), (34, 3, 5), (67, 4, 3)])
@pytest.mark.parametrize("storage,pattern", CASES)
def test_state_round_trip_any_alignment(storage, pattern, shape, walls):
    lat, fluid = _lattice(storage, pattern, *shape, walls)
    gen = torch.Generator(device="cuda").manual_seed(3)
    # small whole multiples of 2^-9: exact in every format, and their moments too
    s = torch.randint(-3, 4, (19,) + tuple(fluid.shape), generator=gen, device="cuda").double() * 2.0 ** -9
    for fmt, dt in DTYPE.items():
        x = s.to(dt)
        for src in (x, _odd(x)):
            lat.set_state(src)
            for own, odt in DTYPE.items():
                a = lat.get_state(own)
                b = _odd(torch.zeros_like(a))
                lat.get_state(own, out=b)
                assert torch.equal(a, b)
                if storage.endswith("m"):  # remainders below 2^-4, rounded to bfloat16's 2^-8 at worst
                    assert float((a.double() - s * fluid).abs().max()) <= 2.0 ** -8 * 2.0 ** -4
                elif not walls or storage == "f64":
                    assert torch.allclose(a.double(), s * fluid, rtol=0, atol=1e-17)
                else:
                    # a value bounced off a moving wall is stored with the wall's term taken off and read
                    # with it put back: two roundings of values below 2^-5
                    u = {"f32": 2.0 ** -24, "f16s": 2.0 ** -11, "bf16s": 2.0 ** -8}[storage]
                    assert float((a.double() - s * fluid).abs().max()) <= 2 * 2.0 ** -5 * u
    lat.close()


@pytest.mark.parametrize("walls", [False, True])
@pytest.mark.parametrize("shape", [(2, 2, 3), (34, 3, 5), (67, 4, 3)])
@pytest.mark.parametrize("storage,pattern", CASES)
def test_fields_any_alignment(storage, pattern, shape, walls):
    """init_equilibrium, macros, get_state and adjoint_seed with arrays that start on an
    odd element, bit for bit as with aligned ones, before a step and after one (the
    swapped AA layout)."""
    lat, fluid = _lattice(storage, pattern, *shape, walls)
    gen = torch.Generator(device="cuda").manual_seed(4)
    field = lambda *lead: torch.randn(*lead, *fluid.shape, generator=gen, device="cuda", dtype=lat.real)  # noqa: E731
    u, rho, g, gr = 0.02 * field(3), 1 + 0.01 * field(), field(3), field()
    seen = []
    for shift in (lambda t: t, _odd):
        lat.init_equilibrium(shift(u), shift(rho))
        for step in range(2):
            lat.step(step)
            state = shift(torch.zeros(19, *fluid.shape, dtype=DTYPE[storage.replace("m", "s")], device="cuda"))
            r, v, grad = shift(torch.zeros_like(rho)), shift(torch.zeros_like(u)), shift(torch.zeros_like(u))
            lat.get_state(storage, out=state)
            lat.macros(r, v)
            lat.adjoint_seed(shift(g), shift(gr), grad)
            du, dr = shift(torch.zeros_like(u)), shift(torch.zeros_like(rho))
            lat.adjoint_init_grad(shift(u), shift(rho), du, dr)  # (reads the seeded adjoint state)
            seen.append([t.clone() for t in (state, r, v, grad, du, dr)])
    for a, b in zip(seen[:2], seen[2:]):
        for x, y in zip(a, b):
            assert torch.equal(x, y)
    # the layouts agree: the state after a step is the one of the two-grid pattern
    if pattern == "aa":
        two, _ = _lattice(storage, "pull", *shape, walls)
        two.init_equilibrium(u, rho)
        for step in range(2):
            two.step(step)
            got, want = seen[step][0].double(), two.get_state(storage).double()
            eps = {"f64": 1e-15, "f32": 1e-7, "f16s": 2.0 ** -11, "bf16s": 2.0 ** -8}[storage]
            # one step's roundings of values below 2^-4 at the storage's precision (a
            # moving wall's term is added before or after one of them)
            assert float((got - want).abs().max()) <= 4 * 2.0 ** -4 * eps
        two.close()
    lat.close()
