"""The initial state bit for bit: lbm_init_equilibrium evaluates one FP32
expression per direction in a fixed order of roundings, and the 16-bit formats
store it rounded once. (Another order of the same expression is as accurate, but
moves single values of a 16-bit state by a whole storage step, and with them the
fields of the run that starts from it.)"""
import numpy as np
import pytest
import torch

from gpu_helpers import ensure_built

pytestmark = pytest.mark.gpu
f32 = np.float32


def _fma(a, b, c):
    """a b + c of FP32 values rounded to FP32 (the product is exact in FP64)."""
    return (np.float64(a) * np.float64(b) + np.float64(c)).astype(f32)


def _equilibrium(rho, u, incomp, e):
    r1 = rho - f32(1)
    mass = f32(1) + r1 if not incomp else np.ones_like(r1)
    ux, uy, uz = u
    usq = _fma(uz, uz, _fma(ux, ux, uy * uy))
    out = []
    for i in range(19):
        w = f32(1 / 3 if i == 0 else (1 / 18 if i <= 6 else 1 / 36))
        eu = np.zeros_like(ux)
        for a in range(3):
            if e[i, a]:
                eu = eu + f32(e[i, a]) * u[a]
        sq = f32(4.5) * eu * eu
        out.append(w * _fma(mass, _fma(f32(-1.5), usq, _fma(f32(3), eu, sq)), r1))
    return np.stack(out)


@pytest.mark.parametrize("pattern", ["pull", "aa"])
@pytest.mark.parametrize("model", ["qian", "incompressible"])
@pytest.mark.parametrize("storage", ["f32", "f16s", "bf16s"])
@pytest.mark.parametrize("shape,with_rho", [((5, 6, 66), True), ((4, 5, 37), True), ((3, 3, 64), False)])
def test_initial_state_bits(storage, model, pattern, shape, with_rho):
    from paper_1112_0850_gb300.lattice import Lattice, lattice_table
    ensure_built()
    nz, ny, nx = shape
    rng = np.random.default_rng(3)
    u = (0.05 * rng.standard_normal((3,) + shape)).astype(f32)
    rho = (1 + 0.02 * rng.standard_normal(shape)).astype(f32) if with_rho else np.ones(shape, f32)
    lat = Lattice(nx, ny, nz, 0.6, storage=storage, pattern=pattern, model=model)
    lat.init_equilibrium(torch.tensor(u).cuda(), torch.tensor(rho).cuda() if with_rho else None)
    got = lat.get_state()
    want = torch.tensor(_equilibrium(rho, u, model == "incompressible", np.asarray(lattice_table()[0])))
    assert torch.equal(got.cpu(), want.to(got.dtype))
    lat.close()
