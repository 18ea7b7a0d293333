"""FP64 storage collides in block fixed point and, outside its range, in FP64:
one step from states inside the range, across its edges (|s|, rho - 1 and j = 1/4)
and beyond it, from values of 1e-200 and of mixed size in one cell, and
of exact zeros, against the same step in extended precision; both streaming
patterns, and a state that is not a number."""
import numpy as np
import pytest
import torch

from gpu_helpers import ensure_built

pytestmark = pytest.mark.gpu


def _step(s, tau, F, incomp, e, w):
    """One stream-collide step of the shifted state s [19][nz][ny][nx], periodic."""
    L = np.longdouble
    s, om, F = s.astype(L), L(1) / L(tau), F.astype(L)
    om = L(float(1.0 / tau))  # (the library's omega: 1/tau rounded to FP64)
    ww = [L(1) / 3 if i == 0 else (L(1) / 18 if i <= 6 else L(1) / 36) for i in range(19)]
    r = s.sum(0)
    j = [sum(int(e[i, a]) * s[i] for i in range(19)) + F[a] / 2 for a in range(3)]
    u = j if incomp else [v / (1 + r) for v in j]
    rho = L(1) if incomp else 1 + r
    usq, uF = sum(v * v for v in u), sum(u[a] * F[a] for a in range(3))
    out = np.empty_like(s)
    for i in range(19):
        eu = sum(int(e[i, a]) * u[a] for a in range(3))
        eF = sum(int(e[i, a]) * F[a] for a in range(3))
        P = s[i] + om * (ww[i] * (r + rho * (3 * eu + L(4.5) * eu * eu - L(1.5) * usq)) - s[i]) \
            + (1 - om / 2) * ww[i] * (3 * (eF - uF) + 9 * eu * eF)
        out[i] = np.roll(P, (int(e[i, 2]), int(e[i, 1]), int(e[i, 0])), (0, 1, 2))
    return out


@pytest.mark.parametrize("incomp", [False, True])
@pytest.mark.parametrize("force", [0.0, 1e-3])
@pytest.mark.parametrize("kind", ["small", "edge", "beyond", "tiny", "mixed"])
@pytest.mark.parametrize("pattern", ["pull", "aa"])
def test_fp64_step_against_extended_precision(pattern, kind, force, incomp):
    from paper_1112_0850_gb300.lattice import Lattice, lattice_table
    ensure_built()
    e, w, _ = lattice_table()
    nx, ny, nz, tau = 37, 5, 4, 0.53
    rng = np.random.default_rng(7)
    shape = (19, nz, ny, nx)
    s = rng.standard_normal(shape) * np.asarray(w)[:, None, None, None]
    scale = {"small": 0.03, "edge": 0.0, "beyond": 0.5, "tiny": 1e-200, "mixed": 0.0}[kind]
    if kind == "edge":  # cells on either side of each limit
        s *= rng.uniform(0.1, 0.8, (1, nz, ny, nx))
        s[3][s[3] > 0.05] = 0.25
        s[4][s[4] > 0.05] = np.nextafter(0.25, 0)
    elif kind == "mixed":
        s *= 10.0 ** rng.uniform(-300, -2, shape)
    else:
        s *= scale
        if kind == "beyond":  # a density near 3/2, all of it above rest in the rest population
            s[0] += 0.5
    s[:, 0, 0, :9] = 0.0
    F = force * max(scale, 1e-200 if kind == "tiny" else 0.1) * np.array([1.0, -0.5, 0.25])
    lat = Lattice(nx, ny, nz, tau, force=F if force else None, storage="f64", pattern=pattern,
                  model="incompressible" if incomp else "qian")
    lat.set_state(torch.tensor(s).cuda())
    for steps in range(1, 4 if kind in ("small", "tiny") else 2):
        lat.step(1)
        s = _step(s, tau, F, incomp, e, w)
        got = lat.get_state().cpu().numpy()
        # per population a few roundings of the cell's largest value (or of what a
        # large velocity makes of it): 16 ulp of the state's largest
        top = np.abs(s.astype(np.float64)).max()
        assert np.abs((got - s).astype(np.float64)).max() <= 16 * steps * 2.0 ** -53 * top, (kind, steps)
    lat.close()


def test_fp64_rest_stays_zero_and_nan_is_reported():
    from paper_1112_0850_gb300.capi import LBMError
    from paper_1112_0850_gb300.lattice import Lattice
    ensure_built()
    lat = Lattice(33, 4, 3, 0.6, storage="f64")
    lat.step(5)
    assert not lat.get_state().abs().any()
    s = torch.zeros(19, 3, 4, 33, dtype=torch.float64, device="cuda")
    s[5, 1, 1, 1] = float("nan")
    lat.set_state(s)
    lat.step(1)
    with pytest.raises(LBMError):
        lat.synchronize()
    lat.close()
