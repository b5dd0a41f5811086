"""Energies of lattices whose every neighbour lies in the outer part of the cut-off
sphere, against long double: the tabulated pair passes have to hold the terms to
their own size there, not to that of a bond (csrc/radial_table.cuh).

An FCC lattice expanded to a nearest distance of 4.2 to 4.95 A (the second shell
is beyond the list), equal sites, one radial term alone: the density (E_V follows
its square root) or the pair term.  Coordinates are multiples of 2^-7 A, so every
separation is exact.

Tolerance, relative, with u = 2^-53.  FP64: |d|^2 + s^2 is rounded at 25 u, which
moves a term g by 25 u |g'| / (2 r g); 4 u for the table and the sums.  FP32 modes:
float-float terms, 2^-44 where the switch is above 0.3.
"""
import numpy as np
import pytest

from paper_1910_01235_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1910_01235_gb300 import mxe as M  # noqa: E402

LD = np.longdouble
SIGMA, X = 2.0**-9, 0.96875


def term(lam, r):
    """exp(lam (2.5 - r)) S(r) with the switch from 4.5 to 5, and S"""
    u = np.clip((LD(5.0) - r) / LD(0.5), LD(0.0), LD(1.0))
    t = 1 - u
    S = u * u * u * (6 * t * t + 3 * t + 1)
    return np.exp(LD(lam * 2.5) - LD(lam) * r) * S, S


def lattice(half, lam, density):
    pot = W.potential_single()
    if density:
        pot.phi_A[:] = 0.0
        pot.f_q[:], pot.f_r0[:] = lam * 2.5, 2.5
    else:
        pot.f_xi[:] = 0.0
        pot.E[:] = 0.0
        pot.phi_A[:], pot.phi_p[:], pot.phi_r0[:] = 1.0, lam * 2.5, 2.5
    s = W.config_vacancy_lattice(4, a=2 * half, pot=pot)
    s.x[:], s.sigma[:] = X, SIGMA
    return s


def reference(half, lam, density):
    """(E_V per site, |g'/g| at the nearest distance, S there)"""
    s, D2 = LD(2.449489742783178098197284 * SIGMA), 2 * LD(half) ** 2
    w = np.array([D2 + s * s + sg * 2 * s * d for d in (LD(half), LD(half), LD(0.0)) for sg in (1, -1)], dtype=LD)
    r = np.sqrt(D2)
    slope = abs(np.log(term(lam, r + LD(1e-6))[0] / term(lam, r - LD(1e-6))[0]) / LD(2e-6))
    avg = term(lam, np.sqrt(w))[0].mean()
    if density:
        rho, mean = 12 * LD(X) * term(lam, r)[0], 12 * LD(X) * avg
        E = -LD(X) * (np.sqrt(rho) + (mean - rho) / (2 * np.sqrt(rho)))
    else:
        E = LD(X) * LD(X) * 6 * avg
    return E, float(slope), float(term(lam, r)[1])


def error(half, lam, density, precision):
    s = lattice(half, lam, density)
    g = M.MxeSystem(s, precision)
    g.build_neighbors()
    g.free_energy_grad()
    E, slope, S = reference(half, lam, density)
    return float(abs(LD(float(g.F4[0])) / s.n / E - 1)), slope, S


@pytest.mark.parametrize("density", [True, False])
@pytest.mark.parametrize("lam", [1.2, 1.96, 2.5])
@pytest.mark.parametrize("half", [3.0, 3.25, 3.390625, 3.453125, 3.5])
def test_fp64(half, lam, density):
    off, slope, _ = error(half, lam, density, "fp64")
    assert off <= 2.0**-53 * (25.0 * slope / (2.0 * half * 2.0**0.5) + 4.0)


@pytest.mark.parametrize("precision", ["mixed", "ff"])
@pytest.mark.parametrize("density", [True, False])
@pytest.mark.parametrize("lam", [1.2, 1.96, 2.5])
@pytest.mark.parametrize("half", [3.0, 3.25, 3.390625])
def test_float_float(half, lam, density, precision):
    off, _, S = error(half, lam, density, precision)
    assert S >= 0.3 and off <= 2.0**-44


@pytest.mark.parametrize("precision", ["mixed", "ff"])
@pytest.mark.parametrize("density", [True, False])
@pytest.mark.parametrize("lam", [1.2, 1.96, 2.5])
@pytest.mark.parametrize("half", [3.453125, 3.484375, 3.5, 3.515625])
def test_float_float_before_the_cutoff(half, lam, density, precision):
    """Where the switch S is small: within the float-float rounding of 1 - S, 2^-47
    of the unswitched term."""
    off, _, S = error(half, lam, density, precision)
    assert S < 0.1 and off <= 2.0**-47 / S
