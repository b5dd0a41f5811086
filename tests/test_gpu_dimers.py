"""Energies of isolated dimers against long double: pairs near the first rows of
the radial tables (csrc/radial_table.cu), alone in their sites' sums.

Dimers along x on a cubic grid, equal sites, one radial term: the density (E_V
follows its square root) or the pair term.  Separations are multiples of 2^-10 A
and exact.

Tolerance, relative, with u = 2^-53.  FP64: 8 u for the table and the sums, and
w = |d|^2 + s^2 is rounded at w u, which moves a term g by w u |g'| / (2 r g).
FP32 modes: float-float terms, 2^-44.
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


def error(d, lam, rs, rc, density, precision):
    """(relative error of E_V, |g'/g| at d) of dimers with separation d"""
    pot = W.potential_single(r_switch=rs, r_cut=rc)
    if density:
        pot.phi_A[:] = 0.0
        pot.f_q[:], pot.f_r0[:] = lam * 2.5, 2.5
    else:
        pot.f_xi[:] = 0.0
        pot.E[:] = 0.0
        pot.phi_A[:], pot.phi_p[:], pot.phi_r0[:] = 1.0, lam * 2.5, 2.5
    s = W.config_vacancy_lattice(4, pot=pot)
    step = np.ceil(2 * (rc + 0.3)) / 2 + 1.5
    grid = np.array([(i, j, k) for i in range(4) for j in range(4) for k in range(8)], dtype=float).T * step
    s.q = np.concatenate([grid, grid + np.array([[d], [0.0], [0.0]])], axis=1)
    s.L = np.array([4 * step, 4 * step, 8 * step])
    s.x[:], s.sigma[:] = X, SIGMA

    def term(r):
        t = np.clip((r - LD(rs)) / (LD(rc) - LD(rs)), LD(0.0), LD(1.0))
        u = 1 - t
        return np.exp(LD(lam * 2.5) - LD(lam) * r) * u * u * u * (6 * t * t + 3 * t + 1)

    sh, D2 = LD(2.449489742783178098197284 * SIGMA), LD(d) * LD(d)
    w = np.array([D2 + sh * sh + sg * 2 * sh * c for c in (LD(d), LD(0.0), LD(0.0)) for sg in (1, -1)], dtype=LD)
    r = np.sqrt(D2)
    slope = float(abs(np.log(term(r + LD(1e-6)) / term(r - LD(1e-6))) / LD(2e-6)))
    avg = term(np.sqrt(w)).mean()
    if density:
        rho, mean = LD(X) * term(r), LD(X) * avg
        E = -LD(X) * (np.sqrt(rho) + (mean - rho) / (2 * np.sqrt(rho)))
    else:
        E = LD(X) * LD(X) * avg / 2
    g = M.MxeSystem(s, precision)
    g.build_neighbors()
    g.free_energy_grad()
    return float(abs(LD(float(g.F4[0])) / s.n / E - 1)), slope


def bound(precision, d, slope):
    return 2.0**-53 * (8.0 + d * slope / 2.0) if precision == "fp64" else 2.0**-44


@pytest.mark.parametrize("precision", ["fp64", "mixed", "ff"])
@pytest.mark.parametrize("density", [True, False])
@pytest.mark.parametrize("lam,rs,rc", [(1.4, 1.4, 2.8), (1.6, 2.4, 3.3), (1.9, 3.0, 4.0)])
@pytest.mark.parametrize("k", [0, 16, 64, 256])
def test_near_a_quarter_of_the_cutoff(k, lam, rs, rc, density, precision):
    d = np.ceil(rc * 256.0) / 1024.0 + (k + 8) / 1024.0
    off, slope = error(d, lam, rs, rc, density, precision)
    assert off <= bound(precision, d, slope)


@pytest.mark.parametrize("precision", ["mixed", "ff"])
@pytest.mark.parametrize("density", [True, False])
@pytest.mark.parametrize("lam,rs,rc", [(1.96, 4.5, 5.0), (2.5, 4.5, 5.0), (3.0, 5.2, 6.0)])
@pytest.mark.parametrize("d", [0.50390625, 0.5078125, 0.6005859375, 0.70703125, 0.7080078125, 0.8125, 0.9990234375, 1.0009765625,
                               1.119140625, 1.248046875, 1.2734375, 1.4140625, 1.4150390625, 1.498046875])
def test_float_float_below_the_main_rows(d, lam, rs, rc, density, precision):
    """Every octave of the graded rows and the distances at which their width changes;
    with a node below 0.5 A, the smallest admissible distance, an error."""
    if d - 2.4495 * SIGMA < 0.5:
        with pytest.raises(M.MxeError) as e:
            error(d, lam, rs, rc, density, precision)
        assert e.value.status == M.ERR_GEOMETRY
        return
    off, _ = error(d, lam, rs, rc, density, precision)
    assert off <= 2.0**-44
