"""The Euler step's site factors P = D x exp(beta mu) and Q = x_v exp(-beta mu)
at the ends of the double range: low temperatures and large barriers, where a
factor under- or overflows although every hop is an ordinary number, and sites
without a species or without vacancies.

Tolerance: a factorised hop carries the rounding of beta mu (|beta mu| < 600:
7e-14 relative, twice); 1e-12 of the largest change, plus the rounding of x.
"""
import numpy as np
import pytest

import oracle as O
from paper_1910_01235_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1910_01235_gb300 import mxe as M  # noqa: E402


@pytest.mark.parametrize("mu0", [-4.9, -4.8, 0.0, 4.8, 5.2])
@pytest.mark.parametrize("Qm", [0.0, 2.0, 5.0])
def test_factors_at_the_ends_of_the_range(mu0, Qm):
    s = W.config_vacancy_lattice(4)
    s.T[:] = 100.0
    rng = np.random.default_rng(5)
    s.x[0] = rng.uniform(0.2, 0.9, s.n)
    s.x[0, ::7], s.x[0, 3::11] = 1.0, 0.0
    mu = mu0 + rng.uniform(-0.01, 0.01, s.x.shape)
    nu0 = 1e13
    D = nu0 * np.exp(-Qm / (8.617333262e-5 * 100.0))
    dt = 1e-3 / D
    g = M.MxeSystem(s, "fp64")
    g.build_neighbors()
    g.diffuse_step(dt, mu_ex=torch.as_tensor(mu, device="cuda"), nu0=nu0, Qm=Qm)
    _, offs, idx = O.neighbors(s.q, s.L, g.r_list)
    st, xo = O.diffuse_step(s, mu, O.bonds(s, g.r_bond, offs, idx), dt, nu0=nu0, Qm=Qm)
    assert st == O.OK
    dx = np.abs(xo - s.x).max()
    assert dx > 1e-5
    assert np.abs(g.x.cpu().numpy() - xo).max() <= 1e-12 * dx + 4e-16
