"""Two species whose density term is one and the same at every site and from
every neighbour (one distinct density term, three pair terms): the geometry
record of a pair is split into its density and pair-term planes although the
densities fill only half of the first.

Tolerance: float-float pair terms carry at most 2^-46 each and the sums cancel
by at most a factor ~30: 1e-11 of the largest component.
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


def shared_density():
    s = W.perturb(W.config_binary_alloy(4), 0.05, 0.02, seed=11)
    P = W.potential_binary()
    P.cross_geomean = False
    P.phi_A[0, 1] = P.phi_A[1, 0] = 0.2
    P.phi_p[0, 1] = P.phi_p[1, 0] = 4.0
    P.phi_r0[0, 1] = P.phi_r0[1, 0] = 2.5
    P.f_q[:] = 5.0
    P.f_xi[:] = 1.0
    P.f_r0[:] = 2.55
    s.pot = P
    return s


@pytest.mark.parametrize("precision", ["fp64", "mixed", "ff"])
def test_energy_and_chemical_potentials(precision):
    s = shared_density()
    g = M.MxeSystem(s, precision)
    g.build_neighbors()
    g.free_energy_grad()
    st, off, idx = O.neighbors(s.q, s.L, g.r_list)
    fe = O.free_energy(s, (off, idx))
    assert st == O.OK and fe["status"] == O.OK
    for a, b in ((g.F4, fe["F4"]), (g.mu_ex, fe["mu_ex"]), (g.mu, fe["mu"])):
        assert np.abs(a.cpu().numpy() - b).max() <= 1e-11 * np.abs(b).max()
