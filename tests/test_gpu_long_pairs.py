"""Pairs from 8 A on whose nodes reach inside the longest tabulated cut-offs
(csrc/radial_table.cuh: squared distances up to 128 in fixed point), against the
oracle; and beyond 11.3 A, in lists with a wide skin.

Tolerance: 1e-11 of the largest component for FP64 and float-float quantities,
1e-4 for FP32 forces.
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


def off(a, b):
    a, b = a.cpu().numpy(), np.asarray(b)
    return np.abs(a - b).max() / np.abs(b).max()


@pytest.mark.parametrize("precision", ["fp64", "mixed", "ff"])
@pytest.mark.parametrize("cells,rc,sigma,skin", [(5, 7.7, 0.2, 0.2), (5, 7.4, 0.35, 0.2), (7, 7.7, 0.2, 4.0)])
def test_wide_sites_at_long_cutoffs(cells, rc, sigma, skin, precision):
    s = W.perturb(W.config_vacancy_lattice(cells, sigma0=sigma), 0.05, 0.02, seed=51)
    s.pot.r_switch, s.pot.r_cut = rc - 0.7, rc
    g = M.MxeSystem(s, precision, skin=skin)
    g.build_neighbors()
    st, offs, idx = O.neighbors(s.q, s.L, g.r_list)
    fe = O.free_energy(s, (offs, idx))
    assert st == O.OK and fe["status"] == O.OK and g.r_list > 8.0
    ftol = 1e-11 if precision == "fp64" else 1e-4
    g.free_energy_grad()
    for k, tol in (("F4", 1e-11), ("mu_ex", 1e-11), ("mu", 1e-11), ("gq", ftol), ("gs", ftol)):
        assert off(getattr(g, k), fe[k]) <= tol
    sto, it, fm, qo, so = O.relax(s, 0.0, 3)
    g.relax(0.0, 3)
    tol = 1e-9 if precision == "fp64" else 1e-5
    assert np.abs(g.q.cpu().numpy() - qo).max() <= tol and np.abs(g.sigma.cpu().numpy() - so).max() <= tol
