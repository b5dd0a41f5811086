"""Potentials with more distinct density terms than the pair kernels hold (two
species, a density for every ordered pair): the contexts keep no pair index and
every call takes the full-list passes.  Energies, gradients and chemical
potentials of one call in every precision, against the oracle.

Tolerances: those of the FP64 and FP32 passes elsewhere (1e-11 of the largest
component; FP32 forces 1e-4).
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


def system(n_f):
    s = W.perturb(W.config_binary_alloy(4), 0.05, 0.02, seed=31)
    s.pot = W.potential_binary()
    s.pot.f_q[1, 0] = 4.5
    if n_f == 4:
        s.pot.f_r0[0, 1] = 2.6
    return s


def off(a, b):
    a, b = a.cpu().numpy(), np.asarray(b)
    return np.abs(a - b).max() / np.abs(b).max()


@pytest.mark.parametrize("n_f", [3, 4])
@pytest.mark.parametrize("precision", ["fp64", "mixed", "ff"])
def test_evaluation(n_f, precision):
    s = system(n_f)
    g = M.MxeSystem(s, precision)
    assert g.potential_terms()[1] == n_f
    g.build_neighbors()
    g.free_energy_grad()
    st, offs, idx = O.neighbors(s.q, s.L, g.r_list)
    fe = O.free_energy(s, (offs, idx))
    assert st == O.OK and fe["status"] == O.OK
    for k in ("F4", "mu_ex", "mu"):
        assert off(getattr(g, k), fe[k]) <= 1e-11
    for k in ("gq", "gs"):
        assert off(getattr(g, k), fe[k]) <= (1e-11 if precision == "fp64" else 1e-4)
