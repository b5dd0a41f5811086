"""Binary alloys with cut-offs on both sides of what fits one block's shared memory
(csrc/radial_table.cu): every call that reads a radial table, against the oracle.

Tolerance: 1e-11 of the largest component as for the other FP64 and float-float
quantities, 1e-4 for FP32 forces.
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


@pytest.mark.parametrize("rc", [5.5, 6.2])
@pytest.mark.parametrize("precision", ["fp64", "mixed", "ff"])
def test_long_cutoffs(rc, precision):
    s = W.perturb(W.config_binary_alloy(4), 0.05, 0.02, seed=41)
    s.pot.r_switch, s.pot.r_cut = rc - 0.5, rc
    g = M.MxeSystem(s, precision)
    g.build_neighbors()
    st, offs, idx = O.neighbors(s.q, s.L, g.r_list)
    fe = O.free_energy(s, (offs, idx))
    assert st == O.OK and fe["status"] == O.OK
    ftol = 1e-11 if precision == "fp64" else 1e-4
    g.free_energy_grad()
    for k, tol in (("F4", 1e-11), ("mu_ex", 1e-11), ("mu", 1e-11), ("gq", ftol), ("gs", ftol)):
        assert off(getattr(g, k), fe[k]) <= tol
    t = g.tangent()
    for k in ("gq", "gs", "mu_ex"):
        assert off(t[k], fe[k]) <= 1e-11
    ex = O.free_energy_exact(s, (offs, idx))
    g.set_embedding("exact")
    g.free_energy_grad()
    assert off(g.F4, ex["F4"]) <= 1e-11 and off(g.mu_ex, ex["mu_ex"]) <= 1e-11
