"""States at the edges of what the radial tables hold (csrc/radial_table.cuh,
csrc/pair_table.cu)."""
import numpy as np
import pytest

import oracle as O
from paper_1910_01235_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1910_01235_gb300 import mxe as M  # noqa: E402


@pytest.mark.parametrize("precision", ["fp64", "mixed", "ff"])
def test_status_of_a_node_on_a_site(precision):
    """The node of a site that falls on its neighbour to the last bit: |d|^2 + s^2
    and 2 s |d_a|, each rounded, differ by -2^-50 here.  Reported as any node
    below 0.5 A, with none of the pair's other nodes below 1.25 A."""
    s = W.config_vacancy_lattice(4, x0=1.0)
    s.q[:, 0] = 0.0
    s.q[:, 1] = (1.6870144847575537, 0.0, 0.0)
    s.sigma[:] = 0.01
    s.sigma[0] = 0.688720779390046
    st, offs, idx = O.neighbors(s.q, s.L, 7.0)
    assert O.free_energy(s, (offs, idx))["status"] == O.ERR_GEOMETRY
    g = M.MxeSystem(s, precision)
    g.build_neighbors()
    with pytest.raises(M.MxeError) as e:
        g.free_energy_grad()
    assert e.value.status == M.ERR_GEOMETRY


@pytest.mark.parametrize("x", [2e-11, 6e-12, 1e-12, 4e-13, 1e-14, 1e-20])
def test_fp64_forces_of_traces_alone(x):
    """One species of traces without density: every weight of a pair is x^2, small
    enough in the middle of this range to have no float pair while the integer
    part still holds it.  The forces scale with x^2, so the bound is that of the
    other FP64 passes, 1e-11 of the largest component."""
    pot = W.potential_single()
    pot.f_xi[:] = 0.0
    pot.E[:] = 0.0
    s = W.perturb(W.config_vacancy_lattice(4, pot=pot), 0.05, 0.02, seed=21)
    s.x[:] = x
    g = M.MxeSystem(s, "fp64")
    g.build_neighbors()
    g.free_energy_grad()
    st, offs, idx = O.neighbors(s.q, s.L, g.r_list)
    fe = O.free_energy(s, (offs, idx))
    assert st == O.OK and fe["status"] == O.OK
    assert np.abs(g.gq.cpu().numpy() - fe["gq"]).max() <= 1e-11 * np.abs(fe["gq"]).max()


@pytest.mark.parametrize("scale", [1e-18, 1e-22, 1e-28, 2e-29])
@pytest.mark.parametrize("precision", ["mixed", "ff"])
def test_faint_pair_terms(scale, precision):
    """A pair term too small for the exponents of a table's rows, alone:
    chemical potentials relative to their own size (float-float terms, 1e-11)."""
    pot = W.potential_single(A=0.3 * scale)
    pot.f_xi[:] = 0.0
    pot.E[:] = 0.0
    s = W.perturb(W.config_vacancy_lattice(4, pot=pot), 0.05, 0.02, seed=22)
    g = M.MxeSystem(s, precision)
    g.build_neighbors()
    g.free_energy_grad()
    st, offs, idx = O.neighbors(s.q, s.L, g.r_list)
    fe = O.free_energy(s, (offs, idx))
    assert st == O.OK and fe["status"] == O.OK
    assert np.abs(g.mu_ex.cpu().numpy() - fe["mu_ex"]).max() <= 1e-11 * np.abs(fe["mu_ex"]).max()
