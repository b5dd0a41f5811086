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
