"""List rebuilds with either margin of the fill without a count pass
(csrc/api.cu, build_lists): short rows, rows above 128 entries, stencils near the
limit of the staged candidates, and rows that outgrow the margin; equal to the
oracle's lists."""
import numpy as np
import pytest

import oracle as O
from paper_1910_01235_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1910_01235_gb300 import mxe as M  # noqa: E402


@pytest.mark.parametrize("cells,rc", [(6, 5.0), (12, 5.0), (16, 6.8), (16, 7.6), (20, 6.8), (20, 7.0)])
def test_rebuilds(cells, rc):
    s = W.perturb(W.config_vacancy_lattice(cells), 0.03, 0.0, seed=13)
    s.pot.r_switch, s.pot.r_cut = rc - 0.5, rc
    g = M.MxeSystem(s, "ff")
    for sigma in (0.1, 0.1, 0.12, 0.25, 0.1):
        g.sigma.fill_(sigma)
        g.build_neighbors()
        st, ro, ri = O.neighbors(s.q, s.L, g.r_list)
        assert st == O.OK
        off, idx = (t.cpu().numpy() for t in g.export_neighbors())
        np.testing.assert_array_equal(off, ro)
        np.testing.assert_array_equal(idx, ri)
