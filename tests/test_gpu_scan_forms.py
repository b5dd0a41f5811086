"""Lists and bonds on both sides of the length from which the row offsets take
three launches (csrc/neighbors.cu: 11,264 counts), first build and rebuild,
equal to the oracle's."""
import numpy as np
import pytest

import oracle as O
from paper_1910_01235_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1910_01235_gb300 import mxe as M  # noqa: E402


@pytest.mark.parametrize("cells,drop", [(14, 0), (15, 2236), (15, 2235), (15, 0), (16, 0)])
def test_lists(cells, drop):
    """10,976, 11,264, 11,265, 13,500 and 16,384 sites."""
    s = W.perturb(W.config_vacancy_lattice(cells), 0.05, 0.02, seed=12)
    keep = s.n - drop
    s.q, s.sigma, s.x = s.q[:, :keep].copy(), s.sigma[:keep].copy(), s.x[:, :keep].copy()
    s.T, s.sublattice = s.T[:keep].copy(), s.sublattice[:keep].copy()
    g = M.MxeSystem(s, "ff")
    for _ in range(2):
        g.build_neighbors()
        st, ro, ri = O.neighbors(s.q, s.L, g.r_list)
        assert st == O.OK
        off, idx = (t.cpu().numpy() for t in g.export_neighbors())
        np.testing.assert_array_equal(off, ro)
        np.testing.assert_array_equal(idx, ri)
        bro, bri = O.bonds(s, g.r_bond, ro, ri)
        boff, bidx = (t.cpu().numpy() for t in g.export_bonds())
        np.testing.assert_array_equal(boff, bro)
        np.testing.assert_array_equal(bidx, bri)
