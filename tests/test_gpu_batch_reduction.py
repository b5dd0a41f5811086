"""Per-system FIRE sums of a batch (csrc/relax.cu) where a system has several
blocks, and unevenly many: no site, 256 sites (one block), 1,372 and 2,048 (two),
5,324 (six).

Against the oracle and against the system alone at the tolerances of the other
relaxation tests.  A system's sums do not depend on the rest of the batch: its
lists, grid and site order are the same in a batch of the same systems in
another order, so the results are equal to the bit.
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


def systems():
    out = []
    for k, c in enumerate((4, 11, 0, 7, 8)):
        s = W.config_vacancy_lattice(max(c, 4), pot=W.potential_variant_s())
        s.x[:] = 0.99
        s = W.perturb(s, 0.02 + 0.01 * k, 0.02, seed=60 + k)
        if c == 0:
            s.q, s.sigma, s.x, s.T = s.q[:, :0], s.sigma[:0], s.x[:, :0], s.T[:0]
            s.sublattice = s.sublattice[:0]
        out.append(s)
    return out


def relaxed(order, K, precision):
    every = systems()
    g = M.MxeBatch([every[b] for b in order], precision)
    g.build_neighbors()
    st, it, _ = g.relax(0.0, K)
    assert st == M.ERR_NO_CONVERGE and it == K
    _, fmax, _ = g.relax_info()
    got = {b: (g.part(g.q, t).cpu().numpy(), g.part(g.sigma, t).cpu().numpy(), fmax[t]) for t, b in enumerate(order)}
    g.close()
    return got


def test_iterations_against_the_oracle():
    K = 12
    got = relaxed([0, 1, 2, 3, 4], K, "fp64")
    for b, s in enumerate(systems()):
        if s.n == 0:
            continue
        st, it, fm, q, sigma = O.relax(s, 0.0, K)
        assert st == O.ERR_NO_CONVERGE and it == K
        np.testing.assert_allclose(got[b][0], q, rtol=0, atol=1e-9)
        np.testing.assert_allclose(got[b][1], sigma, rtol=0, atol=1e-9)
        assert abs(got[b][2] - fm) <= 1e-8


@pytest.mark.parametrize("precision", ["fp64", "mixed", "ff"])
def test_the_rest_of_the_batch_does_not_matter(precision):
    a, b = relaxed([0, 1, 2, 3, 4], 20, precision), relaxed([4, 3, 1, 2, 0], 20, precision)
    for k in range(5):
        np.testing.assert_array_equal(a[k][0], b[k][0])
        np.testing.assert_array_equal(a[k][1], b[k][1])
        assert a[k][2] == b[k][2]


def test_graph_run_against_each_system_alone():
    every = [s for s in systems() if s.n]
    steps, dt, K = 2, 1e-3 * min(s.dt_default() for s in every), 6
    g = M.MxeBatch(every, "fp64")
    g.build_neighbors()
    g.run_staggered(steps, dt, 0.0, K)
    for b, s in enumerate(every):
        h = M.MxeSystem(s, "fp64")
        h.build_neighbors()
        h.run_staggered(steps, dt, 0.0, K)
        assert (g.part(g.x, b) - h.x).abs().max().item() <= 1e-12
        assert (g.part(g.q, b) - h.q).abs().max().item() <= 1e-9
        assert (g.part(g.sigma, b) - h.sigma).abs().max().item() <= 1e-9
        h.close()
    g.close()
