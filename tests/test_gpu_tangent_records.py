"""Tangent records across the geometry records' buffer and their own
(csrc/tangent_table.cu): each split that the precisions and potentials give (24,
32, 40 and 64 bytes an entry), before and after the lists grow.  Values against the
free-energy call of an FP64 context, tangents against central differences of its
gradients; the passes are FP64 in every context.
"""
import numpy as np
import pytest

from paper_1910_01235_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1910_01235_gb300 import mxe as M  # noqa: E402


def system(case):
    if case.startswith("single"):
        s = W.config_vacancy_lattice(5)
        if case == "single_density":
            s.pot.phi_A[:] = 0.0
    else:
        s = W.config_binary_alloy(5)
        if case == "alloy_no_cross":
            s.pot.cross_geomean = False
            s.pot.phi_A[0, 1] = s.pot.phi_A[1, 0] = 0.0
        if case == "alloy_one_density":
            for t in (s.pot.f_xi, s.pot.f_q, s.pot.f_r0):
                t[:] = t[0, 0]
    return W.perturb(s, 0.05, 0.02, seed=61)


@pytest.mark.parametrize("precision", ["fp64", "mixed", "ff"])
@pytest.mark.parametrize("case", ["single", "single_density", "alloy", "alloy_no_cross", "alloy_one_density"])
def test_tangents(case, precision):
    s = system(case)
    rng = np.random.default_rng(62)
    d = [torch.as_tensor(rng.normal(0.0, 1.0, n), device="cuda") for n in ((3, s.n), s.n, (s.S, s.n))]
    ref = M.MxeSystem(s, "fp64")
    ref.build_neighbors()
    ref.free_energy_grad()
    step = 2.0**-14
    want = {}
    for sg in (1.0, -1.0):  # central differences of the gradients
        h = M.MxeSystem(s, "fp64")
        for a, b in zip((h.q, h.sigma, h.x), d):
            a += sg * step * b * (1e-2 if b.shape == h.x.shape else 1.0)
        h.build_neighbors()
        h.free_energy_grad()
        for k in ("gq", "gs", "mu_ex"):
            want[k] = want.get(k, 0.0) + sg * getattr(h, k) / (2.0 * step)
        h.close()
    d[2] = 1e-2 * d[2]
    g = M.MxeSystem(s, precision)
    first = None
    for skin in (0.2, 0.2, 0.9):
        g.skin = skin
        g.build_neighbors()
        t = g.tangent(*d)
        for k in ("gq", "gs", "mu_ex"):
            assert (t[k] - getattr(ref, k)).abs().max().item() <= 1e-11 * getattr(ref, k).abs().max().item()
            # the differences: second order in the step, about 1e-6 of the largest
            assert (t[k + "_t"] - want[k]).abs().max().item() <= 1e-4 * want[k].abs().max().item()
        first = first or t
        for k in t:
            assert (t[k] - first[k]).abs().max().item() <= 1e-11 * first[k].abs().max().item()
