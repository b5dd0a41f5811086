"""FP64 force pass: constant terms times the pair's weights in integers on one
grid per pair (csrc/pair_table.cu), against the oracle where the grid can go
wrong: species that are absent (zero weights) or nearly so, weights of very
different size, scaled potentials (the grid's exponent moves with them), and
cut-offs just beyond the nearest node of a neighbour shell, whose row's constant
term vanishes while its linear and quadratic terms do not.

Tolerance: every product is exact to 2^-55 of the largest term of its pair and
the table to 2^-52, the sums cancel by at most a factor ~100: 1e-11 of the
largest component, as for the other FP64 passes.
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

TOL = 1e-11


def alloy(cells=4, seed=21):
    return W.perturb(W.config_binary_alloy(cells), 0.05, 0.02, seed=seed)


def pure_sites():
    s = alloy()
    one = (np.arange(s.n) % 3 == 0).astype(float)
    s.x[0], s.x[1] = one, 1.0 - one
    return s


def traces():
    s = alloy()
    s.x[0] = 10.0 ** -(np.arange(s.n) % 40).astype(float) * 0.5
    s.x[1] = 1.0 - s.x[0]
    return s


def scaled(factor):
    s = alloy()
    s.pot.phi_A[:] *= factor
    s.pot.E[:] *= factor
    s.T[:] *= factor
    return s


def edge(gap):
    """r_cut^2 = the nearest node of the third shell pairs + gap (unperturbed)."""
    s = W.config_binary_alloy(4)
    d = s.q - s.q[:, :1]
    d -= s.L[:, None] * np.rint(d / s.L[:, None])
    r2 = np.unique(np.round((d * d).sum(0), 9))
    j = np.argmin(np.abs((d * d).sum(0) - r2[3]))
    sh = np.sqrt(6.0) * s.sigma[j]
    near = r2[3] + sh * sh - 2.0 * sh * np.abs(d[:, j]).max()
    s.pot.r_cut = float(np.sqrt(near + gap))
    s.pot.r_switch = s.pot.r_cut - 0.8
    return s


CASES = {"pure_sites": pure_sites, "traces": traces}
CASES.update({f"scaled_{e}": (lambda e=e: scaled(10.0 ** e)) for e in (-12, -6, 6, 12)})
CASES.update({f"edge_{g:g}": (lambda g=g: edge(g)) for g in (-1e-3, 1e-9, 1e-6, 1e-3, 1 / 64, 1 / 32)})


@pytest.mark.parametrize("name", list(CASES))
def test_forces(name):
    s = CASES[name]()
    g = M.MxeSystem(s, "fp64", skin=0.2)
    g.build_neighbors()
    g.free_energy_grad()
    st, offs, idx = O.neighbors(s.q, s.L, g.r_list)
    fe = O.free_energy(s, (offs, idx))
    assert st == O.OK and fe["status"] == O.OK
    for k in ("gs", "gq"):
        a, b = getattr(g, k).cpu().numpy(), np.asarray(fe[k])
        # an ideal lattice's forces cancel to rounding: on the scale of gs
        scale = max(np.abs(b).max(), np.abs(np.asarray(fe["gs"])).max())
        assert np.abs(a - b).max() <= TOL * scale
