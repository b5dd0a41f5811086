"""The tabulated pair passes (csrc/radial_table.cuh, csrc/pair_table.cu) against
the oracle where they can go wrong: one and two species with every slot count
of the table, tables whose density depends on both species, pairs with a node
below the first row and pairs beyond 8 A (both take the direct evaluation), a
potential outside the table's limits (direct kernels), cut-offs that do not
fall on an interval boundary, and a ragged number of pairs.

Tolerances: FP64 contexts and the float-float quantities (mu, energies) carry
a relative error of at most 2^-46 per pair term (float-float rows: 6e-14
truncation and rounding); the sums cancel by at most a factor ~30 here, so
1e-11 of the largest component bounds them; FP64 gradients and relaxed states
are held to 1e-11 as well (per-term errors near 1e-15).
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


def single():
    return W.perturb(W.config_vacancy_lattice(4), 0.05, 0.02), 0.2


def binary():
    return W.perturb(W.config_binary_alloy(5), 0.05, 0.02), 0.2


def slab():  # four terms: no solute-solute interaction
    return W.config_interstitial_slab(4, 4, 4, top=100.0, xmax=0.3), 0.2


def asymmetric():  # general tables: one density term for both species, its own cross pair
    s = W.perturb(W.config_binary_alloy(4), 0.05, 0.02, seed=11)
    P = W.potential_binary()
    P.cross_geomean = False
    P.phi_A[0, 1] = P.phi_A[1, 0] = 0.2
    P.phi_p[0, 1] = P.phi_p[1, 0] = 4.0
    P.phi_r0[0, 1] = P.phi_r0[1, 0] = 2.5
    P.f_q[:] = 5.0
    P.f_xi[:] = 1.0
    P.f_r0[:] = 2.55
    s.pot = P
    return s, 0.2


def ragged_cut():  # breakpoints inside intervals
    s = W.perturb(W.config_binary_alloy(4), 0.05, 0.02, seed=5)
    s.pot.r_switch, s.pot.r_cut = 4.1234, 4.7891
    return s, 0.2


def close():  # two sites 1.5 A apart: nodes at 1.2 A, below the first row (1.25 A)
    s = W.perturb(W.config_binary_alloy(4), 0.02, 0.01, seed=6)
    s.q[:, 1] = s.q[:, 0] + np.array([1.5, 0.05, 0.02])
    return s, 0.2


def far():  # list entries beyond 8 A
    return W.perturb(W.config_vacancy_lattice(5), 0.05, 0.02, seed=7), 3.3


def steep():  # decay rates above the table's limit
    s = W.perturb(W.config_binary_alloy(4), 0.02, 0.01, seed=8)
    s.pot.phi_p[:] = np.where(s.pot.phi_p != 0, 9.0, 0.0)
    return s, 0.2


CASES = {f.__name__: f for f in (single, binary, slab, asymmetric, ragged_cut, close, far, steep)}


def off(a, b):
    a, b = a.cpu().numpy(), np.asarray(b)
    return np.abs(a - b).max() / max(np.abs(b).max(), 1e-300)


@pytest.mark.parametrize("name", list(CASES))
@pytest.mark.parametrize("precision", ["fp64", "mixed", "ff"])
def test_evaluation(name, precision):
    s, skin = CASES[name]()
    g = M.MxeSystem(s, precision, skin=skin)
    g.build_neighbors()
    g.free_energy_grad()
    st, offs, idx = O.neighbors(s.q, s.L, g.r_list)
    fe = O.free_energy(s, (offs, idx))
    assert st == O.OK and fe["status"] == O.OK
    assert off(g.F4, fe["F4"]) <= TOL
    assert off(g.mu_ex, fe["mu_ex"]) <= TOL
    assert off(g.mu, fe["mu"]) <= TOL
    # the FP32 modes' forces carry FP32 node arithmetic (1e-7 per term, FP32
    # positions): 1e-4 of the largest component
    gtol = TOL if precision == "fp64" else 1e-4
    assert off(g.gq, fe["gq"]) <= gtol
    assert off(g.gs, fe["gs"]) <= gtol


@pytest.mark.parametrize("name", ["single", "binary", "slab", "asymmetric", "ragged_cut", "close", "far", "steep"])
def test_relaxation_passes_fp64(name):
    """Three FIRE updates: the tabulated density and force passes of FP64
    contexts (each update moves y by dt v, so a relative force error e gives
    about e of the displacement)."""
    s, skin = CASES[name]()
    g = M.MxeSystem(s, "fp64", skin=skin)
    g.build_neighbors()
    fire = M.make_fire(dt0=1e-3)
    g.relax(0.0, 3, fire)
    st, it, fm, q, sg = O.relax(s, 0.0, 3, O.FireParams(dt0=1e-3), skin=skin)
    dq, dqo = g.q.cpu().numpy() - s.q, q - s.q
    ds, dso = g.sigma.cpu().numpy() - s.sigma, sg - s.sigma
    # differences of absolute positions: 1e-16 x 18 A of rounding on top
    assert np.abs(dq - dqo).max() <= TOL * np.abs(dqo).max() + 1e-14
    assert np.abs(ds - dso).max() <= TOL * np.abs(dso).max() + 1e-14


def test_geometry_status_below_half_angstrom():
    """A node closer than 0.5 A is reported from the tabulated pass as before."""
    s = W.config_binary_alloy(4)
    s.q[:, 1] = s.q[:, 0] + np.array([0.6, 0.0, 0.0])
    for precision in ("fp64", "ff"):
        g = M.MxeSystem(s, precision)
        g.build_neighbors()
        with pytest.raises(M.MxeError) as e:
            g.free_energy_grad()
        assert e.value.status == M.ERR_GEOMETRY


@pytest.mark.parametrize("name", ["single", "binary", "slab", "asymmetric", "ragged_cut", "close"])
def test_tangent_pairs(name):
    """Hessian products of the pair-wise tangent passes against central
    differences of the oracle's gradients (step 1e-5 along a unit-size
    direction: truncation ~h^2 |third derivative| ~1e-8 relative, rounding
    ~1e-16 / h ~1e-11: 1e-6 of the largest component bounds both), the values
    against the oracle, and the Hessian-only form against the full one (the
    same sums in another order: 1e-12)."""
    s, skin = CASES[name]()
    g = M.MxeSystem(s, "fp64", skin=skin)
    g.build_neighbors()
    rng = np.random.default_rng(3)
    dq, ds, dx = rng.normal(size=s.q.shape), rng.normal(size=s.n) * 0.3, rng.normal(size=s.x.shape) * 0.01
    d = [torch.as_tensor(v, dtype=torch.float64, device="cuda") for v in (dq, ds, dx)]
    out = g.tangent(*d)
    st, offs, idx = O.neighbors(s.q, s.L, g.r_list)
    fe = O.free_energy(s, (offs, idx))
    for k in ("gq", "gs", "mu_ex"):
        assert off(out[k], fe[k]) <= TOL
    h, lo_hi = 1e-5, []
    for sign in (1.0, -1.0):
        t = s.copy()
        t.q, t.sigma, t.x = s.q + sign * h * dq, s.sigma + sign * h * ds, s.x + sign * h * dx
        lo_hi.append(O.free_energy(t, (offs, idx)))
    for k in ("gq", "gs", "mu_ex"):
        assert off(out[k + "_t"], (lo_hi[0][k] - lo_hi[1][k]) / (2 * h)) <= 1e-6
    # Hessian products alone
    gq_t, gs_t = torch.zeros_like(out["gq_t"]), torch.zeros_like(out["gs_t"])
    ptr = [M._ptr(v) for v in d]
    assert M.mxe_tangent(g.ctx, g.state, *ptr, 0, 0, 0, M._ptr(gq_t), M._ptr(gs_t), 0, 0) == M.OK
    assert off(gq_t, out["gq_t"].cpu().numpy()) <= 1e-12
    assert off(gs_t, out["gs_t"].cpu().numpy()) <= 1e-12
