"""List builds when the device's memory runs out (csrc/api.cu): the status, and
the context afterwards.  Another allocation takes all but a given rest of the
free memory meanwhile.
"""
import numpy as np
import pytest

from paper_1910_01235_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1910_01235_gb300 import mxe as M  # noqa: E402


class AllBut:
    def __init__(self, rest):
        self.rest = rest

    def __enter__(self):
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        free = torch.cuda.mem_get_info()[0]
        self.held = torch.empty(max(free - self.rest, 0), dtype=torch.uint8, device="cuda")

    def __exit__(self, *exc):
        self.held = None
        torch.cuda.empty_cache()


def evaluate(g):
    g.build_neighbors()
    g.free_energy_grad()
    return [t.clone() for t in (g.F4, g.gq, g.gs, g.mu_ex)]


@pytest.mark.parametrize("rest_mb", [20, 100, 250, 600])
@pytest.mark.parametrize("precision", ["fp64", "ff"])
def test_a_list_that_does_not_fit(precision, rest_mb):
    """A wider list fails in one allocation or another of its growth; the narrow
    one is then built again, with the same results."""
    s = W.perturb(W.config_vacancy_lattice(30), 0.05, 0.02, seed=5)
    g = M.MxeSystem(s, precision)
    narrow = g.skin
    before = evaluate(g)
    with AllBut(rest_mb << 20):
        g.skin = narrow + 3.0
        with pytest.raises(M.MxeError) as e:
            g.build_neighbors()
        assert e.value.status == M.ERR_OOM
        g.skin = narrow
    for a, b in zip(evaluate(g), before):
        assert np.abs((a - b).cpu().numpy()).max() <= 1e-12 * np.abs(b.cpu().numpy()).max()


@pytest.mark.parametrize("precision", ["fp64", "ff"])
def test_a_rebuild_without_room_for_its_rows(precision):
    """The second build of a context fills rows of a fixed stride (29 MB or more
    here); without room for them it counts and fills, as the first."""
    s = W.perturb(W.config_vacancy_lattice(30), 0.05, 0.02, seed=6)
    g = M.MxeSystem(s, precision)
    before = evaluate(g)
    with AllBut(16 << 20):
        g.build_neighbors()
    g.free_energy_grad()
    for a, b in zip((g.F4, g.gq, g.gs, g.mu_ex), before):
        assert np.abs((a - b).cpu().numpy()).max() <= 1e-12 * np.abs(b.cpu().numpy()).max()


def used():
    torch.cuda.synchronize()
    free, total = torch.cuda.mem_get_info()
    return total - free


@pytest.mark.parametrize("case,extra", [("alloy", 4), ("single", 6)])
def test_memory_of_the_first_tangent(case, extra):
    """The first forward-mode pass of a context allocates `extra` doubles per list
    entry (an eighth more for growth), six per site and species, and its rows and
    sums (6 MB at most, with the allocator's granularity): the rest of its records
    lies in the geometry records' buffer."""
    s = W.perturb(W.config_binary_alloy(20) if case == "alloy" else W.config_vacancy_lattice(24), 0.05, 0.02, seed=7)
    g = M.MxeSystem(s, "fp64")
    g.build_neighbors()
    g.free_energy_grad()
    few = W.config_binary_alloy(4) if case == "alloy" else W.config_vacancy_lattice(5)
    small = M.MxeSystem(W.perturb(few, 0.05, 0.02, seed=8), "fp64")
    small.build_neighbors()
    small.tangent()  # the kernels are loaded
    held = torch.empty(256 << 20, dtype=torch.uint8, device="cuda")
    del held  # the outputs come from torch's pool
    before = used()
    t = g.tangent()
    assert used() - before <= 1.125 * 8 * extra * g.n_pairs + 48 * s.S * s.n + (6 << 20)
    assert (t["gq"] - g.gq).abs().max().item() <= 1e-11 * g.gq.abs().max().item()


@pytest.mark.parametrize("rest_mb", [4, 65])
def test_arrays_of_a_first_use_that_do_not_fit(rest_mb):
    """864,000 sites: the exact embedding average takes 62 + 3 MB, the tangents 41 + 0.1 MB."""
    s = W.perturb(W.config_vacancy_lattice(60), 0.05, 0.02, seed=9)
    g = M.MxeSystem(s, "fp64")
    before = evaluate(g)
    out = g.tangent  # bound before the memory is gone
    with AllBut(rest_mb << 20):
        with pytest.raises(M.MxeError) as e:
            g.set_embedding("exact")
        assert e.value.status == M.ERR_OOM
        with pytest.raises((M.MxeError, torch.cuda.OutOfMemoryError)):
            out()
    t = out()
    assert (t["gq"] - before[1]).abs().max().item() <= 1e-11 * before[1].abs().max().item()
    g.set_embedding("exact")
    g.free_energy_grad()
    assert torch.isfinite(g.gq).all().item()
