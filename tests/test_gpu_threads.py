"""List builds of two contexts in two threads, each on its own stream: few and many
candidates a cell, so that the fills ask for different amounts of shared memory."""
import threading
import time

import numpy as np
import pytest

from paper_1910_01235_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1910_01235_gb300 import mxe as M  # noqa: E402


def lists(g):
    with torch.cuda.stream(g.stream):
        out = [t.cpu().numpy() for t in g.export_neighbors()]
    torch.cuda.synchronize()
    return out


def test_two_threads_build_lists():
    contexts, first = [], []
    for cells, rc in ((8, 3.2), (20, 6.8)):  # both above two cells per SM: the same kernel
        s = W.perturb(W.config_vacancy_lattice(cells), 0.03, 0.0, seed=17)
        s.pot.r_switch, s.pot.r_cut = rc - 0.5, rc
        g = M.MxeSystem(s, "ff", stream=torch.cuda.Stream())
        torch.cuda.synchronize()
        g.build_neighbors()
        contexts.append(g)
        first.append(lists(g))
    failed, end = [], time.monotonic() + 3.0

    def builds(g):
        try:
            while time.monotonic() < end:
                g.build_neighbors()
        except Exception as e:  # noqa: BLE001
            failed.append(e)

    threads = [threading.Thread(target=builds, args=(g,)) for g in contexts]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed, failed
    for g, old in zip(contexts, first):
        for a, b in zip(lists(g), old):
            np.testing.assert_array_equal(a, b)
