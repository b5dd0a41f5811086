"""CPU check of the home-frame error band of the cell-staged neighbour kernels
(grids of >= 3 cells per axis), which is built from the cell width alone:
wherever the FP32 test decides outside that band, it agrees with the FP64 rule.
Float32 arithmetic in the kernels' operation order (helpers of
test_neighbor_band); pairs from 1e-9 to 1e-4 relative of the cutoff, across the
band's edge (~3e-6 relative), in boxes up to 10,000 A and positions several
boxes outside."""
import numpy as np
import pytest

from test_neighbor_band import U, fp32_r2, fp64_r2


def home_band(qmax, L, h, r_list):
    d = 8.0 * U * h + 2.0 ** -50 * (qmax + L)
    return np.float32(2.0 * (2.0 * np.sqrt(3.0) * r_list * d + 3.0 * d * d + 4.0 * U * r_list * r_list) * (1.0 + 1e-6))


@pytest.mark.parametrize("L,r_list,boxes", [(144.0, 5.5, 0), (360.0, 6.1, 0), (18.0, 5.6, 1), (17.0, 5.6, 40),
                                            (10_000.0, 5.5, 3)])
def test_decisions_outside_the_home_band_match_fp64(L, r_list, boxes):
    rng = np.random.default_rng(5)
    nc = int(np.floor(L / (r_list * (1.0 + 1e-9))))
    m = 400_000
    qi = rng.uniform(0.0, L, (m, 3)) + L * rng.integers(-boxes, boxes + 1, (m, 3))
    v = rng.normal(size=(m, 3))
    v /= np.linalg.norm(v, axis=1, keepdims=True)
    eps = np.exp(rng.uniform(np.log(1e-9), np.log(1e-4), m)) * rng.choice([-1.0, 1.0], m)
    qj = qi + (r_list * (1.0 + eps))[:, None] * v + L * rng.integers(-1, 2, (m, 3))
    qmax = max(np.abs(qi).max(), np.abs(qj).max())
    band = home_band(qmax, L, L / nc, r_list)
    cut = np.float32(r_list * r_list)
    r2f, staged = fp32_r2(qi, qj, L, nc)
    exact_in = fp64_r2(qi, qj, L) < r_list * r_list
    assert not np.any(exact_in & ~staged)
    says_in, says_out = r2f < np.float32(cut - band), r2f > np.float32(cut + band)
    assert not np.any(says_in & ~exact_in)
    assert not np.any(says_out & exact_in)
    undecided = ~(says_in | says_out)
    assert says_in.any() and says_out.any() and undecided.any()
    assert np.abs(eps[undecided]).max() < 1e-5
