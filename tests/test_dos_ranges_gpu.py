"""The density of states at the ends of its ranges: more frequencies than one
launch takes along a grid's second dimension, frequencies whose phases carry no
information any more, and the numbers of relative times at which the kernel
changes its form."""

import numpy as np
import pytest
import torch

from oracle import nedmft_oracle as O
from paper_0711_0999_gb300 import api
from paper_0711_0999_gb300.build import build_library

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    build_library()


def setup(n_t, seed=4, dt=0.05):
    c, g = (f(0.0, dt * n_t, dt, 0.5, 0.25) for f in (O.contour_grid, api.contour_grid))
    rng = np.random.default_rng(seed)
    return c, g, rng.standard_normal((c.n_c, c.n_c)) + 1j * rng.standard_normal((c.n_c, c.n_c)), rng


def bound(c, gl, m, omega):
    """Rounding of both sums: one rounding per term and addition, and of the phases, 3 eps |omega| t."""
    k = min(m, c.n_t - 1 - m) + 1
    terms = 2 * c.dt * sum(abs(O.retarded(c, gl, m + i, m - i)) for i in range(k))
    return 2 * np.finfo(np.float64).eps * (k + 4 + 3 * np.abs(omega).max() * 2 * c.dt * k) * terms / np.pi


# up to 7 and up to 81 relative times
@pytest.mark.parametrize("n_t", [12, 161])
def test_more_frequencies_than_one_launch_takes(n_t):
    c, g, gl, rng = setup(n_t)
    omega = rng.uniform(-5.0, 5.0, 8 * 65535 + 1003)
    m_index = [n_t // 2 - 1, 0, n_t // 2, -1]
    rho = api.dos(g, torch.as_tensor(gl, device="cuda"), m_index, omega).cpu().numpy()
    for row, m in enumerate(m_index[:3]):
        assert np.abs(rho[row] - O.dos(c, gl, m, omega)).max() <= bound(c, gl, m, omega)
    assert np.isnan(rho[3]).all()


# phases far beyond 2^53: any value of a phase is as good as another, but it is a phase
@pytest.mark.parametrize("n_t", [21, 301, 2301])
def test_huge_frequencies_stay_within_the_sum_of_the_terms(n_t):
    c, g, gl, _ = setup(n_t)
    omega = np.array([1e10, -1e15, 3e18, 1e22, -1e100, 1e300])
    m = n_t // 2
    rho = api.dos(g, torch.as_tensor(gl, device="cuda"), [m], omega).cpu().numpy()[0]
    k = min(m, n_t - 1 - m) + 1
    top = 2 * c.dt * sum(abs(O.retarded(c, gl, m + i, m - i)) for i in range(k)) / np.pi
    assert (np.abs(rho) <= top * (1 + 1e-12)).all()


# 1 to 65 relative times, with few frequencies and with enough for every SM
@pytest.mark.parametrize("n_omega", [1, 33, 700])
def test_numbers_of_relative_times(n_omega):
    c, g, gl, rng = setup(160)
    m_index = [0, 1, 2, 7, 8, 14, 15, 16, 17, 62, 63, 64, 65, 79, 80, 96, 159, 160]
    omega = rng.uniform(-5.0, 5.0, n_omega)
    rho = api.dos(g, torch.as_tensor(gl, device="cuda"), m_index, omega).cpu().numpy()
    for row, m in enumerate(m_index[:-1]):
        assert np.abs(rho[row] - O.dos(c, gl, m, omega)).max() <= bound(c, gl, m, omega), m
    assert np.isnan(rho[-1]).all()
