"""Host side of the batch choice (no GPU needed)."""

import pytest

from paper_0711_0999_gb300 import api
from paper_0711_0999_gb300.build import build_library


@pytest.fixture(scope="module", autouse=True)
def built():
    build_library()


def contour(n_t, n_tau=20):
    return api.contour_grid(0.0, 0.1 * n_t, 0.1, 10.0, 10.0 / n_tau)


def test_fp64_batches_fit_one_launch():
    g = contour(30)
    nq = 200000
    assert api.lattice_workspace_size(g, nq, "fp64", batch=nq) == api.lattice_workspace_size(g, nq, "fp64", batch=65535)
    api.lattice_set_tuning(g, nq, "fp64", batch=nq)
    try:
        assert api.lattice_batch(g, nq, "fp64") == 65535
    finally:
        api.lattice_set_tuning(g, nq, "fp64")
