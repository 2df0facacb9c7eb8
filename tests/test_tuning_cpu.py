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


# 16 bytes an entry, 152 matrices of up to the next multiple of 128 rows, and a tenth for the operands
@pytest.mark.parametrize("n_t,rows", [(700, 1536), (1650, 3456)])
def test_fp64_workspace_of_long_contours(n_t, rows):
    assert api.lattice_workspace_size(contour(n_t, 100), 2809, "fp64") <= 1.1 * 16 * rows**2 * 152
