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


# sizes whose default batch lies above, between and below the fixed candidates
@pytest.mark.parametrize("n_t,nq,prec", [(100, 1024, "fp64"), (190, 1500, "fp64"), (30, 700, "mixed_bf16"),
                                         (190, 1024, "mixed_bf16"), (1000, 2000, "mixed_bf16"), (30, 9, "fp64")])
def test_autotuner_times_the_batch_in_use(n_t, nq, prec):
    g = contour(n_t)
    assert api.lattice_batch(g, nq, prec) in api.autotune_candidates(g, nq, prec)
    api.lattice_set_tuning(g, nq, prec, batch=min(nq, 61))
    try:
        assert api.lattice_batch(g, nq, prec) == min(nq, 61)
        assert min(nq, 61) in api.autotune_candidates(g, nq, prec)
    finally:
        api.lattice_set_tuning(g, nq, prec)
