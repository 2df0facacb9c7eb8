"""Singular inputs of the FP64 lattice step and of the impurity step report
ESINGULAR: a pivot of at most 1e-12 counts as zero, also where a later 32-column
block, its Schur complement, is nothing but rounding noise (which has an inverse
like any other matrix), or where only a leading minor of a block vanishes.
Matrices a good way above that threshold are solved as before.
"""

import numpy as np
import pytest
import torch

from oracle import nedmft_oracle as O
from paper_0711_0999_gb300 import _native as N
from paper_0711_0999_gb300 import api
from paper_0711_0999_gb300.build import build_library

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    build_library()


def contour(n):
    """Grid arguments of a contour of n points."""
    n_tau = 4 + n % 2 if n < 40 else 10 + n % 2
    return (-1.0, -1.0 + 0.125 * ((n - n_tau) // 2), 0.125, 0.25 * n_tau, 0.25)


def noise(rng, *shape):
    return rng.standard_normal(shape) + 1j * rng.standard_normal(shape)


def last_block(n, r, scale):
    """n x n, its leading r x r block well conditioned in any order, the Schur complement of that scale."""
    rng = np.random.default_rng(n)
    m = 1j * np.eye(n) + 0.3 * noise(rng, n, n) / np.sqrt(n)
    m[r:, r:] = m[r:, :r] @ np.linalg.solve(m[:r, :r], m[:r, r:]) + scale * m[r:, r:]
    return m


def leading_minor(seed, n=32):
    """n x n, well conditioned, one leading minor zero (a pivot vanishes in the elimination in order)."""
    rng = np.random.default_rng(seed)
    c = lambda *s: noise(rng, *s)
    k = rng.integers(4, n - 4)
    g = 10 ** rng.uniform(-3, 0.5)
    m = c(n, n) / 8 + 2j * g * np.eye(n)
    m[k, k] = m[k, :k] @ np.linalg.solve(m[:k, :k], m[:k, k])
    return m


def status():
    try:
        api.check_status()
        return N.NEDMFT_OK
    except N.NedmftError as e:
        return e.code


def lattice_of(m):
    """The lattice step whose one matrix B_q - S is m: a point with eps > mu, hence in the contour's row order."""
    n = len(m)
    args = contour(n)
    c, g = O.contour_grid(*args), api.contour_grid(*args)
    assert g.n_c == n
    b = np.linalg.inv(O.g0_matrix(c, O.Model(U=1.0, E=1.0), 1.0, 0.5))
    sig = (b - m) / (c.w[:, None] * c.w[None, :])
    api.lattice_gloc(g, api.make_model(1.0, 1.0), torch.as_tensor(sig, device="cuda"), np.array([1.0]), np.array([0.5]),
                     np.array([1.0]))


def impurity_of(m):
    g = api.contour_grid(*contour(len(m)))
    gl = torch.as_tensor(m, device="cuda")
    api.impurity_update(g, api.make_model(1.0, 1.0), gl, torch.zeros_like(gl))


RANKS = [(64, 32), (64, 63), (65, 64), (96, 64), (97, 96), (128, 96), (512, 480)]


@pytest.mark.parametrize("step", [lattice_of, impurity_of])
@pytest.mark.parametrize("n,r", RANKS)
def test_rank_deficient_matrix_reports_esingular(step, n, r):
    step(last_block(n, r, 0.0))
    assert status() == N.NEDMFT_ESINGULAR


# blocks whose FP32 elimination in order meets rounding noise of 1e-5 .. 1e-4 in the zero's place and gets by
@pytest.mark.parametrize("seed", [122, 156, 245, 287])
def test_vanishing_leading_minor_reports_esingular(seed):
    lattice_of(leading_minor(seed))
    assert status() == N.NEDMFT_ESINGULAR


# The smallest pivots about half the scale: 40 times the threshold, and far above it.  In the impurity step the
# scale is the least singular value of G_loc, and with it the ratio of the rows that its FP32 pivot choice tells
# apart: from 1e-10 on it depends on rounding which rows it takes.
@pytest.mark.parametrize("step,scale", [(lattice_of, 1e-10), (lattice_of, 1e-6), (lattice_of, 1e-3),
                                        (impurity_of, 1e-9), (impurity_of, 1e-6), (impurity_of, 1e-3)])
@pytest.mark.parametrize("n,r", RANKS)
def test_small_pivots_above_the_threshold_are_accepted(step, scale, n, r):
    step(last_block(n, r, scale))
    assert status() == N.NEDMFT_OK
