"""Failure reports of every kernel family by itself: the FP64 kernel that holds
a matrix in shared memory (contours of up to 20 rows, and the entry point with
static scratch up to 112), and the bounded waits of the FP64 tensor-core kernels,
the impurity step's and the network's.

As in test_failure_gpu.py the waits run out by the library's own limit (0 gives
up on the first wait that is not already satisfied); nothing traps, faults or
hangs, and the same call under the default limit is right again.
"""

import ctypes

import numpy as np
import pytest
import torch

from oracle import mlp_oracle as M
from oracle import nedmft_oracle as O
from paper_0711_0999_gb300 import _native as N
from paper_0711_0999_gb300 import api, warmstart
from paper_0711_0999_gb300.build import build_library
from paper_0711_0999_gb300.synth import workload_sigma

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    build_library()
    yield
    api.set_wait_limit(2.0)


def status():
    try:
        api.check_status()
        return N.NEDMFT_OK
    except N.NedmftError as e:
        return e.code


def contour(n):
    """Grid arguments of a contour of n points."""
    n_tau = 4 + n % 2 if n < 40 else 10 + n % 2
    return (-1.0, -1.0 + 0.125 * ((n - n_tau) // 2), 0.125, 0.25 * n_tau, 0.25)


def rel(a, b):
    return float(np.abs(a - b).max() / np.abs(b).max())


def lattice(n, sig, pts, static):
    """G_loc of the FP64 lattice step, through the workspace or the static-scratch entry point."""
    g, mod = api.contour_grid(*contour(n)), api.make_model(1.0, 1.0)
    assert g.n_c == n
    d = [torch.as_tensor(np.ascontiguousarray(a), device="cuda") for a in (sig, *pts)]
    if not static:
        return api.lattice_gloc(g, mod, *d)[0]
    gl = torch.empty((n, n), dtype=torch.complex128, device="cuda")
    P = lambda t: ctypes.c_void_p(t.data_ptr())
    N.check(N.lib().nedmft_lattice_gloc_static(ctypes.byref(g.contour), ctypes.byref(mod), *[P(t) for t in d],
                                               d[1].numel(), P(gl), None, None, None))
    return gl


def solved_as_before(n, static, seed=3):
    c = O.contour_grid(*contour(n))
    sig, pts = workload_sigma(c.t, c.w, 1.0, seed=seed), O.quadrature_points(3)
    ref, _ = O.lattice_gloc(c, O.Model(U=1.0, E=1.0), sig, *pts)
    gl = lattice(n, sig, pts, static)
    torch.cuda.synchronize()
    return status() == N.NEDMFT_OK and rel(gl.cpu().numpy(), ref) < 1e-10


# in shared memory: both entry points at their largest sizes, and small
SHARED = [(12, False), (20, False), (20, True), (80, True), (112, True)]


@pytest.mark.parametrize("n,static", SHARED)
def test_shared_memory_kernel_reports_a_singular_matrix(n, static):
    c = O.contour_grid(*contour(n))
    b = np.linalg.inv(O.g0_matrix(c, O.Model(U=1.0, E=1.0), 0.0, 0.0))  # B_q - S is zero
    lattice(n, b / (c.w[:, None] * c.w[None, :]), O.quadrature_points(1), static)
    assert status() == N.NEDMFT_ESINGULAR
    assert solved_as_before(n, static)


@pytest.mark.parametrize("n,static", SHARED)
def test_shared_memory_kernel_reports_a_non_finite_sigma(n, static):
    c = O.contour_grid(*contour(n))
    sig = workload_sigma(c.t, c.w, 1.0, seed=6)
    sig[n // 3, n // 2] = np.nan
    lattice(n, sig, O.quadrature_points(3), static)
    assert status() == N.NEDMFT_ESINGULAR
    assert solved_as_before(n, static)


@pytest.mark.parametrize("n", [21, 80, 220])
def test_expired_waits_of_the_fp64_lattice_step(n):
    c = O.contour_grid(*contour(n))
    api.set_wait_limit(0.0)
    try:
        lattice(n, workload_sigma(c.t, c.w, 1.0, seed=5), O.quadrature_points(3), False)
        assert status() == N.NEDMFT_ETIMEOUT
    finally:
        api.set_wait_limit(2.0)
    assert solved_as_before(n, False)


@pytest.mark.parametrize("n", [33, 300])
def test_expired_waits_of_the_impurity_step(n):
    args = contour(n)
    c, g, mod = O.contour_grid(*args), api.contour_grid(*args), api.make_model(1.0, 1.0)
    sig = workload_sigma(c.t, c.w, 1.0, seed=5)
    gl, _ = O.lattice_gloc(c, O.Model(U=1.0, E=1.0), sig, *O.quadrature_points(2))
    gd, sd = (torch.as_tensor(a, device="cuda") for a in (gl, sig))
    api.set_wait_limit(0.0)
    try:
        api.impurity_update(g, mod, gd, sd)
        assert status() == N.NEDMFT_ETIMEOUT
    finally:
        api.set_wait_limit(2.0)
    ref, _ = O.impurity_update(c, O.Model(U=1.0, E=1.0), gl, sig)
    new, _ = api.impurity_update(g, mod, gd, sd)
    torch.cuda.synchronize()
    assert status() == N.NEDMFT_OK
    sw = lambda s: c.w[:, None] * s * c.w[None, :]
    assert rel(sw(new.cpu().numpy()), sw(ref)) < 1e-10


# one tile, and more tiles than SMs (the variant with two blocks per SM)
@pytest.mark.parametrize("n", [100, 20001])
def test_expired_waits_of_the_network(n):
    p = warmstart.init_params(3)
    rng = np.random.default_rng(n)
    x, t = rng.normal(size=(n, 17)).astype(np.float32), rng.normal(size=(n, 2)).astype(np.float32)
    dev = [torch.as_tensor(a, device="cuda") for a in (p, x, t)]
    api.set_wait_limit(0.0)
    try:
        warmstart.forward(dev[0], dev[1])
        assert status() == N.NEDMFT_ETIMEOUT
        warmstart.loss_and_grad(*dev)
        assert status() == N.NEDMFT_ETIMEOUT
    finally:
        api.set_wait_limit(2.0)
    y = warmstart.forward(dev[0], dev[1]).cpu().numpy()
    loss, grad = warmstart.loss_and_grad(*dev)
    grad = grad.cpu().numpy().astype(np.float64)
    assert status() == N.NEDMFT_OK
    yr, _ = M.forward(p, x, rounded=True)
    lr, gr = M.loss_and_grad(p, x, t, rounded=True)
    assert np.abs(y - yr).max() < 2e-2 * np.abs(yr).max()
    assert abs(loss.item() - lr) < 1e-4 * abs(lr)
    assert np.linalg.norm(grad - gr) < 2e-2 * np.linalg.norm(gr)
