"""The kernels at the edges of their tiles and of the ranges that select them,
against the oracle (or the CPU restatement of the network).

Tolerances: the FP64 path's contract, 1e-10 relative in the maximum norm
(2e-10 between two kernels that each meet it); the mixed path's, 1e-6; the
network's, that of its gradient test (bf16 operands, FP32 sums in another
order); the density of states', the rounding bound of its sum, written out.
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


def rel(a, b):
    return float(np.abs(a - b).max() / np.abs(b).max())


def contour(n):
    """Grid arguments of a contour of n points."""
    n_tau = 4 + n % 2 if n < 40 else 10 + n % 2
    return (-1.0, -1.0 + 0.125 * ((n - n_tau) // 2), 0.125, 0.25 * n_tau, 0.25)


def points(nq, seed=2):
    """nq points with (eps - mu) of both signs, hence in both row orders, and positive weights."""
    rng = np.random.default_rng(seed)
    wq = rng.uniform(0.5, 1.0, nq)
    return rng.normal(0.25, 1.2, nq), rng.normal(0.0, 1.0, nq), wq / wq.sum()


def setup(n, nq, U=0.5, E=1.0):
    args = contour(n)
    c, g = O.contour_grid(*args), api.contour_grid(*args)
    assert c.n_c == n and g.n_c == n
    return c, g, O.Model(U=U, E=E), api.make_model(U, E), workload_sigma(c.t, c.w, U, seed=n), points(nq)


def lattice(g, mc, sig, eps, ebar, wq, prec="fp64"):
    gl, j, _ = api.lattice_gloc(g, mc, torch.as_tensor(sig, device="cuda"), eps, ebar, wq, precision=prec)
    torch.cuda.synchronize()
    api.check_status()
    return gl.cpu().numpy(), j.cpu().numpy()


# one 32-column step and its neighbours, the 64- and 128-row tiles, the padded sizes 256 and 512
@pytest.mark.parametrize("n,nq", [(19, 3), (20, 3), (21, 1), (21, 2), (32, 5), (33, 4), (64, 3), (65, 3), (96, 7), (127, 2),
                                  (128, 3), (129, 3), (160, 2), (255, 3), (256, 2), (257, 3), (513, 2)])
def test_fp64_lattice_tile_edges(n, nq):
    c, g, mo, mc, sig, (eps, ebar, wq) = setup(n, nq)
    ref, jref = O.lattice_gloc(c, mo, sig, eps, ebar, wq)
    gl, j = lattice(g, mc, sig, eps, ebar, wq)
    assert rel(gl, ref) < 1e-10
    assert np.abs(j - jref.real).max() < 1e-10


@pytest.mark.parametrize("nq", [1023, 1025, 2049])  # around one and two batches
def test_fp64_lattice_batch_edges(nq):
    c, g, mo, mc, sig, (eps, ebar, wq) = setup(24, nq)
    ref, jref = O.lattice_gloc(c, mo, sig, eps, ebar, wq)
    gl, j = lattice(g, mc, sig, eps, ebar, wq)
    assert rel(gl, ref) < 1e-10
    assert np.abs(j - jref.real).max() < 1e-10


# the sizes that both FP64 kernels take: blocked (workspace call) and in shared memory (static scratch)
@pytest.mark.parametrize("n", [20, 21, 40, 63, 96, 111, 112])
def test_fp64_blocked_kernel_agrees_with_the_shared_memory_kernel(n):
    c, g, mo, mc, sig, pts = setup(n, 37)
    gl, j = lattice(g, mc, sig, *pts)
    d = [torch.as_tensor(np.ascontiguousarray(a), device="cuda") for a in (sig, *pts)]
    gs = torch.empty((n, n), dtype=torch.complex128, device="cuda")
    js, ji = (torch.empty(c.n_t, dtype=torch.float64, device="cuda") for _ in range(2))
    P = lambda t: ctypes.c_void_p(t.data_ptr())
    N.check(N.lib().nedmft_lattice_gloc_static(ctypes.byref(g.contour), ctypes.byref(mc), P(d[0]), P(d[1]), P(d[2]), P(d[3]),
                                               37, P(gs), P(js), P(ji), ctypes.c_void_p(0)))
    torch.cuda.synchronize()
    api.check_status()
    assert rel(gl, gs.cpu().numpy()) < 2e-10
    assert np.abs(j - js.cpu().numpy()).max() < 2e-10


# S = W Sigma W with a diagonal from 1 to 10^decades in every 32 rows: dominant, so elimination in order
# is stable, but a block's FP32 inverse has to be corrected more often (or the FP64 elimination to take over)
@pytest.mark.parametrize("decades", [3, 9, 15])
@pytest.mark.parametrize("n", [33, 100])
def test_fp64_pivot_blocks_of_graded_rows(n, decades):
    c, g, mo, mc, sig, (eps, ebar, wq) = setup(n, 4)
    eps = 0.3 + np.abs(eps)  # eps > mu: the row order in which the large entries are the pivots
    sig = sig + np.diag(-4.0 * 10.0 ** (decades * (np.arange(n) % 32) / 31.0) / c.w**2)
    ref, jref = O.lattice_gloc(c, mo, sig, eps, ebar, wq)
    gl, j = lattice(g, mc, sig, eps, ebar, wq)
    assert rel(gl, ref) < 1e-10
    assert np.abs(j - jref.real).max() < 1e-10


# the pivot choice: fewer rows than a 32-column step, a last step of one column, the 256-row chunks of the
# tournament, five chunks (clusters of eight)
@pytest.mark.parametrize("n", [6, 31, 32, 33, 65, 255, 256, 257, 513, 1030])
def test_impurity_step_tile_edges(n):
    c, g, mo, mc, sig, _ = setup(n, 1, U=1.0)
    rng = np.random.default_rng(n)
    gl = np.roll(np.eye(n) + 0.3 * (rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))) / np.sqrt(n), 1, axis=0)
    np.fill_diagonal(gl, 0.0)  # an elimination without row exchanges meets a zero pivot at once
    s_ref, gi_ref = O.impurity_update(c, mo, gl, sig)
    s_new, gimp = api.impurity_update(g, mc, torch.as_tensor(gl, device="cuda"), torch.as_tensor(sig, device="cuda"),
                                      want_gimp=True)
    torch.cuda.synchronize()
    api.check_status()
    sw = lambda s: c.w[:, None] * s * c.w[None, :]
    assert rel(sw(s_new.cpu().numpy()), sw(s_ref)) < 1e-10
    assert rel(gimp.cpu().numpy(), gi_ref) < 1e-10


# one sample, around a 128-sample tile, and more tiles than SMs (the variant with two blocks per SM)
@pytest.mark.parametrize("n", [1, 127, 128, 129, 20001])
def test_network_tile_edges(n):
    p = warmstart.init_params(3)
    rng = np.random.default_rng(n)
    x, t = rng.normal(size=(n, 17)).astype(np.float32), rng.normal(size=(n, 2)).astype(np.float32)
    dev = [torch.as_tensor(a, device="cuda") for a in (p, x, t)]
    loss, grad = warmstart.loss_and_grad(*dev)
    grad = grad.cpu().numpy().astype(np.float64)
    lr, gr = M.loss_and_grad(p, x, t, rounded=True)
    assert abs(loss.item() - lr) < 1e-4 * abs(lr)
    assert np.linalg.norm(grad - gr) < 2e-2 * np.linalg.norm(gr)
    y = warmstart.forward(dev[0], dev[1]).cpu().numpy()
    yr, _ = M.forward(p, x, rounded=True)
    assert np.abs(y - yr).max() < 2e-2 * np.abs(yr).max()


# no, one, two relative times; 1024 and more of them
@pytest.mark.parametrize("n_t,m_index", [(41, [0, 1, 2, 20, 39, 40, -1, 41]), (2100, [1023, 1024, 1025, 1050])])
def test_dos_relative_times(n_t, m_index):
    c, g = (f(0.0, 0.02 * n_t, 0.02, 0.5, 0.25) for f in (O.contour_grid, api.contour_grid))
    rng = np.random.default_rng(n_t)
    gl = rng.standard_normal((c.n_c, c.n_c)) + 1j * rng.standard_normal((c.n_c, c.n_c))
    omega = np.array([-7.3, -1.0, 0.0, 0.4, 25.0])
    rho = api.dos(g, torch.as_tensor(gl, device="cuda"), m_index, omega).cpu().numpy()
    eps = np.finfo(np.float64).eps
    for row, m in enumerate(m_index):
        if not 0 <= m < n_t:
            continue
        k = min(m, n_t - 1 - m) + 1
        terms = 2 * c.dt * sum(abs(O.retarded(c, gl, m + i, m - i)) for i in range(k))
        # both sums: one rounding per term and addition, and the phase's own rounding, 3 eps |omega| t
        tol = 2 * eps * (k + 4 + 3 * np.abs(omega).max() * 2 * c.dt * k) * terms / np.pi
        assert np.abs(rho[row] - O.dos(c, gl, m, omega)).max() <= tol


# the last step of the tensor-core Gauss-Jordan with 1, 16, 64, 65 and 128 columns before the padding, both block
# widths, whole column tiles of padding (513, 641, 897), the 32-column tiles of the residual
@pytest.mark.parametrize("n", [17, 32, 33, 64, 65, 128, 129, 144, 193, 400, 449, 512, 513, 577, 641, 769, 897, 1025])
def test_mixed_lattice_padding_edges(n):
    c, g, mo, mc, sig, (eps, ebar, wq) = setup(n, 3)
    ref, jref = O.lattice_gloc(c, mo, sig, eps, ebar, wq)
    for width in (0,) if n <= 512 else (128, 256):
        api.lattice_set_tuning(g, 3, "mixed_bf16", width=width)
        gl, j = lattice(g, mc, sig, eps, ebar, wq, "mixed_bf16")
        assert rel(gl, ref) < 1e-6
        assert np.abs(j - jref.real).max() < 1e-5
    api.lattice_set_tuning(g, 3, "mixed_bf16")


# what the products leave out (panels and columns of padding) keeps the workspace's old bits: NaN there changes nothing
@pytest.mark.parametrize("n,prec", [(65, "mixed_bf16"), (400, "mixed_bf16"), (513, "mixed_bf16"), (897, "mixed_bf16"),
                                    (33, "fp64"), (129, "fp64"), (400, "fp64")])
def test_lattice_does_not_read_stale_workspace(n, prec):
    c, g, mo, mc, sig, (eps, ebar, wq) = setup(n, 3)
    s = torch.as_tensor(sig, device="cuda")
    out = []
    for fill in (0, 255):
        ws = torch.full((api.lattice_workspace_size(g, 3, prec),), fill, dtype=torch.uint8, device="cuda")
        gl, j, _ = api.lattice_gloc(g, mc, s, eps, ebar, wq, precision=prec, ws=ws)
        torch.cuda.synchronize()
        api.check_status()
        out.append((gl.cpu().numpy(), j.cpu().numpy()))
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])


# weights: zeros and exact ties at the threshold, one heavy point, more points than the sorted choice takes
@pytest.mark.parametrize("nq,kind", [(1, "one"), (300, "ties"), (300, "zeros"), (300, "heavy"), (8192, "random"),
                                     (8193, "random")])
def test_refined_points_of_the_mixed_path(nq, kind):
    c, g, mo, mc, sig, (eps, ebar, wq) = setup(24, nq)
    if kind == "ties":
        wq[:], eps[:], ebar[:] = 1.0 / nq, 0.3, np.where(np.arange(nq) % 2, 0.7, -0.7)
    elif kind == "zeros":
        wq[nq // 3:] = 0.0
    elif kind == "heavy":
        wq[1:] *= 1e-9
    wq /= wq.sum()
    ref, jref = O.lattice_gloc(c, mo, sig, eps, ebar, wq)
    gl, j = lattice(g, mc, sig, eps, ebar, wq, "mixed_bf16")
    assert rel(gl, ref) < 1e-6
    assert np.abs(j - jref.real).max() < 1e-5
