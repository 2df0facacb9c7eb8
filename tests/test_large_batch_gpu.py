"""A pinned batch of more points than a grid's second dimension has blocks (65535)."""

import numpy as np
import pytest
import torch

from paper_0711_0999_gb300 import api
from paper_0711_0999_gb300.build import build_library
from paper_0711_0999_gb300.synth import workload_sigma

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    build_library()


def test_fp64_lattice_step_with_a_pinned_batch_beyond_one_launch():
    nq = 65535 + 70
    g = api.contour_grid(-1.0, 0.25, 0.125, 1.0, 0.25)
    assert g.n_c == 24
    rng = np.random.default_rng(7)
    eps, ebar = rng.normal(0.25, 1.2, nq), rng.normal(0.0, 1.0, nq)
    wq = np.full(nq, 1.0 / nq)
    sig = torch.as_tensor(workload_sigma(g.t, g.w, 0.5, seed=2), device="cuda")
    out = []
    for batch in (0, nq):
        api.lattice_set_tuning(g, nq, "fp64", batch=batch)
        try:
            gl, j, _ = api.lattice_gloc(g, api.make_model(0.5, 1.0), sig, eps, ebar, wq)
            torch.cuda.synchronize()
            api.check_status()
        finally:
            api.lattice_set_tuning(g, nq, "fp64")
        out.append((gl, j))
    # the same matrices; nq sums of weights 1 / nq in another order
    tol = 4 * np.sqrt(nq) * 2.0**-53
    assert float((out[1][0] - out[0][0]).abs().max()) < tol * float(out[0][0].abs().max())
    assert float((out[1][1] - out[0][1]).abs().max()) < tol * 10.0
