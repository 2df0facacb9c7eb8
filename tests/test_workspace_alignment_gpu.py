"""The impurity step takes a workspace at any address, as it did before its operands were written in 32-byte pieces."""

import ctypes

import numpy as np
import pytest
import torch

from oracle import nedmft_oracle as O
from paper_0711_0999_gb300 import _native as N
from paper_0711_0999_gb300 import api
from paper_0711_0999_gb300.build import build_library
from paper_0711_0999_gb300.synth import workload_sigma

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    build_library()


@pytest.mark.parametrize("offset", [16, 48, 240])
def test_impurity_step_in_an_unaligned_workspace(offset):
    args = (-2, 4, 0.2, 10, 0.5)
    c, g, mod = O.contour_grid(*args), api.contour_grid(*args), api.make_model(1.0, 1.0)
    sig = workload_sigma(c.t, c.w, 1.0, seed=5)
    gl, _ = O.lattice_gloc(c, O.Model(U=1.0, E=1.0), sig, *O.quadrature_points(3))
    gd, sd = (torch.as_tensor(a, device="cuda") for a in (gl, sig))
    need = N.lib().nedmft_impurity_workspace_size(ctypes.byref(g.contour))
    buf = torch.empty(need + 512, dtype=torch.uint8, device="cuda")
    base = -buf.data_ptr() % 256
    out = []
    for at in (base, base + offset):
        new, _ = api.impurity_update(g, mod, gd, sd, ws=buf[at:at + need])
        torch.cuda.synchronize()
        api.check_status()
        out.append(new.cpu().numpy())
    assert np.array_equal(out[0], out[1])
