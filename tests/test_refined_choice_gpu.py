"""The choice of the points that the mixed path refines, where its threshold falls
between two roundings of the same running sum."""

import numpy as np
import pytest
import torch

from oracle import nedmft_oracle as O
from paper_0711_0999_gb300 import api
from paper_0711_0999_gb300.build import build_library
from paper_0711_0999_gb300.synth import workload_sigma

pytestmark = pytest.mark.gpu

TAIL = 1e-3  # the share of the weights that is not refined


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    build_library()


def block_sum(v):
    """The kernel's sum of up to 1024 values: pairs of halves."""
    r = np.zeros(1024)
    r[:len(v)] = v
    s = 512
    while s:
        r[:s] += r[s:2 * s]
        s //= 2
    return r[0]


def running_sums(v):
    """Its inclusive scan."""
    r = np.zeros(1024)
    r[:len(v)] = v
    s = 1
    while s < 1024:
        r = r + np.concatenate([np.zeros(s), r[:-s]])
        s *= 2
    return r


def tie_weights(n=300):
    """n weights whose tail lies between red[t - 1] + w_t and red[t], red the scan's running sums, for some t."""
    small = np.random.default_rng(1).uniform(0.5, 1.0, n - 4) * TAIL * 4 / (n - 4)
    heavy = float.fromhex("0x1.3760b63f6d0eep-3")
    w = np.concatenate([small, np.full(3, heavy), [heavy - 4 * np.spacing(heavy)]])
    srt = np.sort(w)
    red, tail = running_sums(srt), TAIL * block_sum(w)
    end = red[:n - 1] + srt[1:]
    assert ((end <= tail) & (tail < red[1:n])).any()
    return w


def test_a_threshold_between_two_roundings_still_refines_the_points():
    args = (-2, 3, 0.05, 5.0, 0.25)
    c, g = O.contour_grid(*args), api.contour_grid(*args)
    assert g.n_c == 220
    sig = workload_sigma(c.t, c.w, 1.0, seed=9)
    wq = tie_weights()
    zero = np.zeros_like(wq)
    ref, _ = O.lattice_gloc(c, O.Model(U=1.0, E=1.0), sig, zero[:1], zero[:1], np.array([wq.sum()]))
    gl, _, _ = api.lattice_gloc(g, api.make_model(1.0, 1.0), torch.as_tensor(sig, device="cuda"), zero, zero, wq,
                                precision="mixed_bf16")
    torch.cuda.synchronize()
    api.check_status()
    assert np.abs(gl.cpu().numpy() - ref).max() < 1e-6 * np.abs(ref).max()
