"""The work whose speed matters to a user of this library, as cases that can be timed and compared.

Each case is one pass through the public entry points, over the range of sizes that runs have: a whole small
DMFT loop, the lattice step of both precisions from the CPU-sized contour to the Mott run's, the impurity step,
the warm-start network's training step and prediction, and the diagnostics of a finished run.
"""

from __future__ import annotations

import math

import torch

from paper_0711_0999_gb300 import api, warmstart

DEVICE = "cuda"
BETA = 10.0


# ------------------------------------------------------------------ the cases

def listed():
    return [
        # The CPU-sized run, whole: 16 x 16 points, Sigma from 0 to convergence at 1e-8.  Every launch is small.
        dict(name="loop_fp64_nc80", kind="loop", t_min=-2.0, dt=0.2, n_t=30, n_tau=20, points=16, U=0.5, E=1.0),
        # One lattice step of that run: all matrices fit shared memory.
        dict(name="lattice_fp64_nc80", kind="lattice", precision="fp64", t_min=-2.0, dt=0.2, n_t=30, n_tau=20,
             points=16, U=0.5, E=1.0),
        # A short contour in FP64, just above the sizes that fit shared memory.
        dict(name="lattice_fp64_nc220", kind="lattice", precision="fp64", t_min=-2.0, dt=0.1, n_t=100, n_tau=20,
             points=10, U=1.0, E=1.0),
        # The coarsest step of the dt -> 0 extrapolation (dt = 0.1, t up to 25), in FP64 on an 8 x 8 grid.
        dict(name="lattice_fp64_nc700", kind="lattice", precision="fp64", t_min=-5.0, dt=0.1, n_t=300, n_tau=100,
             points=8, U=1.5, E=2.0),
        # The production contour in FP64 on a coarse grid: what the mixed path's accuracy is judged by.
        dict(name="lattice_fp64_nc1500", kind="lattice", precision="fp64", t_min=-5.0, dt=0.05, n_t=700, n_tau=100,
             points=7, U=1.0, E=1.0),
        # The lattice step of the warm start's training runs (32 x 32 points).
        dict(name="lattice_mixed_nc400", kind="lattice", precision="mixed_bf16", t_min=-5.0, dt=0.1, n_t=150,
             n_tau=100, points=32, U=0.9, E=1.5),
        # The production lattice step, whole: 53 x 53 points on the mixed path.
        dict(name="lattice_mixed_nc1500", kind="lattice", precision="mixed_bf16", t_min=-5.0, dt=0.05, n_t=700,
             n_tau=100, points=53, U=1.0, E=1.0),
        # The long Mott-insulating contour on the mixed path, a 16 x 16 grid of it.
        dict(name="lattice_mixed_nc3400", kind="lattice", precision="mixed_bf16", t_min=-5.0, dt=1.0 / 30.0,
             n_t=1650, n_tau=100, points=16, U=2.0, E=1.0),
        # The impurity step of the production run: the serial half of every DMFT iteration.
        dict(name="impurity_nc1500", kind="impurity", t_min=-5.0, dt=0.05, n_t=700, n_tau=100, U=1.0, E=1.0),
        # One training minibatch of the warm-start network: loss and gradient.
        dict(name="mlp_grad_2048", kind="mlp_grad", samples=2048),
        # The network's start for the production contour: its prediction on every pair of times, at both training steps.
        dict(name="warm_start_nc1500", kind="warm_start", t_min=-5.0, dt=0.05, n_t=700, n_tau=100, U=1.0, E=1.0),
        # The check of a finished production run: moments, density, and the density of states at five times.
        dict(name="diagnostics_nc1500", kind="diagnostics", t_min=-5.0, dt=0.05, n_t=700, n_tau=100, averages=5,
             omegas=401, U=1.0, E=1.0),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _contour(rng, lo, hi):
    """A contour of lo to hi rows in all (odd numbers among them): steps dt from 0.025 to 0.2, dtau from 0.1 to 1;
    the field comes on in its first third."""
    n = _log_int(rng, lo, hi)
    n_tau = min(_log_int(rng, 10, 100), max(10, n // 3))
    n_t = max(1, (n - n_tau) // 2)
    dt = rng.uniform(0.025, 0.2)
    return dict(t_min=-dt * n_t * rng.uniform(0.1, 0.35), dt=dt, n_t=n_t, n_tau=n_tau)


def draw(rng):
    kind = rng.choice(["loop", "fp64", "fp64", "fp64", "mixed", "mixed", "mixed", "impurity", "impurity", "mlp_grad",
                       "warm_start", "diagnostics"])
    model = dict(U=round(rng.uniform(0.25, 2.0), 3), E=round(rng.uniform(0.25, 4.0), 3))
    if kind == "loop":
        model["U"] = round(rng.uniform(0.25, 0.8), 3)
        return dict(kind="loop", points=rng.randint(4, 16), **_contour(rng, 12, 112), **model)
    if kind in ("fp64", "mixed"):
        c = _contour(rng, 16, 1500) if kind == "fp64" else _contour(rng, 60, 3400)
        n = 2 * c["n_t"] + c["n_tau"]
        pad = 128 * ((n + 127) // 128)
        # no dearer than the largest listed case: FP64 1500 x 49 points, mixed 1500 x 2809 points
        most = (49 * 1536**3 if kind == "fp64" else 2809 * 1536**3) / pad**3
        points = _log_int(rng, 4, max(4, min(32 if kind == "fp64" else 53, int(math.sqrt(0.8 * most)))))
        return dict(kind="lattice", precision="fp64" if kind == "fp64" else "mixed_bf16", points=points, **c, **model)
    if kind == "impurity":
        return dict(kind="impurity", **_contour(rng, 40, 3400), **model)
    if kind == "mlp_grad":
        return dict(kind="mlp_grad", samples=_log_int(rng, 200, 60000))
    if kind == "warm_start":
        return dict(kind="warm_start", **_contour(rng, 100, 1500), **model)
    return dict(kind="diagnostics", averages=rng.randint(1, 12), omegas=_log_int(rng, 50, 1000),
                **_contour(rng, 200, 3000), **model)


# ------------------------------------------------------------------ inputs

def _grid(case):
    return api.contour_grid(case["t_min"], case["t_min"] + case["n_t"] * case["dt"], case["dt"], BETA,
                            BETA / case["n_tau"])


def _times(case):
    """Contour times and weights as complex128 tensors: upper, lower, imaginary branch."""
    nt, ntau, dt, dtau = case["n_t"], case["n_tau"], case["dt"], BETA / case["n_tau"]
    t_max = case["t_min"] + nt * dt
    k = torch.arange(nt, dtype=torch.float64, device=DEVICE)
    z = torch.arange(ntau, dtype=torch.float64, device=DEVICE)
    re = torch.cat([case["t_min"] + k * dt, t_max - k * dt, torch.full_like(z, case["t_min"])])
    im = torch.cat([torch.zeros_like(k), torch.zeros_like(k), -dtau * z])
    w = torch.complex(torch.cat([torch.full_like(k, dt), torch.full_like(k, -dt), torch.zeros_like(z)]),
                      torch.cat([torch.zeros_like(k), torch.zeros_like(k), torch.full_like(z, -dtau)]))
    return torch.complex(re, im), w


def _rng(seed):
    return torch.Generator(device=DEVICE).manual_seed(int(seed))


def _model_values(case, seed):
    """U and E of one run: the case's, a few per cent apart from seed to seed."""
    g = torch.Generator().manual_seed(int(seed) + 17)
    a, b = (torch.rand(2, generator=g) * 0.06 - 0.03).tolist()
    return case["U"] * (1.0 + a), case["E"] * (1.0 + b)


def _sigma(case, U, seed):
    """A self-energy with the structure of the converged ones: the point-split band of the static part
    U<w1>, smooth damped oscillations in both times of size U^2/8, and a little dense noise."""
    t, w = _times(case)
    n = t.numel()
    g = _rng(seed)
    tr, tau = t.real, -t.imag
    amp = U * U / 8.0
    p = torch.rand((6, 4), generator=g, dtype=torch.float64, device=DEVICE)
    c = torch.randn((6, 2), generator=g, dtype=torch.float64, device=DEVICE) / math.sqrt(12.0)
    k = 3.0 * p[:, :2] - 1.5
    d = 0.05 + 0.35 * p[:, 2:]
    u = torch.exp(torch.complex(-d[:, :1] * tau, k[:, :1] * tr)) * torch.complex(c[:, :1], c[:, 1:])
    v = torch.exp(torch.complex(-d[:, 1:] * tau, -k[:, 1:] * tr))
    s = amp * (u.T @ v)
    noise = torch.randn((n, n, 2), generator=g, dtype=torch.float64, device=DEVICE)
    s += 0.05 * amp * torch.view_as_complex(noise)
    j = torch.arange(1, n, device=DEVICE)
    s[j, j - 1] += (U / 2.0) / w[:-1]
    s[0, n - 1] -= (U / 2.0) / w[n - 1]
    return s


def _band_phase(t_re, eps, ebar, E):
    """The antiderivative F(s) of the band energy in the field (E switched on at s = 0)."""
    on = (eps * torch.sin(E * t_re) + ebar * (torch.cos(E * t_re) - 1.0)) / E
    return torch.where(t_re <= 0.0, eps * t_re, on)


def _quadrature(n):
    """The n x n Gauss-Hermite points of exp(-x^2)/sqrt(pi): eps outer, ebar inner, weights summing to 1."""
    k = torch.arange(1, n, dtype=torch.float64)
    x, v = torch.linalg.eigh(torch.diag((k / 2).sqrt(), 1) + torch.diag((k / 2).sqrt(), -1))
    w = v[0] ** 2
    return x.repeat_interleave(n), x.repeat(n), w.repeat_interleave(n) * w.repeat(n)


def _gloc(case, U, E):
    """A local Green's function of the right structure: the noninteracting one, averaged over a 6 x 6 grid."""
    t, _ = _times(case)
    n = t.numel()
    later = torch.ones((n, n), dtype=torch.bool, device=DEVICE).tril()
    out = torch.zeros((n, n), dtype=torch.complex128, device=DEVICE)
    for eps, ebar, wq in zip(*(a.tolist() for a in _quadrature(6))):
        x = eps - U / 2.0
        soft = [math.log1p(math.exp(-abs(BETA * x))) + max(y, 0.0) for y in (-BETA * x, BETA * x)]
        ph = U / 2.0 * t.real - _band_phase(t.real, eps, ebar, E)
        tau = -t.imag
        mag = -x * (tau[:, None] - tau[None, :])
        mag = torch.where(later, mag - soft[0], mag - soft[1])
        g = torch.exp(torch.complex(mag, ph[:, None] - ph[None, :]))
        out += (-1j * wq) * torch.where(later, g, -g)
    return out


def prepare(case, seed):
    kind = case["kind"]
    if kind == "mlp_grad":
        n = case["samples"]
        g = _rng(seed)
        # features in the ranges of the library's own: most within [-1, 1], one-hot branches 0 or 1
        x = torch.rand((n, warmstart.N_IN), generator=g, device=DEVICE) * 2.0 - 1.0
        x[:, 6:9] = torch.nn.functional.one_hot(torch.randint(0, 3, (n,), generator=g, device=DEVICE), 3).float()
        x[:, 12:15] = torch.nn.functional.one_hot(torch.randint(0, 3, (n,), generator=g, device=DEVICE), 3).float()
        t = torch.stack([torch.sin(x[:, 2] * 3.0) * x[:, 0], torch.cos(x[:, 3] * 2.0) * x[:, 1]], 1).contiguous()
        params = torch.as_tensor(warmstart.init_params(seed), device=DEVICE)
        return dict(case=case, x=x, t=t, params=params)
    U, E = _model_values(case, seed)
    grid = _grid(case)
    st = dict(case=case, grid=grid, model=api.make_model(U, E))
    if kind == "lattice":
        eps, ebar, wq = api.quadrature_grid(case["points"])
        st["sigma"] = _sigma(case, U, seed)
        st["points"] = [torch.as_tensor(a, device=DEVICE) for a in (eps, ebar, wq)]
        st["ws"] = api.workspace(api.lattice_workspace_size(grid, case["points"] ** 2, case["precision"]), DEVICE)
    elif kind == "impurity":
        st["gloc"] = _gloc(case, U, E)
        st["sigma"] = _sigma(case, U, seed)
    elif kind == "warm_start":
        st["params"] = torch.as_tensor(warmstart.init_params(seed), device=DEVICE)
    elif kind == "diagnostics":
        st["gloc"] = _gloc(case, U, E)
        nt = case["n_t"]
        st["m"] = [int((k + 1) * nt / (case["averages"] + 1)) for k in range(case["averages"])]
        st["omega"] = torch.linspace(-5.0, 5.0, case["omegas"], dtype=torch.float64, device=DEVICE)
    return st


# ------------------------------------------------------------------ one pass

def run(state):
    case, kind = state["case"], state["case"]["kind"]
    if kind == "lattice":
        eps, ebar, wq = state["points"]
        gloc, j, j_imag = api.lattice_gloc(state["grid"], state["model"], state["sigma"], eps, ebar, wq,
                                           precision=case["precision"], ws=state["ws"])
        return dict(gloc=gloc, j=j, j_imag=j_imag)
    if kind == "impurity":
        sigma_new, _ = api.impurity_update(state["grid"], state["model"], state["gloc"], state["sigma"])
        return dict(sigma=sigma_new)
    if kind == "loop":
        sol = api.dmft_solve(state["grid"], state["model"], case["points"], "fp64", tol=1e-8, max_iter=40)
        return dict(sigma=sol.sigma, gloc=sol.gloc, j=sol.current, iterations=sol.iterations)
    if kind == "mlp_grad":
        loss, grad = warmstart.loss_and_grad(state["params"], state["x"], state["t"])
        return dict(loss=loss, grad=grad)
    if kind == "warm_start":
        return dict(sigma=warmstart.warm_start(state["grid"], state["model"], state["params"]))
    mu0, mu1, mu2, dens = api.moments(state["grid"], state["gloc"])
    rho = api.dos(state["grid"], state["gloc"], state["m"], state["omega"])
    return dict(mu0=mu0, mu1=mu1, mu2=mu2, density=dens, rho=rho)


# ------------------------------------------------------------------ the least work of a pass

def work(case):
    kind = case["kind"]
    if kind == "mlp_grad":
        n, p = case["samples"], sum(a * b + b for a, b in zip(warmstart.DIMS[:-1], warmstart.DIMS[1:]))
        mul = sum(a * b for a, b in zip(warmstart.DIMS[:-1], warmstart.DIMS[1:]))
        return dict(bytes=4.0 * (n * 19 + 2 * p), flops=2.0 * n * (3 * mul - warmstart.DIMS[0] * warmstart.DIMS[1]))
    n = 2 * case["n_t"] + case["n_tau"]
    if kind == "lattice":  # one complex n x n inverse (8 n^3 real operations) for each point
        q = case["points"] ** 2
        return dict(bytes=32.0 * n * n + 24.0 * q + 16.0 * case["n_t"], flops=8.0 * n**3 * q)
    if kind == "impurity":  # two inverses
        return dict(bytes=48.0 * n * n, flops=16.0 * n**3)
    if kind == "loop":  # about 15 iterations
        return dict(bytes=32.0 * n * n, flops=15.0 * 8.0 * n**3 * (case["points"] ** 2 + 2))
    if kind == "warm_start":
        mul = sum(a * b for a, b in zip(warmstart.DIMS[:-1], warmstart.DIMS[1:]))
        return dict(bytes=16.0 * n * n, flops=2.0 * len(warmstart.TRAIN_DTS) * n * n * mul)
    terms = case["averages"] * case["n_t"] / 4.0  # relative times of an average time, on average
    return dict(bytes=32.0 * terms + 8.0 * case["averages"] * case["omegas"] + 150.0 * case["n_t"],
                flops=4.0 * terms * case["omegas"])


# ------------------------------------------------------------------ the same in 64 bits

def _lattice_exact(case, S, U, E, eps, ebar, wq):
    """sum_q w_q inv(B_q - S) and i sum_q w_q ebar_q(t_m) G_q^<(t_m, t_m), B_q the closed-form inverse of G0_q."""
    t, _ = _times(case)
    n, nt, mu = t.numel(), case["n_t"], U / 2.0
    j = torch.arange(1, n, device=DEVICE)
    rows = torch.arange(nt, device=DEVICE)
    tm = t.real[:nt]
    gloc = torch.zeros((n, n), dtype=torch.complex128, device=DEVICE)
    cur = torch.zeros(nt, dtype=torch.complex128, device=DEVICE)
    step = max(1, min(256, int(3e9 / (16 * n * n))))
    for q0 in range(0, eps.numel(), step):
        e, b, w = (a[q0:q0 + step, None] for a in (eps, ebar, wq))
        ph = mu * t.real - _band_phase(t.real[None], e, b, E)
        x = e - mu
        A = (-S).repeat(e.shape[0], 1, 1)
        A.diagonal(dim1=1, dim2=2).add_(1j)
        mag = x * (t.imag[1:] - t.imag[:-1])
        A[:, j, j - 1] += -1j * torch.exp(torch.complex(mag, ph[:, 1:] - ph[:, :-1]))
        A[:, 0, n - 1] += 1j * torch.exp(-x[:, 0] * BETA / case["n_tau"])
        G = torch.linalg.inv(A)
        gloc += torch.einsum("q,qij->ij", w[:, 0].to(G.dtype), G)
        on = torch.where(tm > 0.0, b * torch.cos(E * tm) + e * torch.sin(E * tm), b.expand(-1, nt))
        cur += (w * on * G[:, rows, 2 * nt - rows]).sum(0)
    return gloc, 1j * cur


def _impurity_exact(case, gloc, S, U):
    """W Sigma_new W = -w1 D + w1 (1 - w1) D inv(A_h) D, A_h = inv(G_loc) + S + (1 - w1) D, w1 = 1/2."""
    _, w = _times(case)
    d = torch.cat([U * w[:1], -U * w[1:]])
    D = torch.roll(torch.diag(d), -1, 1)  # one entry per row: d_i at (i, i - 1)
    Ah = torch.linalg.inv(gloc) + S + 0.5 * D
    X = torch.linalg.inv(Ah)
    new = 0.25 * d[:, None] * torch.roll(torch.roll(X, 1, 0), -1, 1) * torch.roll(d, -1)[None, :] - 0.5 * D
    return new / (w[:, None] * w[None, :])


def _layers(params):
    out, at = [], 0
    for a, b in zip(warmstart.DIMS[:-1], warmstart.DIMS[1:]):
        out.append((params[at:at + a * b].view(a, b), params[at + a * b:at + a * b + b]))
        at += a * b + b
    return out


def _network(layers, x):
    for k, (w, b) in enumerate(layers):
        x = x @ w + b
        if k + 1 < len(layers):
            x = torch.tanh(x)
    return x


def _features(case, U, E, a, b, dt):
    """The network's inputs for the pairs (t_a, t_b) of contour rows."""
    t, _ = _times(case)
    nt = case["n_t"]
    branch = torch.nn.functional.one_hot((torch.arange(t.numel(), device=DEVICE) // nt).clamp(max=2), 3).double()

    def of(i):
        r, tau = t.real[i], -t.imag[i]
        return [torch.tanh(r.clamp(min=0.0) / 3.0), r.clamp(max=0.0) / 5.0, tau / BETA, *branch[i].unbind(1)]

    one = torch.ones_like(t.real[a])
    f = [U / 2.5 * one, E / 4.0 * one, torch.tanh((t.real[a] - t.real[b]) / 3.0), *of(a), *of(b), (a >= b).double(),
         dt / 0.1 * one]
    return torch.stack(f, 1)


def exact(case, seed):
    kind = case["kind"]
    if kind == "mlp_grad":
        st = prepare(case, seed)
        p = st["params"].double().requires_grad_()
        loss = ((_network(_layers(p), st["x"].double()) - st["t"].double()) ** 2).mean()
        loss.backward()
        return dict(loss=loss.detach().view(1), grad=p.grad)
    n = 2 * case["n_t"] + case["n_tau"]
    U, E = _model_values(case, seed)
    t, w = _times(case)
    if kind == "lattice":
        if 8.0 * n**3 * case["points"] ** 2 > 4e12:
            return None
        S = w[:, None] * _sigma(case, U, seed) * w[None, :]
        gloc, cur = _lattice_exact(case, S, U, E, *(a.to(DEVICE) for a in _quadrature(case["points"])))
        return dict(gloc=gloc, j=cur.real.contiguous(), j_imag=cur.imag.contiguous())
    if kind == "impurity":
        S = w[:, None] * _sigma(case, U, seed) * w[None, :]
        return dict(sigma=_impurity_exact(case, _gloc(case, U, E), S, U))
    if kind == "loop":
        pts = [a.to(DEVICE) for a in _quadrature(case["points"])]
        S = torch.zeros((n, n), dtype=torch.complex128, device=DEVICE)
        old, it = None, 0
        while True:
            it += 1
            gloc, cur = _lattice_exact(case, S, U, E, *pts)
            if it == 40 or (old is not None and float((gloc - old).abs().max() / gloc.abs().max()) < 1e-8):
                break
            old = gloc
            S = w[:, None] * _impurity_exact(case, gloc, S, U) * w[None, :]
        return dict(sigma=S / (w[:, None] * w[None, :]), gloc=gloc, j=cur.real.contiguous(), iterations=it)
    if kind == "warm_start":
        layers = _layers(torch.as_tensor(warmstart.init_params(seed), device=DEVICE).double())
        dts = warmstart.TRAIN_DTS
        X = torch.zeros((n * n, 2), dtype=torch.float64, device=DEVICE)
        for k, dt in enumerate(dts):
            lag = math.prod((case["dt"] - o) / (dt - o) for i, o in enumerate(dts) if i != k)
            for at in range(0, n * n, 1 << 18):
                e = torch.arange(at, min(n * n, at + (1 << 18)), device=DEVICE)
                X[at:at + e.numel()] += lag * _network(layers, _features(case, U, E, e // n, e % n, dt))
        X = torch.complex(X[:, 0], X[:, 1]).view(n, n)
        d = torch.cat([U * w[:1], -U * w[1:]])
        new = 0.25 * d[:, None] * torch.roll(torch.roll(X, 1, 0), -1, 1) * torch.roll(d, -1)[None, :]
        new -= 0.5 * torch.roll(torch.diag(d), -1, 1)
        return dict(sigma=new / (w[:, None] * w[None, :]))
    g = _gloc(case, U, E)
    nt, dt = case["n_t"], case["dt"]
    m = torch.arange(nt, device=DEVICE)

    def f(i, j):  # i G^R(t_i, t_j)
        return 1j * (g[2 * nt - i, j] - g[i, 2 * nt - j])

    mu = torch.full((3, nt), math.nan, dtype=torch.float64, device=DEVICE)
    if nt > 6:
        c = m[3:nt - 3]
        f1, f2, f3 = (f(c + k, c - k) for k in (1, 2, 3))
        h = 2.0 * dt
        mu[0, 3:nt - 3] = (3.0 * f1 - 3.0 * f2 + f3).real
        mu[1, 3:nt - 3] = (1j * (-5.0 * f1 + 8.0 * f2 - 3.0 * f3)).real / (2.0 * h)
        mu[2, 3:nt - 3] = -((f1 - 2.0 * f2 + f3) / (h * h)).real
    st = prepare(case, seed)
    rho = torch.zeros((len(st["m"]), case["omegas"]), dtype=torch.float64, device=DEVICE)
    for row, a in enumerate(st["m"]):
        top = min(a, nt - 1 - a)
        if top > 0:
            k = torch.arange(top + 1, device=DEVICE)
            at = 2.0 * dt * k.double()
            wk = torch.ones(top + 1, dtype=torch.float64, device=DEVICE)
            wk[0] = wk[-1] = 0.5
            gr = -1j * f(a + k, a - k)
            wave = torch.exp(1j * st["omega"][:, None] * at[None, :])
            rho[row] = -(2.0 * dt * (wave * (wk * gr)[None, :]).sum(1)).imag / math.pi
    return dict(mu0=mu[0], mu1=mu[1], mu2=mu[2], density=(-1j * g[m, 2 * nt - m]).real.contiguous(), rho=rho)
