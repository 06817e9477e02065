"""The calls that a program built on this library spends its time in, over the
range of sizes, forms and options that it is used with: constant-depth steps
(both arithmetic forms, real and complex data, square, rectangular and odd
grids, the adjoint, host buffers, the scalar operator, batches of instances)
and variable-depth steps (the shared Krylov basis, one CG solve per term, the
gradient with respect to state and depth through a rollout).

A case is a dict of plain values.  ``prepare`` makes what a program has in
hand before the call (plan, buffers, inputs on the GPU), ``run`` is one call,
``exact`` the same result in FP64 with plain torch and numpy.
"""
import math
import random

import numpy as np
import torch
from torch.utils.checkpoint import checkpoint

from paper_2008_11607_gb300 import autograd, rexi

TOL = 1e-10


def listed():
    """Sizes and options of the library's own configurations (64^2, 2048^2, the
    1024^2 variable-depth step, the serving mix of 96 instances, the 512^2
    rollout) and ordinary ragged ones between them."""
    return [
        # one small step, FP64, real data, the Gaussian bump: latency and launches
        dict(name="step_fp64_64", family="step", nx=64, ny=64, tau_rho=50.0, form="fp64", real=True, field="bump"),
        # complex data on a ragged rectangular grid: the full-spectrum transforms
        dict(name="step_mixed_360x250_complex", family="step", nx=360, ny=250, tau_rho=120.0, form="mixed", real=False,
             field="noise"),
        # the 2048^2 step, tau rho = 1000, in the mixed form and in FP64
        dict(name="step_mixed_2048", family="step", nx=2048, ny=2048, tau_rho=1000.0, form="mixed", real=True,
             field="smooth"),
        dict(name="step_fp64_2048", family="step", nx=2048, ny=2048, tau_rho=1000.0, form="fp64", real=True,
             field="smooth"),
        # forward and adjoint through torch.autograd, FP64, odd nx (no half-length real transform)
        dict(name="autograd_fp64_375x500", family="autograd", nx=375, ny=500, tau_rho=150.0, form="fp64", real=True,
             field="smooth"),
        # a step on pinned host buffers, copies included
        dict(name="host_mixed_1024", family="host", nx=1024, ny=1024, tau_rho=400.0, form="mixed", real=True,
             field="smooth"),
        # the scalar operator i (d_xx + d_yy): REXIE coefficients with the midpoint shift
        dict(name="scalar_mixed_512x384", family="scalar", nx=512, ny=384, tau_rho=300.0, form="mixed", real=False,
             field="noise"),
        # the serving mix: 96 instances of 128^2..512^2, tau rho 20..800, one batched call
        dict(name="batch_mixed_96", family="batch", count=96, smallest=128, largest=512, rho_lo=20.0, rho_hi=800.0,
             square=True, mix=0, form="mixed", real=True),
        # variable depth, shared Krylov basis kept in memory: the 1024^2 step
        dict(name="depth_mixed_1024", family="depth", nx=1024, ny=1024, tau_rho=400.0, form="mixed", real=True,
             method="shared", kept=True),
        # the same in FP64 on a ragged grid with the workspace that the library asks for (basis regenerated)
        dict(name="depth_fp64_380x310", family="depth", nx=380, ny=310, tau_rho=100.0, form="fp64", real=True,
             method="shared", kept=False),
        # variable depth with the default solver, one CG solve per term
        dict(name="depth_cg_fp64_128x96", family="depth", nx=128, ny=96, tau_rho=15.0, form="fp64", real=True,
             method="cg", kept=False),
        # training: 8 steps with checkpoints every 2, gradients of state and depth
        dict(name="rollout_mixed_512", family="rollout", nx=512, ny=512, tau_rho=200.0, form="mixed", steps=8, every=2,
             rtol=1e-12),
    ]


def _size(rng, lo, hi):
    """A grid length between lo and hi, spread over its logarithm, that the transforms accept."""
    while True:
        n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
        m, p = n, 2
        while m > 1 and p <= 127:
            if m % p:
                p += 1
            else:
                m //= p
        if m == 1 and lo <= n <= hi:
            return n


def _log(rng, lo, hi):
    return float("%.4g" % math.exp(rng.uniform(math.log(lo), math.log(hi))))


def draw(rng):
    family = rng.choice(["step", "step", "step", "step", "autograd", "host", "scalar", "batch", "batch", "depth", "depth",
                         "depth", "cg", "rollout"])
    form = rng.choice(["fp64", "mixed", "mixed"])
    square = rng.random() < 0.4
    if family in ("step", "autograd", "host", "scalar"):
        top = 2048 if family == "step" else 1024
        nx = _size(rng, 32, top)
        ny = nx if square else _size(rng, 32, top)
        real = family != "scalar" and (family in ("autograd", "host") or rng.random() < 0.6)
        return dict(family=family, nx=nx, ny=ny, tau_rho=_log(rng, 10.0, 1000.0), form=form, real=real,
                    field="smooth" if real else "noise")
    if family == "batch":
        return dict(family="batch", count=rng.randint(2, 48), smallest=rng.choice([24, 48, 96, 128]),
                    largest=rng.choice([160, 256, 384, 512]), rho_lo=_log(rng, 10.0, 40.0),
                    rho_hi=_log(rng, 100.0, 800.0), square=square, mix=rng.randint(1, 10 ** 6), form=form,
                    real=rng.random() < 0.7)
    if family == "depth":
        nx = _size(rng, 48, 1024)
        return dict(family="depth", nx=nx, ny=nx if square else _size(rng, 48, 1024), tau_rho=_log(rng, 20.0, 400.0),
                    form=form, real=rng.random() < 0.8, method="shared", kept=rng.random() < 0.5)
    if family == "cg":
        return dict(family="depth", nx=_size(rng, 32, 128), ny=_size(rng, 32, 96), tau_rho=_log(rng, 3.0, 15.0),
                    form=form, real=True, method="cg", kept=False)
    return dict(family="rollout", nx=_size(rng, 48, 400), ny=_size(rng, 48, 400), tau_rho=_log(rng, 20.0, 200.0),
                form=form, steps=rng.randint(1, 4), every=rng.choice([1, 2]), rtol=1e-12)


# ---- inputs ------------------------------------------------------------------

_DEVICE = "cuda"


def _generator(seed, salt=0):
    g = torch.Generator(device=_DEVICE)
    g.manual_seed(1000003 * int(seed) + salt)
    return g


def _smooth(nx, ny, g):
    """Smooth random field, Fourier amplitude |k|^-3, scaled to a largest value of 0.1."""
    kx = torch.fft.fftfreq(nx, 1.0 / nx, device=_DEVICE, dtype=torch.float64)
    ky = torch.fft.fftfreq(ny, 1.0 / ny, device=_DEVICE, dtype=torch.float64)
    k2 = ky[:, None] ** 2 + kx[None, :] ** 2
    k2[0, 0] = 1.0
    amp = k2 ** -1.5
    amp[0, 0] = 0.0
    phase = 2.0 * math.pi * torch.rand(ny, nx, generator=g, device=_DEVICE, dtype=torch.float64)
    v = torch.fft.ifft2(torch.polar(amp, phase)).real
    return 0.1 * v / v.abs().max()


def _field(case, seed, salt=0):
    """The state (3, ny, nx), complex128: "bump" and "smooth" are a height field
    at rest, "noise" a full complex state."""
    nx, ny = case["nx"], case["ny"]
    g = _generator(seed, salt)
    state = torch.zeros(3, ny, nx, dtype=torch.complex128, device=_DEVICE)
    kind = case.get("field", "smooth")
    if kind == "noise":
        re = torch.randn(3, ny, nx, generator=g, device=_DEVICE, dtype=torch.float64)
        im = torch.randn(3, ny, nx, generator=g, device=_DEVICE, dtype=torch.float64)
        return torch.complex(re, im)
    if kind == "bump":  # the Gaussian bump, its centre and width from the seed
        c = torch.rand(3, generator=g, device=_DEVICE, dtype=torch.float64).tolist()
        x = (torch.arange(nx, device=_DEVICE, dtype=torch.float64) + 0.5) / nx - c[0]
        y = (torch.arange(ny, device=_DEVICE, dtype=torch.float64) + 0.5) / ny - c[1]
        x, y = x - x.round(), y - y.round()
        w = 0.04 + 0.02 * c[2]
        state[0] = 0.1 * torch.exp(-(x[None, :] ** 2 + y[:, None] ** 2) / (2.0 * w * w))
        return state
    state[0] = _smooth(nx, ny, g)
    return state


def _depth_field(nx, ny, seed):
    """H = 1 + 0.4 sin(2 pi x) cos(4 pi y) and 8 periodic bumps of amplitude 0.1."""
    g = _generator(seed, 77)
    x = (torch.arange(nx, device=_DEVICE, dtype=torch.float64) + 0.5) / nx
    y = (torch.arange(ny, device=_DEVICE, dtype=torch.float64) + 0.5) / ny
    H = 1.0 + 0.4 * torch.sin(2.0 * math.pi * x)[None, :] * torch.cos(4.0 * math.pi * y)[:, None]
    for cx, cy in torch.rand(8, 2, generator=g, device=_DEVICE, dtype=torch.float64).tolist():
        dx, dy = x - cx, y - cy
        dx, dy = dx - dx.round(), dy - dy.round()
        H = H + 0.1 * torch.exp(-(dx[None, :] ** 2 + dy[:, None] ** 2) / (2.0 * 0.05 ** 2))
    return H.contiguous()


def _instances(case):
    """(nx, ny, tau rho) of a batch: the serving mix's five sizes, or multiples of 8 or 32 between the
    smallest and the largest; log-uniform tau rho."""
    rng = random.Random(20240 + case["mix"])
    step = 32 if case["smallest"] >= 128 else 8
    sizes = [n for n in range(case["smallest"], case["largest"] + 1, step)]
    if case["square"] and case["smallest"] == 128 and case["largest"] == 512:
        sizes = [128, 192, 256, 384, 512]
    out = []
    for _ in range(case["count"]):
        nx = rng.choice(sizes)
        ny = nx if case["square"] else rng.choice(sizes)
        out.append((nx, ny, math.exp(rng.uniform(math.log(case["rho_lo"]), math.log(case["rho_hi"])))))
    return out


# ---- what a program keeps, and one call ----------------------------------------


class _State:
    pass


def prepare(case, seed):
    s = _State()
    s.case = case
    family = case["family"]
    if family == "batch":
        inst = _instances(case)
        sizes = [(nx, ny) for nx, ny, _ in inst]
        s.batch = rexi.Batch(sizes, [t / _rho_cgrid(nx, ny) for nx, ny, t in inst], form=case["form"], tol=TOL)
        s.packed = s.batch.pack([_field(dict(nx=nx, ny=ny, field="smooth" if case["real"] else "noise"), seed, 1 + i)
                                 for i, (nx, ny) in enumerate(sizes)])
        s.out = s.batch.empty()
        s.workspace = s.batch.workspace()
        return s
    if family in ("depth", "rollout"):
        s.depth = _depth_field(case["nx"], case["ny"], seed)
        s.plan = rexi.Plan(case["nx"], case["ny"], depth=s.depth, form=case["form"])
        s.dt = case["tau_rho"] / s.plan.rho
        real = case.get("real", True)
        s.state = _field(dict(case, field="smooth" if real else "noise"), seed)
        if family == "rollout":
            s.plan.set_krylov(rtol=case["rtol"])
            s.plan.set_krylov_method("shared")
            s.grad_out = torch.zeros_like(s.state)
            s.grad_out[0] = _smooth(case["nx"], case["ny"], _generator(seed, 5))
            s.state.requires_grad_(True)
            s.depth.requires_grad_(True)
            return s
        s.plan.set_krylov_method(case["method"])
        n = s.plan.workspace_size(s.dt, TOL, real)
        if case["kept"]:
            n += int(1.3 * case["tau_rho"] + 64) * s.plan.krylov_vector_bytes(real)
        s.workspace = torch.empty(n, dtype=torch.uint8, device=_DEVICE)
        s.out = torch.empty_like(s.state)
        return s
    s.plan = rexi.Plan(case["nx"], case["ny"], form=case["form"])
    if family == "scalar":
        s.plan.set_symbol("schrodinger")
        s.plan.set_coefficients("rexie")
        s.plan.set_shift("midpoint")
    s.dt = case["tau_rho"] / s.plan.rho
    s.state = _field(case, seed)
    if family == "host":
        s.host_in = s.state.cpu().pin_memory()
        s.host_out = torch.empty_like(s.host_in, pin_memory=True)
        s.workspace = s.plan.workspace_host(s.dt, TOL, case["real"])
        del s.state
    elif family == "autograd":
        s.state.requires_grad_(True)
        s.grad_out = _field(dict(case, field="noise"), seed, 9)
    else:
        s.out = torch.empty_like(s.state)
        s.workspace = s.plan.workspace(s.dt, TOL, case["real"])
    return s


def run(s):
    case = s.case
    family = case["family"]
    if family == "batch":
        return s.batch.step(s.packed, s.out, s.workspace, real_input=case["real"])
    if family == "host":
        return s.plan.step_host(s.host_in, s.host_out, s.dt, tol=TOL, real_input=case["real"], workspace=s.workspace)
    if family == "autograd":
        out = autograd.rexi_step(s.state, s.plan, s.dt, tol=TOL, real_input=case["real"])
        (grad,) = torch.autograd.grad(out, (s.state,), s.grad_out)
        return {"out": out.detach(), "grad_state": grad}
    if family == "rollout":
        out = autograd.rexi_rollout(s.state, s.plan, s.dt, case["steps"], every=case["every"], depth=s.depth, tol=TOL)
        gs, gd = torch.autograd.grad(out, (s.state, s.depth), s.grad_out)
        return {"out": out.detach(), "grad_state": gs, "grad_depth": gd}
    return s.plan.step(s.state, s.dt, tol=TOL, real_input=case["real"], out=s.out, workspace=s.workspace)


def work(case):
    """Bytes: each input read once, each output written once (16 bytes per value
    of a state, 8 per depth value).  Flops: the transforms (5 n log2 n per
    complex field, half of that for real data) and the 3 x 3 symbol, or for
    variable depth one stencil application (30 per point) per unit of tau rho."""

    def fourier(nx, ny, real, passes=1):
        n = nx * ny
        fft = 2 * 3 * 5.0 * n * math.log2(n) * (0.5 if real else 1.0)
        return {"bytes": passes * 96.0 * n, "flops": passes * (fft + 150.0 * n * (0.5 if real else 1.0))}

    family = case["family"]
    if family == "batch":
        w = [fourier(nx, ny, case["real"]) for nx, ny, _ in _instances(case)]
        return {"bytes": sum(x["bytes"] for x in w), "flops": sum(x["flops"] for x in w)}
    n = case["nx"] * case["ny"]
    if family == "depth":
        return {"bytes": 104.0 * n, "flops": 30.0 * n * case["tau_rho"] * (1.0 if case["real"] else 2.0)}
    if family == "rollout":  # forward, adjoint and the two bases of the depth gradient of every step
        return {"bytes": (4 * 48.0 + 16.0) * n, "flops": 30.0 * n * case["tau_rho"] * 4 * case["steps"]}
    return fourier(case["nx"], case["ny"], case["real"], 2 if family == "autograd" else 1)


# ---- the same in FP64 with plain torch and numpy -------------------------------

# The rational fit of the Gaussian that REXII is built on (arXiv 2008.11607,
# Appendix A): mu and a_l, l = 0..24, a_{-l} = conj(a_l).
_MU = -5.133333333333333
_A = [
    -6.520430828919864e+01, 4.261818064131437e+01 + 2.761406741120911e+01j, -9.801650304425239e+00 - 2.189295463610722e+01j,
    -1.054225194693395e+00 + 6.791786454153551e+00j, 7.950505668209775e-01 - 8.904997258367445e-01j,
    -1.218558380859130e-01 + 3.321241563407446e-02j, 7.365401806949337e-03 + 2.212802103193251e-03j,
    -2.801087265991056e-04 - 5.566945197754387e-04j, 1.254835436432561e-04 - 2.467200513365371e-04j,
    2.295472292491263e-04 - 8.494118951459107e-05j, 1.858484460459430e-04 + 9.242889460185034e-05j,
    4.068056518449676e-05 + 1.653479957565515e-04j, -8.341508001647741e-05 + 1.045331460447588e-04j,
    -9.970528169841103e-05 - 5.856228484297677e-06j, -3.499639858693093e-05 - 6.129059473910835e-05j,
    2.295021920298455e-05 - 4.099832469456381e-05j, 2.931048772724314e-05 + 1.708815129697846e-07j,
    7.502088478301169e-06 + 1.525082051744077e-05j, -5.815291167450100e-06 + 6.919604247338349e-06j,
    -4.069948458364005e-06 - 1.440010113050771e-06j, 7.932524475429588e-08 - 1.794169428574330e-06j,
    6.120984882186265e-07 - 1.131894636585849e-07j, 5.531365159161319e-08 + 1.585749903175946e-07j,
    -2.867805871375946e-08 + 1.239499740327838e-08j, -1.143081277095316e-09 - 2.763239274253499e-09j,
]
_H = 0.5  # the parameter h of the plans


def _rexii(x, tau_rho):
    """REXII(i x) for a 1-D tensor of real x: sum_n (c1_n h mu + c2_n y) / ((h mu)^2 + y^2), y = x + h n."""
    c = 2.0 * math.sqrt(-math.log(math.sqrt(4.0 * math.pi) * TOL))
    M = math.ceil(tau_rho / _H) + math.ceil(c - 1.0)
    a = np.array([np.conj(v) for v in _A[:0:-1]] + _A, dtype=np.complex128)
    b = np.exp(-1j * _H * np.arange(-M, M + 1)) * math.exp(_H * _H)
    c1 = _H * np.convolve(a.real, b)  # n = -N..N, N = M + 24
    c2 = _H * np.convolve(a.imag, b)
    hmu, N = _H * _MU, M + 24
    out = torch.zeros(x.numel(), dtype=torch.complex128, device=x.device)
    span = max(1, min(64, (1 << 25) // max(1, x.numel())))
    for i in range(0, 2 * N + 1, span):
        n = torch.arange(i - N, min(i + span, 2 * N + 1) - N, dtype=torch.float64, device=x.device)
        A = torch.from_numpy(c1[i:i + span] * hmu).to(x.device)
        B = torch.from_numpy(c2[i:i + span]).to(x.device)
        y = x[:, None] + _H * n[None, :]
        r = 1.0 / (hmu * hmu + y * y)
        yr = y * r
        out += torch.complex(r @ A.real + yr @ B.real, r @ A.imag + yr @ B.imag)
    return out


def _half(n):
    t = torch.arange(n, device=_DEVICE, dtype=torch.float64) * (math.pi / n)
    return torch.cos(t), torch.sin(t)


def _omega2(nx, ny):
    """omega(k)^2 of the C-grid operator (H = g = f = 1, unit square), ky by kx."""
    (cx, sx), (cy, sy) = _half(nx), _half(ny)
    return ((2.0 * nx * sx) ** 2)[None, :] + ((2.0 * ny * sy) ** 2)[:, None] + (cx * cx)[None, :] * (cy * cy)[:, None]


def _rho_cgrid(nx, ny):
    return math.sqrt(_omega2(nx, ny).max().item())


def _spread(values, nx, ny, fold):
    """values on the folded wavenumbers (ny/2 + 1 by nx/2 + 1) at every wavenumber."""
    kx = torch.arange(nx, device=_DEVICE)
    ky = torch.arange(ny, device=_DEVICE)
    return values.reshape(fold)[torch.minimum(ky, ny - ky)[:, None], torch.minimum(kx, nx - kx)[None, :]]


def _exact_fourier(state, dt, tau_rho, real, adjoint=False):
    """r(dt A) state on the C grid (or its adjoint) through the FFT and the 3 x 3 symbol."""
    _, ny, nx = state.shape
    f = torch.fft.fft2(torch.complex(state.real, torch.zeros_like(state.real)) if real else state)
    fold = (ny // 2 + 1, nx // 2 + 1)
    w = torch.sqrt(_omega2(nx, ny)[:fold[0], :fold[1]]).reshape(-1)
    R = _rexii(dt * w, tau_rho)
    R0 = _rexii(torch.zeros(1, device=_DEVICE, dtype=torch.float64), tau_rho)[0]
    s1 = _spread(R.imag / w, nx, ny, fold)
    s2 = _spread((R0 - R.real) / (w * w), nx, ny, fold)
    (cx, sx), (cy, sy) = _half(nx), _half(ny)
    cx, sx, cy, sy = cx[None, :], sx[None, :], cy[:, None], sy[:, None]
    ax, ay = 2.0 * nx * sx, 2.0 * ny * sy
    one = torch.ones(ny, nx, device=_DEVICE, dtype=torch.float64)
    dxf, dxb = torch.complex(-ax * sx * one, ax * cx * one), torch.complex(ax * sx * one, ax * cx * one)
    dyf, dyb = torch.complex(-ay * sy * one, ay * cy * one), torch.complex(ay * sy * one, ay * cy * one)
    P = (cx * cy) * torch.complex(cx * cy + sx * sy, sx * cy - cx * sy)

    def apply(v):
        if not adjoint:
            return torch.stack([-(dxb * v[1] + dyb * v[2]), P * v[2] - dxf * v[0], -dyf * v[0] - P.conj() * v[1]])
        return torch.stack([-(dxf.conj() * v[1] + dyf.conj() * v[2]), -dxb.conj() * v[0] - P * v[2],
                            -dyb.conj() * v[0] + P.conj() * v[1]])

    if adjoint:
        R0, s2 = R0.conj(), s2.conj()
    g = apply(f)
    out = torch.fft.ifft2(R0 * f + s1 * g + s2 * apply(g))
    return torch.complex(out.real, torch.zeros_like(out.real)) if real else out


def _exact_scalar(state, tau_rho):
    """REXIE of i (d_xx + d_yy) with the midpoint shift (per eigenvalue it is REXII of the shifted argument)."""
    _, ny, nx = state.shape
    lam = -(((2.0 * nx * _half(nx)[1]) ** 2)[None, :] + ((2.0 * ny * _half(ny)[1]) ** 2)[:, None])
    lo, hi = lam.min().item(), lam.max().item()
    sigma = 0.5 * (lo + hi)
    dt = tau_rho / max(abs(lo - sigma), abs(hi - sigma))
    fold = (ny // 2 + 1, nx // 2 + 1)
    R = _spread(_rexii((dt * (lam - sigma))[:fold[0], :fold[1]].reshape(-1), tau_rho), nx, ny, fold)
    return torch.fft.ifft2(torch.fft.fft2(state) * R * complex(math.cos(dt * sigma), math.sin(dt * sigma)))


def _exponential(state, H, dt):
    """e^{dt A(H)} state for a real or complex state as a Chebyshev series
    sum_k (2 - [k = 0]) J_k(X) S_k, S_{k+1} = 2 (A / rho) S_k + S_{k-1}."""
    _, ny, nx = state.shape
    rho = math.sqrt(H.detach().max().item() * (4.0 * nx * nx + 4.0 * ny * ny)) + 1.0
    X = dt * rho
    m = 1 << max(9, math.ceil(math.log2(4.0 * X + 400.0)))
    J = np.fft.fft(np.exp(1j * X * np.sin(2.0 * math.pi * np.arange(m) / m))).real / m
    count = int(X + 12.0 * X ** (1.0 / 3.0) + 40.0)

    def A(v):
        e, u, w = v[0], v[1], v[2]
        east = lambda z: torch.roll(z, -1, -1)  # noqa: E731
        west = lambda z: torch.roll(z, 1, -1)  # noqa: E731
        north = lambda z: torch.roll(z, -1, -2)  # noqa: E731
        south = lambda z: torch.roll(z, 1, -2)  # noqa: E731
        de = -H * (nx * (u - west(u)) + ny * (w - south(w)))
        du = -nx * (east(e) - e) + 0.25 * (w + east(w) + south(w) + east(south(w)))
        dw = -ny * (north(e) - e) - 0.25 * (u + west(u) + north(u) + west(north(u)))
        return torch.stack([de, du, dw])

    old, cur = state, A(state) / rho
    out = J[0] * old + 2.0 * J[1] * cur
    for k in range(2, count):
        old, cur = cur, (2.0 / rho) * A(cur) + old
        out = out + 2.0 * J[k] * cur
    return out


def _complex(v):
    return torch.complex(v, torch.zeros_like(v))


def exact(case, seed):
    family = case["family"]
    if family == "batch":
        parts, by_size = [], {}
        for i, (nx, ny, t) in enumerate(_instances(case)):
            st = _field(dict(nx=nx, ny=ny, field="smooth" if case["real"] else "noise"), seed, 1 + i)
            y = _exact_fourier(st, t / _rho_cgrid(nx, ny), t, case["real"])
            by_size.setdefault((nx, ny), []).append(y.reshape(-1))
        for key in by_size:  # a batch lays instances of one size next to each other
            parts += by_size[key]
        return torch.cat(parts)
    nx, ny = case["nx"], case["ny"]
    if family in ("depth", "rollout"):
        H = _depth_field(nx, ny, seed)
        rho = math.sqrt(H.max().item() * (4.0 * nx * nx + 4.0 * ny * ny)) + 1.0
        dt = case["tau_rho"] / rho
        real = case.get("real", True)
        st = _field(dict(case, field="smooth" if real else "noise"), seed)
        if family == "depth":
            return _complex(_exponential(st.real.contiguous(), H, dt)) if real else _exponential(st, H, dt)
        g = _smooth(nx, ny, _generator(seed, 5))
        x = st.real.contiguous().requires_grad_(True)
        H.requires_grad_(True)
        y = x
        for _ in range(case["steps"]):
            y = checkpoint(_exponential, y, H, dt, use_reentrant=False)
        gs, gd = torch.autograd.grad((y[0] * g).sum(), (x, H))
        return {"out": _complex(y.detach()), "grad_state": _complex(gs), "grad_depth": gd}
    st = _field(case, seed)
    if family == "scalar":
        return _exact_scalar(st, case["tau_rho"])
    dt = case["tau_rho"] / _rho_cgrid(nx, ny)
    out = _exact_fourier(st, dt, case["tau_rho"], case["real"])
    if family == "autograd":
        gout = _field(dict(case, field="noise"), seed, 9)
        return {"out": out, "grad_state": _exact_fourier(gout, dt, case["tau_rho"], case["real"], adjoint=True)}
    return out.cpu() if family == "host" else out
