"""Workload cases of the thin-film solver: what its users run, at the sizes they
run it, each through the public entry points of the package.

A case is one call on one kind of film:

  step       tf_newton_adi_step, one time step of one film (the Newton loop
             until max|v/u| < 1e-10), the unit of work of every simulation
  advance    tf_advance, a stretch of an adaptive run from a copy of the film
  ensemble   tf_ensemble_advance, many films of uneven sizes at once
  residual   tf_residual, G and its norms for two films
  adjoint    tf_adjoint_step, the reverse of a fixed-iteration step
  gradient   tf_tape_forward + tf_tape_backward, the gradient of a trajectory
  spectrum   tf_spectrum_run, the radial Fourier analysis of a film

Films: "noise" is a flat film with 1% noise per cell (the start of every
spinodal run), "pattern" a film of cosine modes about the fastest growing
wavenumber, 5% of the height (a run under way).  `cells` is the resolution in
cells per fastest growing wavelength: 16 to 128 in the repository's workloads.
`dt` is the step in the units in which the Newton loop's cost does not depend
on the resolution: ds^4 / f0 for noise (1e-3 takes about five iterations), 1 /
sigma_max for patterns.

A step's film comes back with its status and iteration count, mass and least
height.  The err and gnorm that the calls also report are left out: after a
converged step they hold what the tolerance left over.
"""
import math

import numpy as np
import torch

import paper_1806_10550_gb300 as tf

B = 0.1  # precursor scale of the power law (and of the polymer film)
PRECISION = {"fp64": tf.TF_FP64, "fp32": tf.TF_FP32_BULK}
SOLVER = {"twisted": tf.TF_SOLVER_TWISTED, "partitioned": tf.TF_SOLVER_PARTITIONED}
# model -> (number, C, b, flat height)
MODEL = {"power": (tf.TF_MODEL_POWERLAW, 1.0, B, 1.0), "nlc": (tf.TF_MODEL_NLC, 0.0857, 0.01, 0.5),
         "polymer": (tf.TF_MODEL_POLYMER, 0.00581, B, 3.9)}


def _step(nx, ny, precision="fp32", film="noise", cells=64, dt=1e-3, model="power", solver="twisted", **name):
    return dict(**name, call="step", nx=nx, ny=ny, precision=precision, film=film, cells=cells, dt=dt, model=model,
                solver=solver)


def listed():
    return [
        # one step of the small parity film: all launch latency and short chains
        _step(64, 64, cells=16, name="step_64"),
        # a film of a parameter study cut to an odd size: unaligned rows, ragged ends of lines and tiles
        _step(1023, 769, cells=32, film="pattern", dt=2.5e-3, name="step_ragged"),
        # the medium single film (the run to rupture of the scaling study)
        _step(2048, 2048, cells=32, name="step_2048"),
        # the benchmark film, 64 wavelengths at 128 cells each
        _step(8192, 8192, cells=128, name="step_8192"),
        # every operation in double precision: the mode runs are checked against
        _step(1024, 1024, precision="fp64", name="step_1024_fp64"),
        # a liquid-crystal film (the other mobility models take the general path)
        _step(1024, 1024, model="nlc", cells=128, name="step_1024_nlc"),
        # the start of an adaptive run of a small film in double precision
        dict(name="advance_64_fp64", call="advance", nx=64, ny=64, precision="fp64", cells=16, dt=1e-4, attempts=12),
        # statistics over many films: uneven sizes and contact angles, each with its own controller
        dict(name="ensemble_24", call="ensemble", films=24, least=128, most=1024, cells=32, attempts=4),
        # the residual of an iterate, for monitoring and for callers' own solvers
        dict(name="residual_2048", call="residual", nx=2048, ny=2048, precision="fp32", cells=64, dt=1e-3),
        # the reverse of one step (an optimiser's inner call)
        dict(name="adjoint_512", call="adjoint", nx=512, ny=512, cells=64, dt=1.1e-2, K=3),
        # the gradient of a loss on the film after some steps, in the film and the contact angle
        dict(name="gradient_256", call="gradient", nx=256, ny=256, cells=64, dt=1.1e-2, K=3, steps=9),
        # the dominant wavenumber with every stage of the analysis (a plotted spectrum)
        dict(name="spectrum_4096", call="spectrum", nx=4096, ny=4096, cells=64),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _sizes(rng, lo, hi, most):
    """nx and ny, each over the logarithm of lo..hi, nx ny at most `most`: odd sizes, and every third time a multiple of 32."""
    nx = _log_int(rng, lo, hi)
    ny = _log_int(rng, lo, min(hi, max(lo, most // nx)))
    if rng.random() < 1 / 3:
        nx, ny = max(lo, nx // 32 * 32), max(lo, ny // 32 * 32)
    return nx, ny


def draw(rng):
    kind = rng.choice(["step"] * 7 + ["advance", "ensemble", "residual", "adjoint", "gradient", "spectrum"])
    cells = rng.choice([16, 32, 64, 128])
    if kind == "step":
        film = rng.choice(["noise", "pattern"])
        dt = rng.uniform(3e-4, 1.5e-3) if film == "noise" else rng.uniform(1e-3, 4e-3)
        model = rng.choice(["power"] * 8 + ["nlc", "polymer"])
        if model != "power":  # the noise and steps of the model workloads
            nx, ny = _sizes(rng, 64, 2048, 2048 * 1024)
            return _step(nx, ny, model=model, cells=128, dt=rng.uniform(3e-4, 1.2e-3))
        precision = rng.choice(["fp32"] * 3 + ["fp64"])
        nx, ny = _sizes(rng, 64, 8192, 8192 * 8192) if precision == "fp32" else _sizes(rng, 64, 2048, 1024 * 1024)
        solver = "twisted"
        if precision == "fp32" and nx * ny <= 2048 * 2048 and rng.random() < 0.2:
            solver = "partitioned"
        return _step(nx, ny, precision, film, cells, dt, model, solver)
    if kind == "advance":
        precision = rng.choice(["fp32", "fp64"])
        nx, ny = _sizes(rng, 32, 512, 512 * 256)
        return dict(call="advance", nx=nx, ny=ny, precision=precision, cells=cells, dt=rng.uniform(5e-5, 4e-4),
                    attempts=rng.randint(4, 14))
    if kind == "ensemble":
        least = rng.choice([96, 128, 200])
        return dict(call="ensemble", films=rng.randint(8, 24), least=least, most=rng.choice([512, 768, 1024]), cells=32,
                    attempts=rng.randint(2, 4))
    if kind == "residual":
        nx, ny = _sizes(rng, 64, 4096, 4096 * 2048)
        return dict(call="residual", nx=nx, ny=ny, precision=rng.choice(["fp32", "fp32", "fp64"]), cells=cells, dt=rng.uniform(3e-4, 1e-2))
    if kind == "adjoint":
        nx, ny = _sizes(rng, 48, 1024, 512 * 512)
        return dict(call="adjoint", nx=nx, ny=ny, cells=64, dt=rng.uniform(5e-3, 1.1e-2), K=rng.randint(2, 4))
    if kind == "gradient":
        nx, ny = _sizes(rng, 48, 512, 256 * 256)
        return dict(call="gradient", nx=nx, ny=ny, cells=64, dt=rng.uniform(5e-3, 1.1e-2), K=rng.randint(2, 3), steps=rng.randint(2, 9))
    nx, ny = 1 << rng.randint(8, 13), 1 << rng.randint(8, 12)
    return dict(call="spectrum", nx=nx, ny=ny, cells=rng.choice([32, 64, 128]))


# ---- the films and parameters that a program has in hand ------------------------


def _dpi(model, kappa, b, h):
    """Pi'(h) of a model's disjoining pressure, for a torch tensor h."""
    if model == "power":
        return kappa * (2 * b ** 2 / h ** 3 - 3 * b ** 3 / h ** 4)
    if model == "nlc":  # K[(b/h)^3 - (b/h)^2] + (N/2)(m/h)^2, m = g h^2/(h^2 + beta^2), g = [1 + tanh((h - 2b)/w)]/2
        K, N, beta2, w = 36.0, 1.67, 1.0, 0.05
        t = torch.tanh((h - 2 * b) / w)
        g, dg = (1 + t) / 2, (1 - t * t) / (2 * w)
        d = h * h + beta2
        q, dq = g * h / d, dg * h / d + g * (beta2 - h * h) / d ** 2
        return K * (2 * b ** 2 / h ** 3 - 3 * b ** 3 / h ** 4) + N * q * dq
    cp, a1, a2, d = 1.181, 41.25, -243.75, 191.0  # polymer on SiOx / Si
    return -72 * cp / h ** 10 + a1 / (2 * math.pi * h ** 4) - (a1 - a2) / (2 * math.pi * (h + d) ** 4)


def _geometry(model, cells, theta_c=math.radians(20.0)):
    """kappa, spacing, the most unstable wavenumber and its growth rate, and f0 of the flat film."""
    _, C, b, h0 = MODEL[model]
    kappa = (1 - math.cos(theta_c)) / (b * 0.5)
    f0 = C * h0 ** 3
    f1 = h0 ** 3 * float(_dpi(model, kappa, b, torch.tensor(h0, dtype=torch.float64)))
    qm, sm = math.sqrt(f1 / (2 * f0)), f1 * f1 / (4 * f0)
    return dict(kappa=kappa, ds=2 * math.pi / qm / cells, qm=qm, sm=sm, f0=f0)


def _dt(c, g):
    return c["dt"] / g["sm"] if c.get("film") == "pattern" else c["dt"] * g["ds"] ** 4 / g["f0"]


def _noise(gen, nx, ny, h0, eps=0.01):
    return h0 * (1 + eps * (2 * torch.rand((ny, nx), generator=gen, dtype=torch.float64, device="cuda") - 1))


def _pattern(gen, nx, ny, ds, qm, h0, eps=0.05, modes=32):
    """Cosine modes that the no-flux walls allow, wavenumbers within a few per cent of qm."""
    r = lambda: torch.rand(modes, generator=gen, dtype=torch.float64, device="cuda")  # noqa: E731
    k, ang = qm * (1 + 0.15 * (r() - 0.5)), 0.5 * math.pi * r()
    p = torch.round(k * torch.cos(ang) * nx * ds / math.pi)
    q = torch.round(k * torch.sin(ang) * ny * ds / math.pi)
    x = (torch.arange(nx, dtype=torch.float64, device="cuda") + 0.5) * math.pi / nx
    y = (torch.arange(ny, dtype=torch.float64, device="cuda") + 0.5) * math.pi / ny
    f = torch.cos(q[:, None] * y).T @ ((2 * r() - 1)[:, None] * torch.cos(p[:, None] * x))
    return (h0 * (1 + eps * f / f.abs().max().clamp_min(1e-30))).contiguous()


def _params(c, g, nx, ny, **more):
    model, C, b, _ = MODEL[c.get("model", "power")]
    return tf.tf_params_default(nx=nx, ny=ny, ds=g["ds"], model=model, cap_C=C, b=b, precision=PRECISION[c.get("precision", "fp64")],
                                line_solver=SOLVER[c.get("solver", "twisted")], dt_max=0.01 / g["sm"], **more)


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _film(c, g, gen):
    h0 = MODEL[c.get("model", "power")][3]
    if c.get("film") == "pattern":
        return _pattern(gen, c["nx"], c["ny"], g["ds"], g["qm"], h0)
    return _noise(gen, c["nx"], c["ny"], h0)


def _shapes(c):
    """(nx, ny, contact angle) of an ensemble's films: sides over the logarithm of least..most, half of them
    square powers of two as in the statistics runs, angles of 10 to 40 degrees; the same for every seed."""
    rng, out = np.random.default_rng(c["films"] * 1000 + c["most"]), []
    for i in range(c["films"]):
        n = 2 ** int(rng.integers(math.ceil(math.log2(c["least"])), int(math.log2(c["most"])) + 1))
        a, b = (int(math.exp(rng.uniform(math.log(c["least"]), math.log(c["most"])))) for _ in range(2))
        out.append((*((n, n) if i % 2 == 0 else (a, b)), math.radians(float(rng.uniform(10.0, 40.0)))))
    return out


def _ensemble(c, seed):
    """(nx, ny, geometry, film) of each film."""
    gen = _gen(seed)
    return [(nx, ny, _geometry("power", c["cells"], th), _noise(gen, nx, ny, 1.0)) for nx, ny, th in _shapes(c)]


def _residual_films(c, seed):
    gen, g = _gen(seed), _geometry("power", c["cells"])
    old = _noise(gen, c["nx"], c["ny"], 1.0)
    return g, old, old * (1 + 1e-4 * torch.randn(old.shape, generator=gen, dtype=torch.float64, device="cuda"))


def _reverse_films(c, seed):
    """The film and the cotangent of its final state (twice the misfit to another film)."""
    gen, g = _gen(seed), _geometry("power", c["cells"])
    h = _noise(gen, c["nx"], c["ny"], 1.0)
    return g, h, 2 * (h - _noise(gen, c["nx"], c["ny"], 1.0))


def _spectrum_film(c, seed):
    gen, g = _gen(seed), _geometry("power", c["cells"])
    h = _pattern(gen, c["nx"], c["ny"], g["ds"], g["qm"], 1.0, modes=128)
    return g, h + 0.002 * (2 * torch.rand(h.shape, generator=gen, dtype=torch.float64, device="cuda") - 1)


THETA_C = math.radians(20.0)


def prepare(c, seed):
    call = c["call"]
    if call == "ensemble":
        films = _ensemble(c, seed)
        torch.cuda.synchronize()  # the films' own streams start behind their inputs
        streams = [torch.cuda.Stream() for _ in films]
        ctxs = [tf.Context(tf.tf_params_default(nx=nx, ny=ny, ds=g["ds"], kappa=g["kappa"], dt_max=0.01 / g["sm"], precision=tf.TF_FP32_BULK),
                           stream=s) for (nx, ny, g, _), s in zip(films, streams)]
        return dict(c=c, ctxs=ctxs, streams=streams, h0=[f[3] for f in films], h=[torch.empty_like(f[3]) for f in films],
                    dt0=[1e-7 / f[2]["sm"] for f in films])
    if call == "residual":
        g, old, cur = _residual_films(c, seed)
        ctx = tf.Context(_params(c, g, c["nx"], c["ny"], kappa=g["kappa"]))
        return dict(c=c, ctx=ctx, h=cur, old=old, G=torch.empty_like(old), dt=_dt(c, g))
    if call in ("adjoint", "gradient"):
        g, h, cot = _reverse_films(c, seed)
        ctx = tf.Context(_params(c, g, c["nx"], c["ny"], contact_angle=THETA_C))
        s = dict(c=c, ctx=ctx, h=h, cot=cot, out=torch.empty_like(h), gh=torch.empty_like(h), dt=_dt(c, g))
        if call == "gradient":
            s["tape"] = tf.tf_tape_create(ctx, c["steps"], c["K"], s["dt"])
        return s
    if call == "spectrum":
        g, h = _spectrum_film(c, seed)
        sp = tf.tf_spectrum_params_default(H0=1.0, q_cut=5 * g["qm"])
        return dict(c=c, plan=tf.tf_spectrum_plan_create(c["nx"], c["ny"], g["ds"], sp), h=h)
    g = _geometry(c.get("model", "power"), c["cells"])
    h = _film(c, g, _gen(seed))
    ctx = tf.Context(_params(c, g, c["nx"], c["ny"], kappa=g["kappa"]))
    return dict(c=c, ctx=ctx, h=h, out=torch.empty_like(h), dt=_dt(c, g))


def run(s):
    c = s["c"]
    call = c["call"]
    if call == "step":
        i = tf.tf_newton_adi_step(s["ctx"], s["h"], s["out"], s["dt"])
        return dict(h=s["out"], status=i["status"], iterations=i["iterations"], mass=i["mass"], hmin=i["hmin"])
    if call == "advance":
        s["out"].copy_(s["h"])
        i, rec = tf.tf_advance(s["ctx"], s["out"], 0.0, 1e30, s["dt"], c["attempts"])
        cols = {k: np.array([r[k] for r in rec]) for k in ("t", "dt", "accepted", "iterations", "status", "mass", "hmin")}
        return dict(h=s["out"], info=i, records=cols)
    if call == "ensemble":
        for h, h0, st in zip(s["h"], s["h0"], s["streams"]):
            with torch.cuda.stream(st):
                h.copy_(h0)
        infos = tf.tf_ensemble_advance(s["ctxs"], s["h"], 0.0, 1e30, s["dt0"], c["attempts"])
        return dict(h=s["h"], info={k: np.array([i[k] for i in infos]) for k in infos[0]})
    if call == "residual":
        n = tf.tf_residual(s["ctx"], s["h"], s["old"], s["dt"], s["G"])
        return dict(G=s["G"], gnorm=n["gnorm"], mass=n["mass"], hmin=n["hmin"])
    if call == "adjoint":
        r = tf.tf_adjoint_step(s["ctx"], s["h"], s["dt"], c["K"], s["cot"], g_h=s["gh"], h_new=s["out"])
        return dict(h=r["h_new"], g_h=r["g_h"], g_kappa=r["g_kappa"], g_theta=r["g_theta"])
    if call == "gradient":
        h = tf.tf_tape_forward(s["tape"], s["h"], s["out"])
        r = tf.tf_tape_backward(s["tape"], s["cot"], s["gh"])
        return dict(h=h, g_h=r["g_h0"], g_kappa=r["g_kappa"], g_theta=r["g_theta"])
    return tf.tf_spectrum_run(s["plan"], s["h"], peak_cap=8)


# Floating-point operations per cell: the residual (mobilities, Laplacian, four
# faces, divergence), a line system (its band rows and its elimination), and the
# reverse of an iteration (two transposed solves, two line products, one of D).
RESIDUAL, LINE, REVERSE = 45, 60, 260
ITERATIONS = 5  # of a step, about


def work(c):
    call = c["call"]
    if call == "ensemble":
        cells = sum(nx * ny for nx, ny, _ in _shapes(c))
        return dict(bytes=16 * cells, flops=cells * c["attempts"] * ITERATIONS * (RESIDUAL + 2 * LINE))
    cells = c["nx"] * c["ny"]
    iteration = RESIDUAL + 2 * LINE
    if call == "step":
        return dict(bytes=16 * cells, flops=cells * ITERATIONS * iteration)
    if call == "advance":
        return dict(bytes=16 * cells, flops=cells * c["attempts"] * ITERATIONS * iteration)
    if call == "residual":
        return dict(bytes=24 * cells, flops=cells * 2 * RESIDUAL)
    if call == "adjoint":
        return dict(bytes=32 * cells, flops=cells * c["K"] * (iteration + REVERSE))
    if call == "gradient":
        return dict(bytes=32 * cells, flops=cells * c["steps"] * c["K"] * (iteration + REVERSE))
    return dict(bytes=8 * cells, flops=cells * 2.5 * (math.log2(c["nx"]) + math.log2(c["ny"]) / 8))


# ---- the same in plain torch, 64 bits --------------------------------------------


def _diff(u, d):
    """u at the next cell along d less u, over the inner faces."""
    return u[:, 1:] - u[:, :-1] if d == 1 else u[1:] - u[:-1]


def _pad(F, d):
    """Differences of face values over the cells, no flux through the walls."""
    z = F.new_zeros((F.shape[0], 1) if d == 1 else (1, F.shape[1]))
    return torch.diff(torch.cat([z, F, z], d), dim=d)


def _lap(u, ds):
    return (_pad(_diff(u, 1), 1) + _pad(_diff(u, 0), 0)) / ds ** 2


def _mean(f, d):
    return (f[:, 1:] + f[:, :-1]) / 2 if d == 1 else (f[1:] + f[:-1]) / 2


def _D(u, model, kappa, ds):
    """div[f0 grad lap u + f1 grad u] in flux form."""
    _, C, b, _ = MODEL[model]
    f0, f1, L = C * u ** 3, u ** 3 * _dpi(model, kappa, b, u), _lap(u, ds)
    return sum(_pad((_mean(f0, d) * _diff(L, d) + _mean(f1, d) * _diff(u, d)) / ds, d) / ds for d in (1, 0))


def _dct(x):
    """DCT-II sums along the last axis, by one FFT of the reordered line."""
    n = x.shape[-1]
    V = torch.fft.fft(torch.cat([x[..., ::2], x[..., 1::2].flip(-1)], -1))
    k = torch.arange(n, dtype=torch.float64, device=x.device) * (-math.pi / (2 * n))
    return V.real * torch.cos(k) - V.imag * torch.sin(k)


def _idct(X):
    n = X.shape[-1]
    k = torch.arange(n, dtype=torch.float64, device=X.device) * (math.pi / (2 * n))
    Y = torch.cat([torch.zeros_like(X[..., :1]), X[..., 1:].flip(-1)], -1)
    v = torch.fft.ifft(torch.complex(X * torch.cos(k) + Y * torch.sin(k), X * torch.sin(k) - Y * torch.cos(k))).real
    x = torch.empty_like(X)
    x[..., ::2], x[..., 1::2] = v[..., : (n + 1) // 2], v[..., (n + 1) // 2:].flip(-1)
    return x


def _implicit_step(u0, model, g, dt):
    """The root u of u + dt/2 D(u) = u0 - dt/2 D(u0): Newton corrections with the flat film's operator, which the cosine modes
    diagonalise, down to rounding."""
    ny, nx = u0.shape
    ds, kappa = g["ds"], g["kappa"]
    _, C, b, _ = MODEL[model]
    lam = [-(2 / ds * torch.sin(torch.arange(n, dtype=torch.float64, device=u0.device) * (math.pi / (2 * n)))) ** 2 for n in (nx, ny)]
    m = u0.mean()
    L = lam[1][:, None] + lam[0]
    P = 1 + dt / 2 * (C * m ** 3 * L + m ** 3 * _dpi(model, kappa, b, m)) * L
    rhs, u, before = u0 - dt / 2 * _D(u0, model, kappa, ds), u0.clone(), math.inf
    for _ in range(80):
        r = u + dt / 2 * _D(u, model, kappa, ds) - rhs
        e = _idct(_idct((_dct(_dct(r).T).T / P)).T).T
        u = u - e
        size = float(e.abs().max())
        if size < 1e-15 or (size < 1e-12 and size > before / 2):
            break
        before = size
    return u


def _adi_step(u0, kappa, ds, dt, K):
    """K pseudo-Newton ADI iterations, dense line systems (x lines, then y lines); differentiable."""
    _, C, b, _ = MODEL["power"]
    c = 0.5 * dt
    rhs = u0 - c * _D(u0, "power", kappa, ds)
    u = u0
    for _ in range(K):
        f0, f1, L = C * u ** 3, u ** 3 * _dpi("power", kappa, b, u), _lap(u, ds)
        d0, d1 = 3 * C * u ** 2, kappa * 3 * b ** 3 / u ** 2
        x = -(u + c * _D(u, "power", kappa, ds) - rhs)
        for d in (1, 0):
            t = (lambda a: a) if d == 1 else (lambda a: a.T)  # lines along the last axis
            U, LL, F0, F1, D0, D1 = (t(a) for a in (u, L, f0, f1, d0, d1))
            n = U.shape[1]
            Df = torch.diff(torch.eye(n, dtype=u.dtype, device=u.device), dim=0) / ds  # faces x cells
            Ll = -Df.T @ Df  # along-line second difference with walls
            dL, dU = _diff(LL, 1) / ds, _diff(U, 1) / ds
            J = _mean(F0, 1)[:, :, None] * (Df @ Ll) + _mean(F1, 1)[:, :, None] * Df
            M = torch.abs(Df) * ds / 2  # mean of a face's two cells
            J = J + M * (dL[:, :, None] * D0[:, None, :] + dU[:, :, None] * D1[:, None, :])
            A = torch.eye(n, dtype=u.dtype, device=u.device) - c * (Df.T @ J)
            x = t(torch.linalg.solve(A, t(x)[:, :, None])[:, :, 0])
        u = u + x
    return u


def _exact_reverse(c, seed):
    g, h, cot = _reverse_films(c, seed)
    steps, n = c.get("steps", 1), max(c["nx"], c["ny"])
    if steps * c["K"] * c["nx"] * c["ny"] * n > 5e8:
        return None  # the dense line systems of the reverse take too long
    h = h.requires_grad_()
    kappa = torch.tensor(g["kappa"], dtype=torch.float64, device="cuda", requires_grad=True)
    u, dt = h, _dt(c, g)
    for _ in range(steps):
        u = _adi_step(u, kappa, g["ds"], dt, c["K"])
    gh, gk = torch.autograd.grad(u, (h, kappa), cot)
    return dict(h=u.detach(), g_h=gh, g_kappa=float(gk), g_theta=float(gk) * math.sin(THETA_C) / (B * 0.5))


def _exact_spectrum(c, seed):
    g, h = _spectrum_film(c, seed)
    nx, ny, ds, cut, ppi, n_eval = c["nx"], c["ny"], g["ds"], 5 * g["qm"], 10, 400
    w = math.gcd(nx, ny)
    ax, ay, scale = ny // w, nx // w, math.pi * w / (ds * nx * ny)
    keycut = math.floor((cut / scale) ** 2)
    n_p, n_q = min(nx, math.isqrt(keycut) // ax + 1), min(ny, math.isqrt(keycut) // ay + 1)
    A = (_dct(_dct(h - 1.0).T).T.abs() / (nx * ny)).cpu().numpy()
    # Gaussian over the wave indices, the spectrum of the reflected film outside them
    G = np.exp(-np.arange(-3, 4) ** 2 / 2.0)
    G /= G.sum()

    def smooth(a, n, m):  # along axis 0
        out = 0.0
        for k in range(-3, 4):
            i = np.mod(np.arange(m) + k, 2 * n)
            j = np.where(i < n, i, 2 * n - i)
            out = out + G[k + 3] * np.where((i == n)[:, None], 0.0, a[np.minimum(j, n - 1)])
        return out

    S = smooth(smooth(A[: min(ny, n_q + 3)].T, nx, n_p).T, ny, n_q)
    key = (np.arange(n_p) * ax)[None, :].astype(np.int64) ** 2 + (np.arange(n_q) * ay)[:, None].astype(np.int64) ** 2
    keys, at, count = np.unique(key[key <= keycut], return_inverse=True, return_counts=True)
    rq, rv = scale * np.sqrt(keys.astype(np.float64)), np.bincount(at.reshape(-1), weights=S[key <= keycut]) / count
    K = max(1, -(-(len(rq) - 1) // ppi))
    t = np.concatenate([[0.0], rq[ppi * np.arange(1, K)], [cut]])
    j = np.minimum(np.arange(len(rq)) // ppi, K - 1)
    s = (rq - t[j]) / (t[j + 1] - t[j])
    dg, of, rh = np.zeros(K + 1), np.zeros(K + 1), np.zeros(K + 1)
    np.add.at(dg, j, (1 - s) ** 2), np.add.at(dg, j + 1, s ** 2), np.add.at(of, j, s * (1 - s))
    np.add.at(rh, j, (1 - s) * rv), np.add.at(rh, j + 1, s * rv)
    a = np.zeros(K + 1)
    for i in range(2, K + 1):  # tridiagonal, unknowns 1..K
        f = of[i - 1] / dg[i - 1]
        dg[i] -= f * of[i - 1]
        rh[i] -= f * rh[i - 1]
    a[K] = rh[K] / dg[K]
    for i in range(K - 1, 0, -1):
        a[i] = (rh[i] - of[i] * a[i + 1]) / dg[i]
    q = cut * np.arange(n_eval) / (n_eval - 1)
    y = np.interp(q, t, a)
    for p in (3, 2, 1):
        y = np.array([y[max(0, e - p): e + p + 1].mean() for e in range(n_eval)])
    return dict(amplitude=A[:n_q, :n_p], smoothed=S, radial_q=rq, radial_value=rv, node_q=t, node_value=a, curve_q=q, curve_value=y)


def exact(c, seed):
    call = c["call"]
    if call == "spectrum":
        return _exact_spectrum(c, seed)
    if call in ("adjoint", "gradient"):
        return _exact_reverse(c, seed)
    if call == "residual":
        g, old, cur = _residual_films(c, seed)
        half = _dt(c, g) / 2
        G = cur + half * _D(cur, "power", g["kappa"], g["ds"]) - (old - half * _D(old, "power", g["kappa"], g["ds"]))
        return dict(G=G, gnorm=float(G.abs().max()), mass=float(cur.sum()), hmin=float(cur.min()))
    if call == "ensemble":
        return dict(h=[_attempts(h, g, 1e-7 / g["sm"], c["attempts"])[0] for _, _, g, h in _ensemble(c, seed)], info=None)
    model = c.get("model", "power")
    g = _geometry(model, c["cells"])
    h = _film(c, g, _gen(seed))
    if call == "step":
        u = _implicit_step(h, model, g, _dt(c, g))
        return dict(h=u, mass=float(u.sum()), hmin=float(u.min()))
    u, cols = _attempts(h, g, _dt(c, g), c["attempts"])
    return dict(h=u, info=None, records=cols)


def _attempts(h, g, dt, attempts):
    """Accepted steps of the adaptive run: a quarter more after every five, at most 0.01 / sigma_max."""
    cols, t = {k: [] for k in ("t", "dt", "mass", "hmin")}, 0.0
    for a in range(attempts):
        h = _implicit_step(h, "power", g, dt)
        for k, v in zip(cols, (t, dt, float(h.sum()), float(h.min()))):
            cols[k].append(v)
        t += dt
        if (a + 1) % 5 == 0:
            dt = min(dt * 1.25, 0.01 / g["sm"])
    return h, {k: np.array(v) for k, v in cols.items()}
