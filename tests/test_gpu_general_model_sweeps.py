"""The line sweeps of the models other than the (3, 2) power law at the edges
of their block shapes, and films at any 8-byte address.

A sweep over n lines of these models runs in blocks of 4 lines up to 608 (FP64)
or 1216 (FP32-bulk), of 8 up to 1216 or 2432, of 16 up to 2432 in FP64 and
beyond 2432 in FP32-bulk, and of 32 beyond 2432 in FP64.  One Newton iteration
is compared with the FP64 oracle to each side of every edge, with short lines
across, at the tolerances of the models' iteration parity.
"""
import math

import numpy as np
import pytest

import oracle as O
import paper_1806_10550_gb300 as tf
from paper_1806_10550_gb300 import synthetic as S

pytestmark = pytest.mark.gpu

KAPPA = 1.2061475842818314
EDGES = [(608, 24), (609, 50), (1216, 7), (1217, 77), (2432, 49), (2433, 25)]
MODELS = {  # model, its parameters, flat height
    "nlc": (tf.TF_MODEL_NLC, O.MODEL_NLC, dict(cap_C=0.0857, b=0.01), 0.5),
    "polymer": (tf.TF_MODEL_POLYMER, O.MODEL_POLYMER, dict(cap_C=0.00581, b=0.1), 3.9),
    "power43": (tf.TF_MODEL_POWERLAW, O.MODEL_POWERLAW, dict(n=4, m=3, kappa=KAPPA), 1.0),
}


@pytest.fixture(scope="module")
def torch():
    import torch as T
    if not T.cuda.is_available():
        pytest.skip("no CUDA device")
    tf.library()
    return T


def setup(which, nx, ny, mode):
    gm, om_id, kw, h0 = MODELS[which]
    qm, wm = O.lsa(O.Model(nx=4, ny=4, ds=1.0, model=om_id, **kw), h0)
    ds = 2 * math.pi / qm / 8
    return (O.Model(nx=nx, ny=ny, ds=ds, model=om_id, **kw),
            tf.tf_params_default(nx=nx, ny=ny, ds=ds, model=gm, precision=mode, **kw), h0, wm)


@pytest.mark.parametrize("which", list(MODELS))
@pytest.mark.parametrize("mode", [tf.TF_FP64, tf.TF_FP32_BULK])
@pytest.mark.parametrize("lines,n", EDGES)
@pytest.mark.parametrize("along_x", [True, False])
def test_iteration_at_block_shape_edges(torch, which, mode, lines, n, along_x):
    nx, ny = (n, lines) if along_x else (lines, n)
    om, p, h0, wm = setup(which, nx, ny, mode)
    dt = 0.001 / wm
    h_old = S.spinodal_film(nx, ny, h0, 0.02, seed=11 * nx + ny)
    ctx = tf.Context(p)
    w, v, hn = (torch.empty((ny, nx), dtype=torch.float64, device="cuda") for _ in range(3))
    hk = torch.from_numpy(h_old).cuda()
    tf.tf_newton_iteration(ctx, hk, hk, dt, hn, w=w, v=v)
    r = O.newton_iteration(om, h_old, O.explicit_part(om, h_old, dt), dt)
    tol = 1e-11 if mode == tf.TF_FP64 else 2e-4
    sw, sv = np.max(np.abs(r["w"])), np.max(np.abs(r["v"]))
    assert np.max(np.abs(w.cpu().numpy() - r["w"])) <= tol * sw
    assert np.max(np.abs(v.cpu().numpy() - r["v"])) <= tol * sv
    assert np.max(np.abs(hn.cpu().numpy() - r["unew"])) <= 1e-14 * h0 + tol * sv
    ctx.close()


@pytest.mark.parametrize("which", list(MODELS))
@pytest.mark.parametrize("mode", [tf.TF_FP64, tf.TF_FP32_BULK])
@pytest.mark.parametrize("films", [8, 30, 64])
def test_films_at_once_equal_films_alone(torch, which, mode, films):
    """1600, 6000 and 12800 lines at once."""
    params = []
    for i in range(films):
        _, p, h0, wm = setup(which, 200 - (i % 3), 170 + (i % 2), mode)
        params.append(p)
    dt = 0.001 / wm
    start = [torch.from_numpy(S.spinodal_film(p.nx, p.ny, h0, 0.01, seed=50 + i)).cuda() for i, p in enumerate(params)]
    torch.cuda.synchronize()
    ctxs = [tf.Context(p, stream=torch.cuda.Stream()) for p in params]
    grids = [h.clone() for h in start]
    torch.cuda.synchronize()
    tf.tf_ensemble_advance(ctxs, grids, 0.0, 1e30, [dt] * films, 2)
    for p, h, g in zip(params[:3], start, grids):
        ctx = tf.Context(p)
        tf.tf_advance(ctx, h, 0.0, 1e30, dt, 2)
        assert torch.equal(h, g)
        ctx.close()
    for c in ctxs:
        c.close()


@pytest.mark.parametrize("mode", [tf.TF_FP64, tf.TF_FP32_BULK])
@pytest.mark.parametrize("nx,ny", [(96, 80), (48, 700), (700, 48), (48, 1300), (1300, 48), (48, 2500), (2500, 48)])
def test_films_at_an_8_byte_address(torch, mode, nx, ny):
    """Grids whose address is a multiple of 8 and not of 16: the tile copies
    by elements, with the results of the vector copies, bit for bit."""
    ds, dt = 3.9, 1.0
    p = tf.tf_params_default(nx=nx, ny=ny, ds=ds, kappa=KAPPA, precision=mode)
    h = torch.from_numpy(S.spinodal_film(nx, ny, 1.0, 0.01, seed=nx + ny)).cuda()
    ctx = tf.Context(p)

    def grid(offset):
        g = torch.zeros(nx * ny + 2, dtype=torch.float64, device="cuda")[offset:offset + nx * ny].view(ny, nx)
        assert g.data_ptr() % 16 == 8 * (offset % 2)
        return g
    got = []
    for offset in (0, 1):
        h0, h1, G, w, v = (grid(offset) for _ in range(5))
        h0.copy_(h)
        info = tf.tf_newton_adi_step(ctx, h0, h1, dt)
        norms = tf.tf_residual(ctx, h1, h0, dt, G)
        it = tf.tf_newton_iteration(ctx, h0, h0, dt, h1.clone() if offset == 0 else grid(1), w=w, v=v)
        got.append((info, norms, it, h1, G, w, v))
    assert got[0][:3] == got[1][:3]
    for a, b in zip(got[0][3:], got[1][3:]):
        assert torch.equal(a, b)
    ctx.close()


def test_sweeps_of_general_exponents_cost_what_the_other_models_do(torch):
    """4096^2 in FP32-bulk: an x sweep of (n, m) = (4, 3), whose mobilities are a
    few products, takes less than 1.3 times one of the NLC model with its tanh
    and reciprocals (least of five each)."""
    n, best = 4096, {}
    for which in ("nlc", "power43"):
        _, p, h0, wm = setup(which, n, n, tf.TF_FP32_BULK)
        p.newton_fixed_iter = 2
        h = h0 * (1.0 + 0.01 * torch.rand((n, n), dtype=torch.float64, device="cuda"))
        out = torch.empty_like(h)
        ctx = tf.Context(p)
        for _ in range(6):
            tf.tf_timing_enable(ctx, True)
            tf.tf_newton_adi_step(ctx, h, out, 1e-3 / wm)
            t = tf.tf_timing_get(ctx)
            best[which] = min(best.get(which, 1e30), t["x_ms"] / t["x_launches"])
        ctx.close()
    assert best["power43"] < 1.3 * best["nlc"], best
