"""The line sweeps at the edges of their block shapes.

A sweep over n lines runs in blocks of 4, 8, 16 or 32 lines: up to 608, 1216
and 2432 lines in FP64, up to 608 and 2432 (4, 8) and 16 beyond in FP32-bulk.
One Newton iteration is compared with the FP64 oracle one line to each side of
every edge (and at 4864 lines, two blocks of 16 an SM), with short lines
across (one chunk of 24 cells, a chunk and a ragged tail, a few cells) and
with the lines along x and along y.  Films advanced at once run in larger
blocks than a film alone; their results are the same bits.
"""
import numpy as np
import pytest

import oracle as O
import paper_1806_10550_gb300 as tf
from paper_1806_10550_gb300 import synthetic as S

pytestmark = pytest.mark.gpu

KAPPA = 1.2061475842818314
EDGES = [(608, 24), (609, 50), (1216, 7), (1217, 77), (2432, 49), (2433, 25), (4864, 26), (4865, 3)]


@pytest.fixture(scope="module")
def torch():
    import torch as T
    if not T.cuda.is_available():
        pytest.skip("no CUDA device")
    tf.library()
    return T


@pytest.mark.parametrize("mode", [tf.TF_FP64, tf.TF_FP32_BULK])
@pytest.mark.parametrize("lines,n", EDGES)
@pytest.mark.parametrize("along_x", [True, False])
def test_iteration_at_block_shape_edges(torch, mode, lines, n, along_x):
    nx, ny = (n, lines) if along_x else (lines, n)
    ds, dt = 1.9, 2.0
    om = O.Model(nx=nx, ny=ny, ds=ds, kappa=KAPPA)
    h_old = S.spinodal_film(nx, ny, 1.0, 0.05, seed=11 * nx + ny)
    ctx = tf.Context(tf.tf_params_default(nx=nx, ny=ny, ds=ds, kappa=KAPPA, precision=mode))
    w, v, hn = (torch.empty((ny, nx), dtype=torch.float64, device="cuda") for _ in range(3))
    hk = torch.from_numpy(h_old).cuda()
    info = tf.tf_newton_iteration(ctx, hk, hk, dt, hn, w=w, v=v)
    r = O.newton_iteration(om, h_old, O.explicit_part(om, h_old, dt), dt)
    # single-precision solves, or FP64 solves in another order of operations,
    # as in the parity tests of one iteration
    rel = 2e-4 if mode == tf.TF_FP32_BULK else 1e-11
    sw, sv = np.max(np.abs(r["w"])), np.max(np.abs(r["v"]))
    assert np.max(np.abs(w.cpu().numpy() - r["w"])) <= rel * sw
    assert np.max(np.abs(v.cpu().numpy() - r["v"])) <= rel * sv
    assert np.max(np.abs(hn.cpu().numpy() - r["unew"])) <= 1e-15 + rel * sv
    assert info["err"] == pytest.approx(r["err"], rel=1e-3)
    ctx.close()


@pytest.mark.parametrize("mode", [tf.TF_FP64, tf.TF_FP32_BULK])
@pytest.mark.parametrize("films", [3, 8, 30, 64])
def test_films_at_once_equal_films_alone(torch, mode, films):
    """600, 1600, 6000 and 12800 lines at once: blocks of 4, 8, 16 and 32 lines."""
    ds, dt = 3.9, 1.0
    params = [tf.tf_params_default(nx=200 - (i % 3), ny=170 + (i % 2), ds=ds, kappa=KAPPA, precision=mode) for i in range(films)]
    start = [torch.from_numpy(S.spinodal_film(p.nx, p.ny, 1.0, 0.01, seed=50 + i)).cuda() for i, p in enumerate(params)]
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
