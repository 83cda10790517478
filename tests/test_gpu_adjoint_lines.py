"""The adjoint's transposed line solves at the edges of their block shapes
(blocks of 4, 8 and 16 lines: up to 608, 1216 and more lines), with short
lines across: the directional derivative <g_h, v> against the central
difference of <g, step(h + eps v)>.

eps v is at most 1e-6 of the height: the difference's truncation error is
of order (eps v)^2 = 1e-12 of the derivative and its rounding about 1e-16 /
1e-6 = 1e-10 of a sum of cells whose signs vary (a factor of the square root
of their number at most, 180 here), so 1e-6 of the derivative's scale
|g| |v| bounds both.
"""
import numpy as np
import pytest

import paper_1806_10550_gb300 as tf
from paper_1806_10550_gb300 import synthetic as S

pytestmark = pytest.mark.gpu

KAPPA = 1.2061475842818314


@pytest.fixture(scope="module")
def torch():
    import torch as T
    if not T.cuda.is_available():
        pytest.skip("no CUDA device")
    tf.library()
    return T


@pytest.mark.parametrize("nx,ny", [(608, 26), (25, 609), (1216, 7), (13, 1217), (2433, 12), (9, 2434), (3, 700), (700, 3)])
def test_directional_derivative(torch, nx, ny):
    K, dt, eps = 3, 2.0, 1e-6
    p = tf.tf_params_default(nx=nx, ny=ny, ds=3.9, kappa=KAPPA, precision=tf.TF_FP64, newton_fixed_iter=K)
    ctx = tf.Context(p)
    rng = np.random.default_rng(nx + 7 * ny)
    h = torch.from_numpy(S.spinodal_film(nx, ny, 1.0, 0.02, seed=nx * 3 + ny)).cuda()
    g, v = (torch.from_numpy(rng.uniform(-1.0, 1.0, (ny, nx))).cuda() for _ in range(2))
    gh, out = torch.empty_like(h), torch.empty_like(h)
    tf.tf_adjoint_step(ctx, h, dt, K, g, g_h=gh, h_new=out)
    sums = []
    for s in (1.0, -1.0):
        tf.tf_newton_adi_step(ctx, h + s * eps * v, out, dt)
        sums.append(out.clone())
    fd = float((g * ((sums[0] - sums[1]) / (2 * eps))).sum())
    ad = float((gh * v).sum())
    assert abs(fd - ad) <= 1e-6 * float(g.norm() * v.norm())
    ctx.close()
