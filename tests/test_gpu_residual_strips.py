"""tf_residual on the strip kernel (FP32-bulk, (3, 2) power law) at the edges of
its segments: strips of 60 columns, in segments of 2, 4, 8 or 16 rows by the
size of the film, one row or column to each side of whole strips and segments.
G against the FP64 oracle to 1e-12 of its largest value (or absolutely, when
that is below 1), its norm, the mass and the least height of the iterate.
"""
import numpy as np
import pytest

import oracle as O
import paper_1806_10550_gb300 as tf
from paper_1806_10550_gb300 import synthetic as S

pytestmark = pytest.mark.gpu

KAPPA = 1.2061475842818314
SHAPES = [(59, 2), (60, 3), (61, 4), (121, 1), (1, 121), (2, 5), (4001, 92), (3999, 185), (4020, 187), (4001, 371)]


@pytest.fixture(scope="module")
def torch():
    import torch as T
    if not T.cuda.is_available():
        pytest.skip("no CUDA device")
    tf.library()
    return T


@pytest.mark.parametrize("nx,ny", SHAPES)
def test_reported_residual(torch, nx, ny):
    ds, dt = 1.7, 3.0
    om = O.Model(nx=nx, ny=ny, ds=ds, kappa=KAPPA)
    h_old = S.spinodal_film(nx, ny, 1.0, 0.05, seed=nx + 3 * ny)
    h_k = h_old + 0.01 * S.spinodal_film(nx, ny, 0.0, 1.0, seed=7) + 0.001
    ctx = tf.Context(tf.tf_params_default(nx=nx, ny=ny, ds=ds, kappa=KAPPA, precision=tf.TF_FP32_BULK))
    G = torch.full((ny, nx), float("nan"), dtype=torch.float64, device="cuda")
    norms = tf.tf_residual(ctx, torch.from_numpy(h_k).cuda(), torch.from_numpy(h_old).cuda(), dt, G)
    ref = O.residual(om, h_k, O.explicit_part(om, h_old, dt), dt)
    got = G.cpu().numpy()
    scale = np.max(np.abs(ref))
    assert np.max(np.abs(got - ref)) <= 1e-12 * max(1.0, scale)
    assert norms["gnorm"] == np.max(np.abs(got))
    assert norms["hmin"] == np.min(h_k)
    assert abs(norms["mass"] - h_k.sum()) <= nx * ny * 2.0 ** -37 + 1e-13 * h_k.sum()
    ctx.close()
