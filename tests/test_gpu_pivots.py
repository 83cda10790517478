"""Zero and non-finite pivots of the line solves, in every block shape.

The linear model's first pivot is 1 + 4 k3 c0 - 2 k1 c1 with k3 = theta dt /
(2 ds^4) and k1 = theta dt / (2 ds^2): with ds = 1, dt = 1, theta = 1/2, c0 = 1
and c1 = 4 it is zero exactly, in either precision.  A film with one cell that is
not a number has lines whose pivots are none either.  Both are reported as such,
before the positivity of the iterate is looked at, by each of the kernels that a
sweep over 30, 700, 1300 and 2500 lines runs in.
"""
import pytest

import oracle as O
import paper_1806_10550_gb300 as tf
from paper_1806_10550_gb300 import synthetic as S

pytestmark = pytest.mark.gpu

SHAPES = [(30, 26), (24, 700), (700, 24), (50, 1300), (1300, 50), (24, 2500), (2500, 24)]


@pytest.fixture(scope="module")
def torch():
    import torch as T
    if not T.cuda.is_available():
        pytest.skip("no CUDA device")
    tf.library()
    return T


@pytest.mark.parametrize("mode", [tf.TF_FP64, tf.TF_FP32_BULK])
@pytest.mark.parametrize("nx,ny", SHAPES)
def test_zero_pivot_is_reported(torch, mode, nx, ny):
    p = tf.tf_params_default(nx=nx, ny=ny, ds=1.0, model=tf.TF_MODEL_LINEAR, c0=1.0, c1=4.0, precision=mode)
    h = torch.from_numpy(S.spinodal_film(nx, ny, 1.0, 0.01, seed=nx + ny)).cuda()
    ctx = tf.Context(p)
    for _ in range(2):
        assert tf.tf_newton_adi_step(ctx, h, torch.empty_like(h), 1.0)["status"] == tf.TF_STEP_ZERO_PIVOT
    assert tf.tf_newton_iteration(ctx, h, h, 1.0, torch.empty_like(h))["status"] == tf.TF_STEP_ZERO_PIVOT
    # another step size has other pivots; its iterates leave the domain, as the oracle's do
    om = O.Model(nx=nx, ny=ny, ds=1.0, model=O.MODEL_LINEAR, c0=1.0, c1=4.0)
    ref = O.step(om, O.Control(), h.cpu().numpy(), 0.125)[1]["status"]
    assert tf.tf_newton_adi_step(ctx, h, torch.empty_like(h), 0.125)["status"] == ref == tf.TF_STEP_NONPOSITIVE
    ctx.close()


@pytest.mark.parametrize("mode", [tf.TF_FP64, tf.TF_FP32_BULK])
@pytest.mark.parametrize("model", [dict(kappa=1.2061475842818314), dict(n=4, m=3, kappa=1.2061475842818314)])
@pytest.mark.parametrize("nx,ny", SHAPES)
def test_pivot_that_is_not_a_number_is_reported(torch, mode, model, nx, ny):
    p = tf.tf_params_default(nx=nx, ny=ny, ds=3.9, precision=mode, **model)
    h = torch.from_numpy(S.spinodal_film(nx, ny, 1.0, 0.01, seed=nx + ny)).cuda()
    ctx = tf.Context(p)
    assert tf.tf_newton_adi_step(ctx, h, torch.empty_like(h), 0.5)["status"] == tf.TF_STEP_CONVERGED
    bad = h.clone()
    bad[ny - 3, nx // 3] = float("nan")
    if mode == tf.TF_FP64:
        assert tf.tf_newton_adi_step(ctx, bad, torch.empty_like(h), 0.5)["status"] == tf.TF_STEP_ZERO_PIVOT
    else:  # the FP32 film takes bits of positive floats: the update's cell is not finite
        assert tf.tf_newton_adi_step(ctx, bad, torch.empty_like(h), 0.5)["status"] in (tf.TF_STEP_ZERO_PIVOT,
                                                                                       tf.TF_STEP_NONPOSITIVE)
    assert tf.tf_newton_adi_step(ctx, h, torch.empty_like(h), 0.5)["status"] == tf.TF_STEP_CONVERGED
    ctx.close()
