"""A step queues its next iteration before it reads the last one's result.

With timing on, each iteration waits for the one before; with it off, the
kernels behind a step's last iteration return at once.  Both must give the
same status, iteration count, scalars and bits: steps that converge, that
use up their iterations (1, 2 and 3 of them, into either iterate buffer),
that run a fixed number, and that leave the model's domain, one after another
on one context.
"""
import pytest

import paper_1806_10550_gb300 as tf
from paper_1806_10550_gb300 import synthetic as S

pytestmark = pytest.mark.gpu

KAPPA = 1.2061475842818314
# newton_max_iter, newton_fixed_iter, dt, statuses
CASES = [(10, 0, 2.0, (tf.TF_STEP_CONVERGED,)), (1, 0, 2.0, (tf.TF_STEP_NOT_CONVERGED,)),
         (2, 0, 2.0, (tf.TF_STEP_NOT_CONVERGED,)), (3, 0, 2.0, (tf.TF_STEP_NOT_CONVERGED,)),
         (10, 1, 2.0, (tf.TF_STEP_CONVERGED,)), (10, 4, 2.0, (tf.TF_STEP_CONVERGED,)),
         (10, 0, 1e7, (tf.TF_STEP_NONPOSITIVE, tf.TF_STEP_ZERO_PIVOT, tf.TF_STEP_NOT_CONVERGED))]


@pytest.fixture(scope="module")
def torch():
    import torch as T
    if not T.cuda.is_available():
        pytest.skip("no CUDA device")
    tf.library()
    return T


@pytest.mark.parametrize("mode", [tf.TF_FP64, tf.TF_FP32_BULK])
@pytest.mark.parametrize("max_iter,fixed,dt,statuses", CASES)
def test_same_step_with_and_without(torch, mode, max_iter, fixed, dt, statuses):
    nx, ny = 96, 80
    p = tf.tf_params_default(nx=nx, ny=ny, ds=3.9, kappa=KAPPA, precision=mode, newton_max_iter=max_iter,
                             newton_fixed_iter=fixed)
    h = torch.from_numpy(S.spinodal_film(nx, ny, 1.0, 0.01, seed=3)).cuda()
    got = []
    for timed in (True, False):
        ctx = tf.Context(p)
        tf.tf_timing_enable(ctx, timed)
        a, b = torch.empty_like(h), torch.empty_like(h)
        first = tf.tf_newton_adi_step(ctx, h, a, dt)
        second = tf.tf_newton_adi_step(ctx, h, b, dt)  # behind the first step's tail
        assert first["status"] in statuses
        assert {k: repr(v) for k, v in first.items()} == {k: repr(v) for k, v in second.items()}
        assert torch.equal(a.view(torch.int64), b.view(torch.int64))
        got.append((first, a))
        ctx.close()
    assert {k: repr(v) for k, v in got[0][0].items()} == {k: repr(v) for k, v in got[1][0].items()}
    assert torch.equal(got[0][1].view(torch.int64), got[1][1].view(torch.int64))
