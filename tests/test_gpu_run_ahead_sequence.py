"""Steps of different outcomes on one context, and the skipped iteration.

A step queues one iteration behind its last, which must return at once, also
after steps that failed.  Its writes could not be seen (they go to buffers
that the step or the next one writes again), so the skip is measured: a step
that may run further iterations takes no longer than one whose limit is the
number it needs.
"""
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


@pytest.mark.parametrize("mode", [tf.TF_FP64, tf.TF_FP32_BULK])
def test_steps_of_different_outcomes_on_one_context(torch, mode):
    nx, ny = 96, 80
    p = tf.tf_params_default(nx=nx, ny=ny, ds=3.9, kappa=KAPPA, precision=mode)
    h = torch.from_numpy(S.spinodal_film(nx, ny, 1.0, 0.01, seed=3)).cuda()
    bad = h.clone()
    bad[ny // 2, nx // 2] = -0.25
    one = tf.Context(p)
    statuses = set()
    for film, dt in ((h, 2.0), (h, 1e7), (h, 0.5), (bad, 2.0), (h, 2.0), (h, 1e-3), (h, 1e7), (bad, 1e7), (h, 2.0)):
        a, b = torch.empty_like(h), torch.empty_like(h)
        got = tf.tf_newton_adi_step(one, film, a, dt)
        fresh = tf.Context(p)
        ref = tf.tf_newton_adi_step(fresh, film, b, dt)
        fresh.close()
        assert {k: repr(v) for k, v in got.items()} == {k: repr(v) for k, v in ref.items()}
        assert torch.equal(a.view(torch.int64), b.view(torch.int64))
        statuses.add(got["status"])
    assert tf.TF_STEP_CONVERGED in statuses and len(statuses) > 1
    one.close()


def test_the_iteration_behind_the_last_is_skipped(torch):
    """2048^2: an iteration takes about 200 us, a launch that returns at once
    a few.  The least of ten times of a step that may run 12 iterations and
    needs k is within half an iteration of one limited to k."""
    n = 2048
    h = torch.from_numpy(S.spinodal_film(n, n, 1.0, 0.01, seed=3)).cuda()
    out = torch.empty_like(h)

    def context(limit):
        return tf.Context(tf.tf_params_default(nx=n, ny=n, ds=3.9, kappa=KAPPA, precision=tf.TF_FP32_BULK,
                                               newton_max_iter=limit))

    free = context(12)
    info = tf.tf_newton_adi_step(free, h, out, 2.0)
    assert info["status"] == tf.TF_STEP_CONVERGED and 1 < info["iterations"] < 12
    limited = context(info["iterations"])
    best = {}
    for _ in range(10):
        for ctx in (free, limited):
            e0, e1 = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            e0.record()
            again = tf.tf_newton_adi_step(ctx, h, out, 2.0)
            e1.record()
            torch.cuda.synchronize()
            assert again == info
            best[ctx] = min(best.get(ctx, 1e30), e0.elapsed_time(e1))
    assert best[free] < best[limited] * (1.0 + 0.5 / info["iterations"])
    free.close()
    limited.close()
