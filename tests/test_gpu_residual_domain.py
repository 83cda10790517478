"""tf_residual on films that left the model's domain (FP32-bulk).

A caller that watches its own iterates meets heights that are zero, negative,
not finite, or positive but outside the floats: G and its norm must then be
those of the film that was given.  tf_residual_noalloc, which forms the same
G from the same arithmetic, is the reference; the two form b^n with different
double-float kernels, each accurate to about 2^-46 of the terms it adds
(the residual comparison's 1e-12), and G within 2^-46 of itself.  Away from the
cell (its stencil reaches two cells along each axis) G is also compared with
the FP64 oracle's.  Lengths in any unit give the same film: G is compared
again over units whose fluxes leave the floats in one kernel's scaling.
"""
import ctypes as C

import numpy as np
import pytest

import oracle as O
import paper_1806_10550_gb300 as tf
from paper_1806_10550_gb300 import synthetic as S

pytestmark = pytest.mark.gpu

KAPPA = 1.2061475842818314
# 1e-40 is below the normal floats, 1e-25 above them but with a trailing part
# below, 3e38 and 1e39 to each side of the largest float
HEIGHTS = [-0.5, 0.0, -0.0, float("nan"), float("inf"), -float("inf"), 1e-40, 1e-25, 2.0 ** 127, 1e39]


@pytest.fixture(scope="module")
def torch():
    import torch as T
    if not T.cuda.is_available():
        pytest.skip("no CUDA device")
    L = tf.library()
    L.tf_residual_noalloc.argtypes = [C.POINTER(tf.TfParams), C.c_void_p, C.c_void_p, C.c_void_p, C.c_double,
                                      C.c_void_p, C.POINTER(tf.TfNorms)]
    L.tf_residual_noalloc.restype = C.c_int
    return T


# inside a strip of 60 columns, on its edge, and in a corner of the film
@pytest.mark.parametrize("nx,ny,i,j", [(150, 70, 30, 35), (150, 70, 60, 16), (61, 33, 0, 32)])
@pytest.mark.parametrize("height", HEIGHTS)
def test_residual_of_an_iterate_outside_the_domain(torch, nx, ny, i, j, height):
    ds, dt = 1.7, 3.0
    h_old = S.spinodal_film(nx, ny, 1.0, 0.05, seed=nx + ny)
    good = h_old + 0.01 * S.spinodal_film(nx, ny, 0.0, 1.0, seed=7)
    h_k = good.copy()
    h_k[j, i] = height
    p = tf.tf_params_default(nx=nx, ny=ny, ds=ds, kappa=KAPPA, precision=tf.TF_FP32_BULK)
    hk, ho = torch.from_numpy(h_k).cuda(), torch.from_numpy(h_old).cuda()
    G, R = (torch.full((ny, nx), -7.0, dtype=torch.float64, device="cuda") for _ in range(2))
    ctx = tf.Context(p)
    got = tf.tf_residual(ctx, hk, ho, dt, G)
    n = tf.TfNorms()
    rc = tf.library().tf_residual_noalloc(C.byref(p), C.c_void_p(torch.cuda.current_stream().cuda_stream),
                                          C.c_void_p(hk.data_ptr()), C.c_void_p(ho.data_ptr()), dt,
                                          C.c_void_p(R.data_ptr()), C.byref(n))
    assert rc == tf.TF_OK
    g, r = G.cpu().numpy(), R.cpu().numpy()
    assert np.array_equal(np.isnan(g), np.isnan(r))
    inf = np.isinf(r)
    assert np.array_equal(np.isinf(g), inf) and np.array_equal(g[inf], r[inf])
    fin = np.isfinite(r)
    assert np.all(np.abs(g[fin] - r[fin]) <= 1e-12 * np.maximum(1.0, np.abs(r[fin])))
    assert got["gnorm"] == np.nanmax(np.abs(g))
    assert got["hmin"] == n.hmin and got["mass"] == n.mass
    # without G: the norm alone, of the same film
    assert tf.tf_residual(ctx, hk, ho, dt)["gnorm"] == got["gnorm"]
    om = O.Model(nx=nx, ny=ny, ds=ds, kappa=KAPPA)
    ref = O.residual(om, good, O.explicit_part(om, h_old, dt), dt)
    jj, ii = np.mgrid[0:ny, 0:nx]
    away = np.abs(jj - j) + np.abs(ii - i) > 2
    assert np.max(np.abs(g - ref)[away]) <= 1e-12 * max(1.0, np.max(np.abs(ref)))
    # the context serves good films afterwards
    tf.tf_residual(ctx, torch.from_numpy(good).cuda(), ho, dt, G)
    assert np.max(np.abs(G.cpu().numpy() - ref)) <= 1e-12 * max(1.0, np.max(np.abs(ref)))
    ctx.close()


@pytest.mark.parametrize("aspect", [1.0, 100.0])  # ds / h
@pytest.mark.parametrize("unit", [1e-12, 1e-10, 1e-9, 1e-8, 1e-7, 1e-6, 1e-3, 1.0, 1e3, 1e6, 1e9, 1e11, 1e13])
def test_residual_in_any_unit_of_length(torch, unit, aspect):
    """With theta = 1, where b^n is h_old, G of the two entry points: to 1e-12
    of its largest value, and not finite in the same cells (beyond 1e12 the
    mobilities overflow the floats in either)."""
    nx, ny = 150, 70
    ds, b = 1.7 * unit * aspect, 0.1 * unit
    dt = 3.0 * unit * aspect ** 4
    h_old = unit * S.spinodal_film(nx, ny, 1.0, 0.05, seed=5)
    h_k = h_old + 0.01 * unit * S.spinodal_film(nx, ny, 0.0, 1.0, seed=7)
    p = tf.tf_params_default(nx=nx, ny=ny, ds=ds, b=b, kappa=KAPPA / unit, theta=1.0, precision=tf.TF_FP32_BULK)
    hk, ho = torch.from_numpy(h_k).cuda(), torch.from_numpy(h_old).cuda()
    G, R = (torch.full((ny, nx), -7.0, dtype=torch.float64, device="cuda") for _ in range(2))
    ctx = tf.Context(p)
    got = tf.tf_residual(ctx, hk, ho, dt, G)
    ctx.close()
    n = tf.TfNorms()
    rc = tf.library().tf_residual_noalloc(C.byref(p), C.c_void_p(torch.cuda.current_stream().cuda_stream),
                                          C.c_void_p(hk.data_ptr()), C.c_void_p(ho.data_ptr()), dt,
                                          C.c_void_p(R.data_ptr()), C.byref(n))
    assert rc == tf.TF_OK
    g, r = G.cpu().numpy(), R.cpu().numpy()
    fin = np.isfinite(r)
    assert np.array_equal(np.isfinite(g), fin)
    if fin.any():
        assert np.max(np.abs(g - r)[fin]) <= 1e-12 * np.max(np.abs(r[fin]))
    assert got["hmin"] == n.hmin and got["mass"] == n.mass
