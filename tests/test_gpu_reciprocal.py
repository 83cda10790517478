"""rcp3, the reciprocal of the FP64 line solves, against CUDA's division.

The seed r0 depends on the upper 32 bits of its argument only, so its error
1 - x r0 is measured over all 2^20 upper significands, with the lower word at
both of its ends (the error is monotonic between them); it must be at most
2^-18.  Then r0 (1 + e + e^2) leaves e^3 <= 2^-54 of the quotient, half a unit
in the last place, beside the half of the last rounding: one unit in all.
Arguments that take the division give its bits.
"""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

from paper_1806_10550_gb300 import _build

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "tf_kernels.cuh"
namespace {
__global__ void k_reciprocals(const double* x, double* r, double* q, double* e, size_t n) {
  const size_t k = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  if (k >= n) return;
  const double v = x[k];
  double r0;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r0) : "d"(v));
  r[k] = tf::rcp3(v);
  q[k] = 1.0 / v;
  e[k] = fma(-v, r0, 1.0);
}
}  // namespace
extern "C" int reciprocals(const double* x, double* r, double* q, double* e, size_t n) {
  k_reciprocals<<<(unsigned)((n + 255) / 256), 256>>>(x, r, q, e, n);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def reciprocals(tmp_path_factory):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    d = tmp_path_factory.mktemp("reciprocal")
    src, lib = str(d / "reciprocal.cu"), str(d / "libreciprocal.so")
    with open(src, "w") as f:
        f.write(SOURCE)
    subprocess.run([_build._nvcc(), *_build.ARCH, *_build.FLAGS, "-I", _build.CSRC, "-shared", "-o", lib, src],
                   check=True)
    L = C.CDLL(lib)
    L.reciprocals.argtypes = [C.c_void_p] * 4 + [C.c_size_t]

    def run(x):
        x = torch.from_numpy(np.ascontiguousarray(x, dtype=np.float64)).cuda()
        out = [torch.empty_like(x) for _ in range(3)]
        torch.cuda.synchronize()
        assert L.reciprocals(*(C.c_void_p(t.data_ptr()) for t in (x, *out)), x.numel()) == 0
        return [t.cpu().numpy() for t in out]
    return run


def doubles(exponent, significand, sign=0):
    """Doubles of a biased exponent, a 52-bit significand and a sign bit."""
    return (np.uint64(sign) << np.uint64(63) | np.asarray(exponent, np.uint64) << np.uint64(52)
            | np.asarray(significand, np.uint64)).view(np.float64)


def units_off(r, q):
    """Units in the last place between two arrays of normal numbers of one sign."""
    return np.max(np.abs(r.view(np.int64) - q.view(np.int64)))


@pytest.mark.parametrize("exponent", [64, 1022, 1023, 1024, 1982])
def test_seed_and_reciprocal_over_all_upper_significands(reciprocals, exponent):
    upper = np.arange(2 ** 20, dtype=np.uint64) << np.uint64(32)
    for lower in (0, 2 ** 32 - 1):
        for sign in (0, 1):
            r, q, e = reciprocals(doubles(exponent, upper | np.uint64(lower), sign))
            assert np.max(np.abs(e)) <= 2.0 ** -18
            assert units_off(r, q) <= 1


def test_random_arguments(reciprocals):
    rng = np.random.default_rng(5)
    n = 1 << 21
    x = doubles(rng.integers(64, 1983, n), rng.integers(0, 2 ** 52, n, dtype=np.uint64),
                0) * rng.choice([-1.0, 1.0], n)
    r, q, _ = reciprocals(x)
    assert units_off(r, q) <= 1


def test_arguments_that_take_the_division(reciprocals):
    rng = np.random.default_rng(6)
    sig = rng.integers(0, 2 ** 52, 1000, dtype=np.uint64)
    x = np.concatenate([doubles(e, sig, s) for e in (0, 1, 63, 1983, 2046) for s in (0, 1)]
                       + [[0.0, -0.0, np.inf, -np.inf, 5e-324, -5e-324]])
    r, q, _ = reciprocals(x)
    assert np.array_equal(r.view(np.int64), q.view(np.int64))
    r, q, _ = reciprocals(np.array([np.nan, -np.nan]))
    assert np.all(np.isnan(r)) and np.all(np.isnan(q))
