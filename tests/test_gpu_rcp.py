"""fast_rcp (csrc/fixpow.cuh) and safe_rcp (csrc/common.cuh) against exact reciprocals.

Bound of fast_rcp as derived beside it: |q x - 1| <= 2^-53 (1 + 2^-3), over the exponents it
serves (biased 123 to 1922), at the ends of binades and of the 20 leading bits, both signs.
Outside them safe_rcp divides: the correctly rounded quotient, zeros, infinities and NaN
included."""
import ctypes
from fractions import Fraction

import numpy as np
import pytest

from device_code import compile_device

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "common.cuh"
using namespace rich;
namespace rich { void set_cuda_error(cudaError_t, const char*) {} }
__global__ void k(int n, const double* q, double* f, double* s) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) {
    f[i] = fast_rcp(q[i]);
    s[i] = safe_rcp(q[i]);
  }
}
extern "C" int rcp(int n, const double* q, double* f, double* s) {
  k<<<(n + 255) / 256, 256>>>(n, q, f, s);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def rcp(tmp_path_factory):
    lib = compile_device(SOURCE, tmp_path_factory.mktemp("rcp"))

    def run(q):
        t = torch.tensor(q, dtype=torch.float64, device="cuda")
        f, s = torch.empty_like(t), torch.empty_like(t)
        torch.cuda.synchronize()
        assert lib.rcp(len(q), *(ctypes.c_void_p(v.data_ptr()) for v in (t, f, s))) == 0
        return f.cpu().numpy(), s.cpu().numpy()

    return run


def _doubles(exponents, mantissas, signs):
    bits = (np.asarray(signs, dtype=np.uint64) << np.uint64(63)) | (
        np.asarray(exponents, dtype=np.uint64) << np.uint64(52)) | np.asarray(mantissas, dtype=np.uint64)
    return bits.view(np.float64)


def test_inside_the_window(rcp):
    rng = np.random.default_rng(1)
    e = np.concatenate([np.arange(123, 1923), rng.integers(123, 1923, 30000)])
    m = np.concatenate([rng.integers(0, 1 << 52, 16800), rng.integers(0, 1 << 20, 5000) << 32,
                        (rng.integers(0, 1 << 20, 5000) << 32) | 0xffffffff, np.zeros(2500, dtype=np.int64),
                        np.full(2500, (1 << 52) - 1)])
    q = _doubles(e, m, rng.integers(0, 2, len(e)))
    f, s = rcp(q)
    np.testing.assert_array_equal(f, s)
    bound = Fraction(9, 8) / 2 ** 53
    assert all(abs(Fraction(float(a)) * Fraction(float(b)) - 1) <= bound for a, b in zip(q, f))


def test_outside_the_window(rcp):
    rng = np.random.default_rng(2)
    e = np.concatenate([rng.integers(0, 123, 2000), rng.integers(1923, 2047, 2000), [122] * 8, [1923] * 8])
    q = _doubles(e, rng.integers(0, 1 << 52, len(e)), rng.integers(0, 2, len(e)))
    q = np.concatenate([q, [0.0, -0.0, np.inf, -np.inf, np.nan, 5e-324, -5e-324]])
    with np.errstate(divide="ignore", over="ignore"):
        np.testing.assert_array_equal(rcp(q)[1], 1.0 / q)
