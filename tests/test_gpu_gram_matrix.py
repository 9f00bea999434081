"""The Gram matrix of FGMRES' basis (csrc/gram.cuh), summed in integers, against exact dots.

Unit vectors whose rounding to the integers' units is lost alike by all entries (a constant,
a smooth one), random ones, one concentrated near a face, one with a single large entry and a
tail; few cells and many.  Exact values by products split without error (T. J. Dekker, 1971)
and math.fsum.

Bar: what sums in FP64 leave, 33 additions on the way from a thread to the result, each
rounding by at most 2^-53 of sum |a b| <= 1 and independent of the others: four standard
deviations, 4 sqrt(33) 2^-53 / sqrt(3) < 1.5e-15; and the integers' units, 2^-58, for vectors
whose largest entry is like the others'.  (With one unit of 2^-60 for all vectors, the
constant of 16M cells is off by 2^-60 sqrt(n) = 3.5e-15.)  A single large entry keeps the
unit at 2^-60: 2^-60 ||.||_1 is added."""
import ctypes
import math

import numpy as np
import pytest

from device_code import compile_device

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "gram.cuh"
using namespace rich;
namespace rich { void set_cuda_error(cudaError_t, const char*) {} }
extern "C" int gram_row(long long n, int nv, const double* V, const double* w, double* part, double* gram, unsigned* peak,
                        unsigned* ticket, double* s, double* mirror) {
  const double* v = V + (long long)(nv - 1) * n;
  const long long g = (n + kGsThreads - 1) / kGsThreads;
  k_gs_peak<<<(int)(g < kGsBlocks ? g : kGsBlocks), kGsThreads>>>(n, v, 1.0, peak + nv - 1);
  k_gs_dots<<<(int)(g < kGsBlocks ? g : kGsBlocks), kGsThreads>>>(n, nv, V, w, part, gram, peak, ticket, s, mirror);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return compile_device(SOURCE, tmp_path_factory.mktemp("gram"))


def _exact(a, b):
    def split(x):
        t = 134217729.0 * x
        hi = t - (t - x)
        return hi, x - hi
    p = a * b
    (ah, al), (bh, bl) = split(a), split(b)
    e = ((ah * bh - p) + ah * bl + al * bh) + al * bl
    return math.fsum(p) + math.fsum(e)


def _vectors(n):
    rng = np.random.default_rng(n)
    x = (np.arange(n) + 0.5) / n
    const = math.floor(2.0 ** 60 / math.sqrt(n)) + 0.499  # between two units of 2^-60
    spike = np.full(n, 0.4 / math.sqrt(n))
    spike[n // 3] = 0.9
    vs = {"constant": np.full(n, const * 2.0 ** -60), "smooth": np.sqrt(2.0 / n) * np.cos(3.0 * x),
          "random": rng.standard_normal(n), "front": np.exp(-40.0 * x) * (1.0 + 0.1 * rng.random(n)), "spike": spike}
    return {k: v if k == "constant" else v / np.linalg.norm(v) for k, v in vs.items()}


@pytest.mark.parametrize("n,names", [(1000, ("constant", "smooth", "random", "front", "spike")),
                                     (300007, ("constant", "smooth", "random", "front", "spike")),
                                     (16000003, ("smooth", "constant"))])
def test_gram_row_against_exact_dots(lib, n, names):
    vs = _vectors(n)
    dev = lambda k, dt=torch.float64: torch.zeros(k, dtype=dt, device="cuda")
    V = torch.tensor(np.concatenate([vs[k] for k in names]), device="cuda")
    w = torch.ones(n, dtype=torch.float64, device="cuda")
    part, gram, s, mirror = dev(128 * 456), dev(64 * 64), dev(256), dev(256)
    peak, ticket = dev(64, torch.int32), dev(1, torch.int32)
    p = lambda t: ctypes.c_void_p(t.data_ptr())
    torch.cuda.synchronize()
    for nv in range(1, len(names) + 1):
        assert lib.gram_row(ctypes.c_longlong(n), nv, p(V), p(w), p(part), p(gram), p(peak), p(ticket), p(s),
                            p(mirror)) == 0
    got = gram.cpu().numpy().reshape(64, 64)
    for j, b in enumerate(names):
        for i, a in enumerate(names[:j + 1]):
            tol = 1.5e-15 + 2.0 ** -58
            if "spike" in (a, b):
                tol += 2.0 ** -60 * max(np.abs(vs[a]).sum(), np.abs(vs[b]).sum())
            assert got[i, j] == got[j, i]
            assert abs(got[i, j] - _exact(vs[a], vs[b])) <= tol, (a, b)
