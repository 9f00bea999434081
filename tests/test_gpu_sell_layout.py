"""The SELL layout made on the device (k_sell_rank of csrc/sell.cu) against the host's
(rich_sell_layout): the same permutation, rows of equal length in their order, and the same
slice widths.  Sizes around a slice and a window of 1024 rows; empty rows, all rows alike,
one long row."""
import ctypes

import numpy as np
import pytest

from device_code import compile_device

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "sell.cu"
using namespace rich;
extern "C" int rank(int n, const int* rp, int nslice, int* perm, int* slots) {
  k_sell_rank<<<(n + kSellSigma - 1) / kSellSigma, kSellSigma>>>(n, rp, nslice, perm, slots);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    from paper_2112_05051_gb300 import build
    return compile_device(SOURCE, tmp_path_factory.mktemp("sell"), [build.LIB])


@pytest.mark.parametrize("n", [1, 31, 32, 33, 1023, 1024, 1025, 2048, 5000])
@pytest.mark.parametrize("rows", ["random", "alike", "empty ones", "one long"])
def test_device_layout_is_the_host_layout(lib, n, rows):
    from paper_2112_05051_gb300 import richards as rb
    rb.load()
    rng = np.random.default_rng(n)
    length = {"random": rng.integers(1, 40, n), "alike": np.full(n, 7), "empty ones": rng.integers(0, 3, n),
              "one long": np.where(np.arange(n) == n // 2, 3000, 2)}[rows]
    rp = np.concatenate([[0], np.cumsum(length)]).astype(np.int32)
    perm, sptr, _ = rb.sell_layout(rp)
    ns = (n + 31) // 32
    dev = lambda a: torch.tensor(a, dtype=torch.int32, device="cuda")
    d_rp, d_perm, d_slots = dev(rp), dev(np.full(32 * ns, -7)), dev(np.full(ns, -7))
    torch.cuda.synchronize()
    assert lib.rank(n, *(ctypes.c_void_p(t.data_ptr()) if not isinstance(t, int) else t
                         for t in (d_rp, ns, d_perm, d_slots))) == 0
    np.testing.assert_array_equal(d_perm.cpu().numpy(), perm)
    np.testing.assert_array_equal(d_slots.cpu().numpy(), np.diff(sptr))
