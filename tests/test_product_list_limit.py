"""The memory rule of the Galerkin product lists (csrc/plist_limit.h), compiled on the host.

Lists may take half the free device memory, counted with the padding of their slices: 32
entries of one slice all take the longest one's slots.  The slots are laid out here as the
device does (windows of 1024 entries sorted by decreasing count, slices of 32)."""
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def fits(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("plist")
    (d / "t.cpp").write_text(
        '#include "plist_limit.h"\n#include <cstdio>\n#include <cstdlib>\n'
        "int main(int, char** a) { printf(\"%d\", rich::plist_fits(atof(a[1]), atof(a[2]), atof(a[3]))); }\n")
    exe = str(d / "t")
    subprocess.run([gxx, "-O1", "-I", os.path.join(ROOT, "paper_2112_05051_gb300", "csrc"), str(d / "t.cpp"), "-o", exe],
                   check=True)
    return lambda slots, nnz, free: subprocess.run([exe, repr(float(slots)), repr(float(nnz)), repr(float(free))],
                                                   capture_output=True, text=True, check=True).stdout == "1"


def _slots(counts):
    total = 0
    for w in range(0, len(counts), 1024):
        c = -np.sort(-counts[w:w + 1024])
        total += 32 * int(c[::32].sum())
    return total


@pytest.mark.parametrize("counts", [np.full(32, 7), np.r_[np.full(31, 1), 4000], np.arange(1, 3000),
                                    np.r_[np.full(1023, 2), 60000]], ids=["even", "one long", "ramp", "long in a window"])
def test_padding_counts_towards_the_limit(fits, counts):
    nnz, products, slots = len(counts), int(counts.sum()), _slots(counts)
    need = 8.0 * slots + 24.0 * (nnz + 1)
    assert slots >= products
    assert fits(slots, nnz, 2 * need) and not fits(slots, nnz, 2 * need - 1)
    if slots > products:  # between the two sizes: what the products alone would still allow is refused
        free = 2 * (8.0 * (slots + products) / 2 + 24.0 * (nnz + 1))
        assert fits(products, nnz, free) and not fits(slots, nnz, free)
