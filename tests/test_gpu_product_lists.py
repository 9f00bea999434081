"""Galerkin refresh by product lists whose entries are long: aggregates of up to 1024 cells
give entries of R (A P) with more than 512 products, which are filed by a block's warps in
any order and written anew in A-entry order.  Against the refresh that searches each
product's place (product_lists = 0), level by level, and against a second context bit for bit
(an entry summed in another order than the lists' would differ between the two).

Bar: both sum the same products; an entry has at most 4096 of them, whose rounding is within
4096 x 2^-52 < 1e-12 of the sum of their magnitudes, itself within ten times the largest
entry of its level: 1e-11 (in MIXED, FP32 products: 4096 x 2^-23 x 10 < 5e-3)."""
import numpy as np
import pytest

from paper_2112_05051_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _levels(dims, lists, prec, **amg):
    from paper_2112_05051_gb300 import richards as rb
    rb.load()
    grid = synth.Grid(*dims)
    rng = np.random.default_rng(3)
    z = (np.arange(grid.nz) + 1.0) / (grid.nz + 1)
    p = np.broadcast_to((-61.5 + 40.8 * np.exp(-(1.0 - z) / 0.2))[:, None, None], grid.shape).ravel()
    p = torch.tensor(p + rng.uniform(-0.3, 0.3, grid.n), device="cuda")
    ctx = rb.Context(grid, synth.Soil(), synth.infiltration_bc(), synth.KMEAN_ARITH, None, precision=prec)
    ctx.jacobian(p, 1.0)
    info = ctx.amg_setup(rb.default_amg_opts(seed=3, product_lists=lists, aggregation=rb.AGG_MATCHING, **amg))
    ctx.jacobian(p + 0.5, 2.0)
    ctx.amg_update(rb.AMG_REFRESH)
    out = [ctx.export_level(k, info)[1:] for k in range(info.levels)]
    longest = max(np.bincount(ctx.export_prolongator(k, info)[1]).max() for k in range(info.levels - 1))
    ctx.close()
    return out, longest


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("dims,amg,long_entries", [((24, 24, 24), dict(max_agg_size=1024, coarse_max=4), True),
                                                   ((33, 17, 29), dict(max_agg_size=512, coarse_max=4), True),
                                                   ((40, 40, 40), dict(max_agg_size=8, coarse_max=50), True),
                                                   ((16, 14, 12), dict(max_agg_size=8, coarse_max=20), False)])
def test_long_entries_against_the_searching_refresh(dims, amg, long_entries, prec):
    a, longest = _levels(dims, 1, prec, **amg)
    b, _ = _levels(dims, 1, prec, **amg)
    c, _ = _levels(dims, 0, prec, **amg)
    assert (longest > 512) == long_entries and len(a) == len(c) > 1
    for x, y, s in zip(a, b, c):
        for k in range(3):
            np.testing.assert_array_equal(x[k], y[k])
        np.testing.assert_array_equal(x[0], s[0])
        np.testing.assert_array_equal(x[1], s[1])
        assert np.abs(x[2] - s[2]).max() <= (1e-11 if prec == 0 else 5e-3) * np.abs(s[2]).max()
