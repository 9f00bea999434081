"""The coarsest level's inverse (symmetric blocked Gauss-Jordan) through the V-cycle.

With one level (max_levels = 1) the V-cycle is z = A_aux^-1 r, so A_aux z must give r
back.  Sizes around the 32-wide tiles: one pivot, one tile, exact multiples, one more or
less, and the largest tests afford.  Bar: the residual of a stable inverse, 1e-10 ||r|| (the
matrices' condition is below 1e5), in MIXED (an FP32 inverse of the FP64 matrix) 1e-2."""
import numpy as np
import pytest

from oracle import discretization as disc
from paper_2112_05051_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(1, 1, 1), (5, 2, 1), (31, 1, 1), (8, 4, 1), (33, 1, 1), (8, 8, 1), (13, 5, 1),
                                  (127, 1, 1), (16, 8, 8), (11, 10, 19)])
def test_single_level_inverse(dims):
    from paper_2112_05051_gb300 import richards as rb
    rb.load()
    grid = synth.Grid(*dims)
    rng = np.random.default_rng(sum(dims))
    p = rng.uniform(-60, -20, grid.n)
    bc = synth.infiltration_bc()
    A = disc.aux_matrix(grid, synth.Soil(), bc, 0, p, 0.1, None)
    r = rng.standard_normal(grid.n)
    for prec, tol in ((0, 1e-10), (1, 1e-2)):
        ctx = rb.Context(grid, synth.Soil(), bc, 0, None, precision=prec)
        ctx.jacobian(torch.tensor(p, device="cuda"), 0.1)
        ctx.amg_setup(rb.default_amg_opts(seed=1, max_levels=1))
        for _ in range(2):  # built at the setup, replayed by the refresh
            z = torch.empty(grid.n, dtype=torch.float64, device="cuda")
            ctx.vcycle(torch.tensor(r, device="cuda"), z)
            assert np.linalg.norm(A @ z.cpu().numpy() - r) <= tol * np.linalg.norm(r)
            ctx.amg_update(rb.AMG_REFRESH)
        ctx.close()
