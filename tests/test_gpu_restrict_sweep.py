"""The restriction that also writes the next level's first sweep, D_l1^-1 b: V-cycles whose
coarsest level is dense or is itself smoothed, with none, one or several pre-sweeps, against
the oracle's cycle.  Bar as in the other V-cycle tests: 1e-10 of the largest entry."""
import numpy as np
import pytest

from oracle import amg
from oracle import discretization as disc
from paper_2112_05051_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,max_levels", [((48, 44, 40), 2), ((40, 36, 32), 2), ((31, 29, 27), 16), ((7, 5, 3), 16)])
@pytest.mark.parametrize("nu1,nu2", [(0, 2), (1, 1), (2, 1), (3, 0)])
def test_vcycle_against_the_oracle(dims, max_levels, nu1, nu2):
    from paper_2112_05051_gb300 import richards as rb
    rb.load()
    grid = synth.Grid(*dims)
    rng = np.random.default_rng(sum(dims))
    z = (np.arange(grid.nz) + 1.0) / (grid.nz + 1)
    p = np.broadcast_to((-61.5 + 40.8 * np.exp(-(1.0 - z) / 0.2))[:, None, None], grid.shape).ravel()
    p = p + rng.uniform(-0.5, 0.5, grid.n)
    r = rng.standard_normal(grid.n)
    coarse_max = 2000 if max_levels == 2 else 60
    ctx = rb.Context(grid, synth.Soil(), synth.infiltration_bc(), 0, None)
    ctx.jacobian(torch.tensor(p, device="cuda"), 1.0)
    info = ctx.amg_setup(rb.default_amg_opts(seed=3, coarse_max=coarse_max, max_levels=max_levels, nu1=nu1, nu2=nu2))
    A = disc.aux_matrix(grid, synth.Soil(), synth.infiltration_bc(), 0, p, 1.0, None)
    h = amg.setup(A, 0.08, 3, coarse_max, max_levels=max_levels)
    assert info.levels == len(h.levels)
    ref = amg.vcycle(h, r, nu1, nu2)
    x = torch.empty(grid.n, dtype=torch.float64, device="cuda")
    for _ in range(2):  # launched, then replayed
        ctx.vcycle(torch.tensor(r, device="cuda"), x)
        assert np.abs(x.cpu().numpy() - ref).max() <= 1e-10 * np.abs(ref).max()
    ctx.close()
