"""The Jacobian and A_aux of grids whose planes fill no warp (fewer than 32 columns: a thread
per cell) and of the narrowest that march, alone and stacked in a batch, against the oracle.  Bar: the FP64 parity bar of the Jacobian, 1e-10 of the largest entry; zero entries
are zero."""
import numpy as np
import pytest

from oracle import discretization as disc
from paper_2112_05051_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SOIL = synth.Soil()
BC = synth.BC(kind=(1, 0, 0, 1, 1, 1), value=(-22.0, 0, 0, -44.0, -61.5, -20.7))


@pytest.mark.parametrize("kmean", [0, 1, 2, 3, synth.kmean_split(3, 1)])
@pytest.mark.parametrize("dims,nb", [((1, 1, 1), 1), ((1, 1, 700), 1), ((1, 1, 33), 3), ((3, 1, 129), 1), ((1, 7, 50), 2),
                                     ((9, 7, 41), 1), ((9, 7, 6), 5), ((5, 6, 6), 5),
                                     ((31, 1, 65), 1), ((8, 4, 65), 1), ((8, 8, 40), 1), ((63, 1, 3000), 1)])
def test_narrow_planes_against_the_oracle(dims, nb, kmean):
    from paper_2112_05051_gb300 import richards as rb
    rb.load()
    grid = synth.Grid(*dims, lx=1.0, ly=0.9, lz=1.3)
    rng = np.random.default_rng(sum(dims) + nb)
    p = rng.uniform(-70.0, -15.0, (nb, grid.n))
    p[:, ::11] = 0.5
    ks = 10.0 ** rng.uniform(-4, -1, (nb, grid.n))
    if nb == 1:
        ctx = rb.Context(grid, SOIL, BC, kmean, ks[0])
    else:
        ctx = rb.BatchContext(grid, nb, SOIL, BC, kmean, ks.reshape(-1), precision=rb.PREC_FP64)
    J7, A7 = (torch.full((7 * p.size,), float("nan"), dtype=torch.float64, device="cuda") for _ in range(2))
    ctx.jacobian(torch.tensor(p.reshape(-1), device="cuda"), 0.8, J7, A7)
    for got, stencil in ((J7, disc.jacobian_stencil), (A7, disc.aux_stencil)):
        want = np.concatenate([stencil(grid, SOIL, BC, kmean, p[b], 0.8, ks[b]) for b in range(nb)])
        got = got.cpu().numpy().reshape(7, -1).T
        np.testing.assert_array_equal(got == 0, want == 0)
        assert np.abs(got - want).max() <= 1e-10 * np.abs(want).max()
    ctx.close()
