"""Residual, its norms and round-off scale, and the Jacobian on grids whose tiles have edges.

Grids above the cell variant's limit (40,000 cells): exact multiples of the tiles, ragged
ones, one layer, few columns, planes too thin for tiles; every mean and kind of face; a
batch stacked along z.  Bars: the FP64 parity bar of the residual and the Jacobian (1e-10
of the largest entry), norms 1e-12 relative, as in test_gpu_physics.py."""
import numpy as np
import pytest

from oracle import constitutive as cst
from oracle import discretization as disc
from paper_2112_05051_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SOIL = synth.Soil()
TOL = 1e-10
GRIDS = [(64, 32, 20), (35, 33, 37), (257, 160, 1), (8, 8, 700), (5, 3, 2700), (401, 17, 7), (16, 16, 157)]
MIXED = synth.BC(kind=(1, 0, 0, 1, 1, 1), value=(-22.0, 0, 0, -44.0, -61.5, -20.7))


def _nrel(a, b):
    return np.abs(a - b).max() / max(np.abs(b).max(), 1e-300)


def _check(rb, grid, bc, kmean, p, ks, s_old, dt, ctx, ref, jref, aref):
    pd, sd = torch.tensor(p, device="cuda"), torch.tensor(s_old, device="cuda")
    F = torch.full_like(pd, float("nan"))
    norms = ctx.residual(pd, sd, dt, F)
    assert _nrel(F.cpu().numpy(), ref[0]) <= TOL
    assert norms[0] == pytest.approx(np.linalg.norm(ref[0]), rel=1e-12)
    assert norms[1] == pytest.approx(np.abs(ref[0]).max(), rel=1e-12)
    F3 = torch.full_like(pd, float("nan"))
    n3 = ctx.residual3(pd, sd, dt, F3)
    assert torch.equal(F, F3) and n3[:2] == norms
    if ref[1] is not None:
        assert n3[2] == pytest.approx(ref[1], rel=1e-12)
    J7, A7 = (torch.full((7 * len(p),), float("nan"), dtype=torch.float64, device="cuda") for _ in range(2))
    ctx.jacobian(pd, dt, J7, A7)
    for got, want in ((J7, jref), (A7, aref)):
        got = got.cpu().numpy().reshape(7, -1).T
        np.testing.assert_array_equal(got == 0, want == 0)
        for col in range(7):
            assert _nrel(got[:, col], want[:, col]) <= TOL or np.abs(want[:, col]).max() == 0


@pytest.mark.parametrize("dims", GRIDS)
@pytest.mark.parametrize("kmean,bcname", [(0, "mixed"), (1, "paper"), (2, "mixed"), (3, "noflux"),
                                          (synth.kmean_split(1, 2), "mixed")])
def test_tiles_against_the_oracle(dims, kmean, bcname):
    from paper_2112_05051_gb300 import richards as rb
    rb.load()
    grid = synth.Grid(*dims, lx=1.0, ly=0.9, lz=1.3)
    bc = {"mixed": MIXED, "paper": synth.paper_infiltration_bc(grid, -61.5), "noflux": synth.all_noflux_bc()}[bcname]
    rng = np.random.default_rng(sum(dims) + kmean)
    p = rng.uniform(-70.0, -15.0, grid.n)
    p[::11] = 0.5
    ks = 10.0 ** rng.uniform(-4, -1, grid.n) if kmean else None
    s_old = cst.saturation(p + rng.uniform(-5, 5, grid.n), SOIL)
    F, scale = disc.residual(grid, SOIL, bc, kmean, p, s_old, 0.8, ks, with_scale=True)
    scale = float(np.linalg.norm(scale)) if np.ndim(scale) else float(scale)
    ctx = rb.Context(grid, SOIL, bc, kmean, ks)
    _check(rb, grid, bc, kmean, p, ks, s_old, 0.8, ctx, (F, scale),
           disc.jacobian_stencil(grid, SOIL, bc, kmean, p, 0.8, ks), disc.aux_stencil(grid, SOIL, bc, kmean, p, 0.8, ks))
    ctx.close()


@pytest.mark.parametrize("dims,nb", [((33, 30, 14), 3), ((64, 48, 5), 4)])
def test_batch_tiles_against_the_oracle(dims, nb):
    from paper_2112_05051_gb300 import richards as rb
    rb.load()
    grid = synth.Grid(*dims)
    rng = np.random.default_rng(4)
    p = rng.uniform(-70.0, -15.0, (nb, grid.n))
    ks = 10.0 ** rng.uniform(-4, -1, (nb, grid.n))
    s_old = cst.saturation(p + rng.uniform(-5, 5, p.shape), SOIL)
    bc = synth.infiltration_bc()
    F = np.concatenate([disc.residual(grid, SOIL, bc, 1, p[b], s_old[b], 0.5, ks[b]) for b in range(nb)])
    J = np.concatenate([disc.jacobian_stencil(grid, SOIL, bc, 1, p[b], 0.5, ks[b]) for b in range(nb)])
    A = np.concatenate([disc.aux_stencil(grid, SOIL, bc, 1, p[b], 0.5, ks[b]) for b in range(nb)])
    ctx = rb.BatchContext(grid, nb, SOIL, bc, 1, ks.reshape(-1), precision=rb.PREC_FP64)
    _check(rb, grid, bc, 1, p.reshape(-1), ks, s_old.reshape(-1), 0.5, ctx, (F, None), J, A)
    ctx.close()
