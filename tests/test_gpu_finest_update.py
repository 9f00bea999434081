"""amg_update on hierarchies whose finest level is kept scaled (l1-Jacobi) and on others (hybrid
Gauss-Seidel, one level): nothing is computed that the V-cycle does not read, and what it reads
follows the matrix.  Going to another pressure and back with the coarse levels kept gives the
first V-cycle bit for bit, and so does a refresh that follows such an update."""
import ctypes

import pytest

from paper_2112_05051_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _launches(rb):
    v = ctypes.c_longlong()
    rb.load().rich_kernel_launches(ctypes.byref(v))
    return v.value


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("opts", [{}, {"smoother": 1}, {"max_levels": 1}])
def test_update_of_the_finest_level(prec, opts):
    from paper_2112_05051_gb300 import richards as rb
    rb.load()
    grid = synth.Grid(21, 18, 15)
    gen = torch.Generator().manual_seed(7)
    p = [(-60.0 + 10.0 * k + 0.1 * torch.randn(grid.n, generator=gen, dtype=torch.float64)).cuda() for k in range(2)]
    r = torch.randn(grid.n, generator=gen, dtype=torch.float64).cuda()

    def context():
        ctx = rb.Context(grid, synth.Soil(), synth.infiltration_bc(), synth.KMEAN_ARITH, precision=prec)
        ctx.jacobian(p[0], 1.0)
        ctx.amg_setup(rb.default_amg_opts(seed=3, coarse_max=100, **opts))
        return ctx

    def cycle(ctx):
        z = torch.empty_like(r)
        ctx.vcycle(r, z)
        return z

    ctx = context()
    first = cycle(ctx)
    ctx.jacobian(p[1], 1.0)
    before = _launches(rb)
    ctx.amg_update(rb.AMG_SETUP_ONCE)
    if not opts:  # CSR values (exports), row factors, scaled stencil
        assert _launches(rb) - before <= 3
    other = cycle(ctx)
    assert not torch.equal(other, first)
    ctx.jacobian(p[0], 1.0)
    ctx.amg_update(rb.AMG_SETUP_ONCE)
    assert torch.equal(cycle(ctx), first)
    ctx.jacobian(p[1], 1.0)
    ctx.amg_update(rb.AMG_REFRESH)
    fresh = context()
    fresh.jacobian(p[1], 1.0)
    fresh.amg_update(rb.AMG_REFRESH)
    assert torch.equal(cycle(ctx), cycle(fresh))
    ctx.close()
    fresh.close()
