"""FGMRES' orthogonalisation, whose Gram matrix is summed in 60-bit integers: after k steps
the iterate is that of an FGMRES in torch whose basis is orthogonalised by two sweeps of
modified Gram-Schmidt, with the library's own V-cycle and Jacobian product.

Right-hand sides spread over all cells and in a single one; sizes below and above the two
elements a thread takes at a time and the sixteen products between two carries; k so that
the basis fills one to three sweeps of four vectors and leaves each remainder.  Bar: both
bases are orthogonal to some units of rounding, and the iterate is a least-squares solution
with a Hessenberg matrix of condition below 1e4: 1e4 x 64 x 1.1e-16 < 1e-10."""
import pytest

from paper_2112_05051_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _reference(ctx, b, k):
    V, Z, H = [b / b.norm()], [], torch.zeros(k + 1, k, dtype=torch.float64, device="cuda")
    for j in range(k):
        z, w = torch.empty_like(b), torch.empty_like(b)
        ctx.vcycle(V[j], z)
        ctx.jacobian_apply(z, w)
        for _ in range(2):
            for i in range(j + 1):
                h = torch.dot(V[i], w)
                H[i, j] += h
                w = w - h * V[i]
        H[j + 1, j] = w.norm()
        V.append(w / w.norm())
        Z.append(z)
    g = torch.zeros(k + 1, 1, dtype=torch.float64, device="cuda")
    g[0] = b.norm()
    y = torch.linalg.lstsq(H, g).solution[:, 0]
    return sum(y[j] * Z[j] for j in range(k))


@pytest.mark.parametrize("dims,k", [((7, 5, 3), 2), ((19, 17, 13), 7), ((61, 53, 50), 8), ((160, 150, 131), 10)])
@pytest.mark.parametrize("spread", [True, False])
def test_iterate_against_modified_gram_schmidt(dims, k, spread):
    from paper_2112_05051_gb300 import richards as rb
    rb.load()
    grid = synth.Grid(*dims)
    gen = torch.Generator().manual_seed(sum(dims))
    z = (torch.arange(grid.nz, dtype=torch.float64) + 1.0) / (grid.nz + 1)
    p = (-61.5 + 40.8 * torch.exp(-(1.0 - z) / 0.2))[:, None, None].expand(grid.shape).reshape(-1)
    p = (p + torch.rand(grid.n, generator=gen, dtype=torch.float64) - 0.5).cuda()
    b = torch.zeros(grid.n, dtype=torch.float64)
    if spread:
        b = torch.randn(grid.n, generator=gen, dtype=torch.float64)
    else:
        b[grid.n // 2] = -3.0
    b = b.cuda()
    ctx = rb.Context(grid, synth.Soil(), synth.infiltration_bc(), synth.KMEAN_ARITH, None)
    ctx.jacobian(p, 1.0)
    ctx.amg_setup(rb.default_amg_opts(seed=4, coarse_max=20))
    ref = _reference(ctx, b, k)
    x = torch.zeros_like(b)
    ctx.krylov_solve(b, x, kind=rb.KRYLOV_FGMRES, restart=k + 2, eta=1e-30, maxit=k, check_status=False)
    assert float((x - ref).norm()) <= 1e-10 * float(ref.norm())
    ctx.close()
