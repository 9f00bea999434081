"""FGMRES where the new vector all but lies in the basis: an exact inverse of A_aux as the
preconditioner (one level) of a Jacobian that differs from it by little, so that w - V h is
less than 1e-2 of w and the explicit second pass of the orthogonalisation runs.

After k steps the iterate is that of an FGMRES in torch whose basis is orthogonalised by two
sweeps of modified Gram-Schmidt.  Bar as in test_gpu_gram.py: 1e-10 of the iterate (the
Hessenberg matrix is near the identity)."""
import pytest

from paper_2112_05051_gb300 import synth
from test_gpu_gram import _reference

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("head,k", [(0.5, 1), (2.0, 2), (4.0, 3)])
@pytest.mark.parametrize("dims", [(9, 8, 7), (16, 16, 12)])
def test_iterate_with_explicit_second_projections(dims, head, k):
    from paper_2112_05051_gb300 import richards as rb
    rb.load()
    grid = synth.Grid(*dims)
    gen = torch.Generator().manual_seed(sum(dims))
    p = (-head * (1.0 + 0.2 * torch.rand(grid.n, generator=gen, dtype=torch.float64))).cuda()
    b = torch.randn(grid.n, generator=gen, dtype=torch.float64).cuda()
    ctx = rb.Context(grid, synth.Soil(), synth.infiltration_bc(), synth.KMEAN_ARITH, None)
    ctx.jacobian(p, 1.0)
    ctx.amg_setup(rb.default_amg_opts(seed=4, max_levels=1))
    z, w = torch.empty_like(b), torch.empty_like(b)
    ctx.vcycle(b / b.norm(), z)
    ctx.jacobian_apply(z, w)
    left = w - torch.dot(w, b) / torch.dot(b, b) * b
    assert float(left.norm()) < 1e-2 * float(w.norm())  # the explicit pass's condition
    ref = _reference(ctx, b, k)
    x = torch.zeros_like(b)
    ctx.krylov_solve(b, x, kind=rb.KRYLOV_FGMRES, restart=k + 2, eta=1e-30, maxit=k, check_status=False)
    assert float((x - ref).norm()) <= 1e-10 * float(ref.norm())
    ctx.close()
