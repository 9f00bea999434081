"""The V-cycle on grids whose finest-level kernels march several layers per thread (above
1.2M cells), against the same cycle from the exported matrices in torch FP64.

The exported levels and prolongators are what the oracle tests pin on small grids; here
they define the reference: l1-Jacobi sweeps, residual, R = P^T, dense coarsest solve.
Layer counts that are no multiple of the layers per thread, odd lines.  Bars as in the
oracle tests: 1e-10 (FP64) and 1e-4 (MIXED) of the largest entry."""
import numpy as np
import pytest

from paper_2112_05051_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _csr(rp, col, val, shape):
    t = lambda a, d: torch.as_tensor(a, dtype=d, device="cuda")  # noqa: E731
    return torch.sparse_csr_tensor(t(rp, torch.int64), t(col, torch.int64), t(val, torch.float64), shape)


def _mv(A, x):
    return (A @ x.unsqueeze(1)).squeeze(1)


def _cycle(levels, l, b, nu):
    A, l1, P, R = levels[l]
    if l == len(levels) - 1:
        return torch.linalg.solve(A.to_dense(), b)
    x = torch.zeros_like(b)
    for _ in range(nu):
        x = x + (b - _mv(A, x)) / l1
    x = x + _mv(P, _cycle(levels, l + 1, _mv(R, b - _mv(A, x)), nu))
    for _ in range(nu):
        x = x + (b - _mv(A, x)) / l1
    return x


@pytest.mark.parametrize("dims", [(130, 101, 99), (161, 129, 121)])
@pytest.mark.parametrize("nu", [1, 2])
def test_large_grid_vcycle_against_exported_levels(dims, nu):
    from paper_2112_05051_gb300 import richards as rb
    rb.load()
    grid = synth.Grid(*dims)
    rng = np.random.default_rng(sum(dims))
    z = (np.arange(grid.nz) + 1.0) / (grid.nz + 1)
    p = np.broadcast_to((-61.5 + 40.8 * np.exp(-(1.0 - z) / 0.2))[:, None, None], grid.shape).ravel()
    p = torch.tensor(p + rng.uniform(-0.5, 0.5, grid.n), device="cuda")
    r = torch.tensor(rng.standard_normal(grid.n), device="cuda")
    opts = rb.default_amg_opts(seed=2, nu1=nu, nu2=nu, smooth_levels=2)
    for prec, tol in ((rb.PREC_FP64, 1e-10), (rb.PREC_MIXED, 1e-4)):
        ctx = rb.Context(grid, synth.Soil(), synth.infiltration_bc(), synth.KMEAN_ARITH, None, precision=prec)
        ctx.jacobian(p, 1.0)
        info = ctx.amg_setup(opts)
        if prec == rb.PREC_FP64:
            levels = []
            for l in range(info.levels):
                _, rp, col, val = ctx.export_level(l, info)
                n = info.n[l]
                A = _csr(rp, col, val, (n, n))
                l1 = torch.as_tensor(np.add.reduceat(np.abs(val), rp[:-1]), device="cuda")
                P = R = None
                if l + 1 < info.levels:
                    import scipy.sparse as sp
                    Pm = sp.csr_matrix(tuple(reversed(ctx.export_prolongator(l, info))), shape=(n, info.n[l + 1]))
                    Rm = Pm.T.tocsr()
                    P = _csr(Pm.indptr, Pm.indices, Pm.data, Pm.shape)
                    R = _csr(Rm.indptr, Rm.indices, Rm.data, Rm.shape)
                levels.append((A, l1, P, R))
            ref = _cycle(levels, 0, r, nu)
        for _ in range(2):
            x = torch.empty_like(r)
            ctx.vcycle(r, x)
            assert float((x - ref).abs().max()) <= tol * float(ref.abs().max())
        ctx.close()
