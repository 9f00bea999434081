"""FCG's iterations as a device-side loop against single launches of the same kernels.

graph = 0 launches every iteration and reads its decisions; graph = 1 runs the loop as one
CUDA graph from the second application of a hierarchy on.  Same kernels, so iterates,
counts and reasons agree bit for bit: at the limits of the loop (one to three iterations,
maxit, a zero and a non-finite right-hand side, a stagnation window), with a fresh
solution buffer every time, and after a refresh."""
import numpy as np
import pytest

from paper_2112_05051_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _run(graph, prec, dims, levels):
    from paper_2112_05051_gb300 import richards as rb
    rb.load()
    grid = synth.Grid(*dims)
    rng = np.random.default_rng(7)
    z = (np.arange(grid.nz) + 1.0) / (grid.nz + 1)
    front = -61.5 + 40.8 * np.exp(-(1.0 - z) / 0.2)
    p = torch.tensor(np.broadcast_to(front[:, None, None], grid.shape).ravel() + rng.uniform(-0.3, 0.3, grid.n),
                     device="cuda")
    b = torch.tensor(rng.standard_normal(grid.n), device="cuda")
    ctx = rb.Context(grid, synth.Soil(), synth.infiltration_bc(), synth.KMEAN_ARITH, None, precision=prec)
    ctx.jacobian(p, 1.0)
    ctx.amg_setup(rb.default_amg_opts(seed=3, coarse_max=100, max_levels=levels, graph=graph))
    bad = b.clone()
    bad[grid.n // 2] = float("nan")
    out = []

    def solve(rhs, **kw):
        x = torch.full_like(b, float("nan"))
        s, st = ctx.krylov_solve(rhs, x, kind=rb.KRYLOV_FCG, check_status=False, **kw)
        out.append((s, st.iterations, st.converged, st.res0, st.res, x.cpu().numpy()))

    for _ in range(2):
        for kw in (dict(maxit=1), dict(maxit=2), dict(maxit=3), dict(eta=1e-9), dict(eta=1e-30, maxit=35, stall=0.999),
                   dict(eta=0.5)):
            solve(b, **kw)
        solve(torch.zeros_like(b))
        solve(bad)
        solve(b, eta=1e-9)
        ctx.jacobian(p + 0.5, 2.0)
        ctx.amg_update(rb.AMG_REFRESH)
    ctx.close()
    return out


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("dims,levels", [((24, 22, 20), 10), ((33, 5, 41), 2), ((1, 1, 60), 1)])
def test_loop_equals_single_launches(dims, levels, prec):
    one, loop = _run(0, prec, dims, levels), _run(1, prec, dims, levels)
    assert [r[0] for r in one[:3]] == [-4, -4, -4] and [r[1] for r in one[:3]] == [1, 2, 3] or levels == 1
    assert one[6][0] == 0 and one[6][1] == 0 and not one[6][5].any()  # b = 0: x = 0 at once
    assert one[7][0] == -7
    for a, c in zip(one, loop):
        assert a[:3] == c[:3]
        np.testing.assert_array_equal(np.array(a[3:5]), np.array(c[3:5]))
        if a[0] != -7:
            np.testing.assert_array_equal(a[5], c[5])
