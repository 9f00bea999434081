"""One batch context used both ways: step_batch (FCG over nbatch problems, each with its own
scalars) and the lone calls it inherits, krylov_solve and step (one problem over the whole
stack), in both orders and with the iterations as a graph (graph = 1) or launched singly
(graph = 0).  The same kernels run either way, so iterates, counts and statuses agree bit for
bit; a lone solve also meets its own tolerance on the whole stack."""
import numpy as np
import pytest

from paper_2112_05051_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _run(order, graph, prec, nbatch):
    from paper_2112_05051_gb300 import richards as rb
    rb.load()
    grid = synth.Grid(14, 13, 12)
    ks = np.concatenate([synth.ks_field(grid, 40 + b, 0.5, (4.0, 4.0, 2.0)) for b in range(nbatch)])
    ctx = rb.BatchContext(grid, nbatch, synth.Soil(), synth.infiltration_bc(), synth.KMEAN_ARITH, ks, precision=prec)
    opts = rb.default_newton_opts(kind=rb.KRYLOV_FCG, seed=3, coarse_max=100, smooth_levels=2, graph=graph)
    p = torch.full((ctx.n,), synth.P_INITIAL, dtype=torch.float64, device="cuda")
    b = torch.randn(ctx.n, generator=torch.Generator().manual_seed(5), dtype=torch.float64).cuda()
    ctx.jacobian(p - 1.0, 0.25)
    ctx.amg_setup(opts.amg)
    out = []
    for op in order:
        if op == "batch":
            status, st = ctx.step_batch(p, 0.25, opts)
            out.append((status, [s.linear_its for s in st], [s.newton_its for s in st], p.cpu().numpy()))
        elif op == "step":
            status, st = ctx.step(p, 0.25, opts, check_status=False)
            out.append((status, st.linear_its, st.newton_its, p.cpu().numpy()))
        else:
            x, y = torch.full_like(b, float("nan")), torch.empty_like(b)
            status, st = ctx.krylov_solve(b, x, kind=rb.KRYLOV_FCG, check_status=False)
            ctx.jacobian_apply(x, y)
            assert status == 0 and float((y - b).norm()) <= 1.01e-7 * float(b.norm())
            out.append((status, st.iterations, st.res, x.cpu().numpy()))
    ctx.close()
    return out


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("order,nbatch", [(("batch", "solve", "batch", "solve"), 3), (("solve", "batch", "solve"), 3),
                                          (("step", "batch", "step"), 2), (("batch", "solve"), 1)])
def test_batch_and_lone_solves_on_one_context(order, nbatch, prec):
    for a, b in zip(_run(order, 0, prec, nbatch), _run(order, 1, prec, nbatch)):
        assert a[:3] == b[:3]
        np.testing.assert_array_equal(a[3], b[3])


@pytest.mark.parametrize("graph", [0, 1])
def test_batch_without_iterations(graph):
    """maxit = 0: no iteration is made, also not by a loop captured before, and no problem moves."""
    from paper_2112_05051_gb300 import richards as rb
    rb.load()
    grid = synth.Grid(9, 8, 7)
    ctx = rb.BatchContext(grid, 2, synth.Soil(), synth.infiltration_bc(), synth.KMEAN_ARITH, None)
    kw = dict(kind=rb.KRYLOV_FCG, seed=3, coarse_max=100, graph=graph)
    p = torch.full((ctx.n,), synth.P_INITIAL, dtype=torch.float64, device="cuda")
    for warm in (False, True):
        if warm:  # a step whose solves run (and capture) the loop, wherever it ends
            assert max(s.linear_its for s in ctx.step_batch(p, 0.25, rb.default_newton_opts(**kw))[1]) > 2
        before = p.clone()
        status, st = ctx.step_batch(p, 0.25, rb.default_newton_opts(maxit=0, **kw))
        assert status == [-4, -4] and [s.linear_its for s in st] == [0, 0]
        assert torch.equal(p, before)
    ctx.close()


def test_launch_count_of_a_batch_whose_first_problem_sits_out():
    """rich_kernel_launches counts the loop's iterations by the problem that makes most of them:
    the same count with graph = 0 and 1 where the first problem is steady from the start
    (hydrostatic, no flux) and the second is not."""
    import ctypes

    from paper_2112_05051_gb300 import richards as rb
    rb.load()
    grid = synth.Grid(9, 8, 7)
    z = (np.arange(grid.nz) + 1.0) / (grid.nz + 1)
    steady = np.broadcast_to((-30.0 - z)[:, None, None], grid.shape).ravel()
    wet = steady + np.random.default_rng(2).uniform(-3, 3, grid.n)
    p0 = torch.tensor(np.concatenate([steady, wet]), device="cuda")

    def launches():
        v = ctypes.c_longlong()
        rb.load().rich_kernel_launches(ctypes.byref(v))
        return v.value

    counts = []
    for graph in (0, 0, 1):  # the first run meets the autotuner's timings
        ctx = rb.BatchContext(grid, 2, synth.Soil(), synth.all_noflux_bc(), synth.KMEAN_ARITH, None)
        opts = rb.default_newton_opts(kind=rb.KRYLOV_FCG, seed=3, coarse_max=100, graph=graph)
        n0 = launches()
        status, st = ctx.step_batch(p0.clone(), 0.25, opts)
        counts.append(launches() - n0)
        assert status[0] == 0 and st[0].linear_its == 0 and st[1].linear_its > 4
        ctx.close()
    assert counts[1] == counts[2]
