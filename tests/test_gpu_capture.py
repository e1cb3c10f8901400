"""Steps captured into CUDA graphs after one eager step of the same grid, with forms that set in later than that step
(lanes per item, boundary with a lane per problem, source by FFT, digit products): the capture allocates nothing
and its replay gives what an eager step gives, to the rounding of the forms (tests/test_gpu_hist.py's bound)."""
import pytest
import torch

pytestmark = pytest.mark.gpu
TOL = 5e-12


@pytest.mark.parametrize("nk,nt,T,first,steps", [(128, 300, 100, 6, (12, 60, 300)), (64, 300, 150, 20, (21, 300)), (256, 60, 400, 12, (20, 60))])
@pytest.mark.parametrize("precision", [0, 2])
def test_captured_steps(nk, nt, T, first, steps, precision):
    import paper_1911_01211_gb300 as ng
    ng.load_library()
    k = 5
    g = ng.Grid(nt=nt, ntau=T, nf=1, nbatch=nk, korder=k, h=0.02, beta=4.0, mu=0.1)
    G, S, eps = ng.Herm(g), ng.Herm(g, ldk=1), ng.Func(g)
    gen = torch.Generator(device="cuda").manual_seed(nk)
    for H, s in ((G, 0.3), (S, 0.1)):
        for t in H.tensors().values():
            torch.view_as_real(t).normal_(0.0, s, generator=gen)
    ctx, own = ng.Context(k), ng.Context(k)
    if precision == 2:      # the double-float copies are allocated by the first step that reads them
        ctx.set_bulk_split(ng.NG_BULK_THREAD)
        ctx.dyson_timestep(g, first, G, S, eps, precision=precision)
        ctx.set_bulk_split(ng.NG_BULK_AUTO)
    ctx.dyson_timestep(g, first, G, S, eps, precision=precision)
    torch.cuda.synchronize()
    for n in steps:
        rows = (G.ret[n * (n + 1) // 2:(n + 1) * (n + 2) // 2], G.les[n * (n + 1) // 2:(n + 1) * (n + 2) // 2],
                G.tv[n * (T + 1):(n + 1) * (T + 1)])
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            ctx.dyson_timestep(g, n, G, S, eps, precision=precision)
        for r in rows:
            r.zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert ctx.status_sync() == (ng.NG_OK, 0)
        got = [r.clone() for r in rows]
        own.dyson_timestep(g, n, G, S, eps)
        assert own.status_sync() == (ng.NG_OK, 0)
        for x, y in zip(got, rows):
            assert ((x - y).abs().amax((0, 1, 2)) <= TOL * y.abs().amax((0, 1, 2))).all()
    ctx.close()
    own.close()
