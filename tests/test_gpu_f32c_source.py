"""The left-mixing row of an NG_F32C step with its Matsubara source by FFT, whose columns next to the ends of the tau axis the
transform's warps complete, against the direct sums: axes on which most or all columns lie next to an end, batches on
either side of the block sizes (152, 304 problems), shared and per-problem self-energies.

Tolerance: the direct sums read FP32 copies (2^-24 of each factor), sum |terms| is below 40 times the largest
element: 2 * 40 * 2^-24 = 4.8e-6 of the largest element."""
import pytest
import torch

pytestmark = pytest.mark.gpu
TOL = 4.8e-6


@pytest.mark.parametrize("nf,nk,shared", [(1, 3, True), (1, 64, True), (1, 160, False), (1, 310, True), (2, 2, False), (2, 65, True)])
@pytest.mark.parametrize("T,k", [(4, 1), (12, 5), (13, 5), (24, 5), (25, 4), (40, 5), (127, 3)])
def test_ends_of_the_axis(nf, nk, shared, T, k):
    import paper_1911_01211_gb300 as ng
    ng.load_library()
    n = 2 * k + 3
    g = ng.Grid(nt=n, ntau=T, nf=nf, nbatch=nk, korder=k, h=0.02, beta=4.0, mu=0.1)
    G, S, eps = ng.Herm(g), ng.Herm(g, ldk=1 if shared else None), ng.Func(g)
    gen = torch.Generator(device="cuda").manual_seed(T)
    for H, s in ((G, 0.3), (S, 1.0)):
        for t in H.tensors().values():
            torch.view_as_real(t).normal_(0.0, s, generator=gen)
    out = []
    for src in (ng.NG_TVSRC_DIRECT, ng.NG_TVSRC_AUTO):
        ctx = ng.Context(k)
        ctx.set_tv_source(src)
        ctx.dyson_timestep(g, n, G, S, eps, precision=ng.NG_F32C)
        assert ctx.status_sync()[1] == 0
        out.append(G.tv[n * (T + 1):].clone())
        ctx.close()
    x, y = out
    assert ((x - y).abs().amax((0, 1, 2)) <= TOL * x.abs().amax((0, 1, 2))).all()
