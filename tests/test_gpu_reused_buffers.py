"""The step of 4 and 8 orbitals on buffers that were used before with another time step, mesh of tau and chemical
potential, by the same context: as by a context of its own."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nf,nb", [(4, 1), (4, 3), (8, 1)])
def test_other_grid_same_buffers(nf, nb):
    import paper_1911_01211_gb300 as ng
    ng.load_library()
    n, k = 40, 5
    grids = [ng.Grid(nt=n, ntau=30, nf=nf, nbatch=nb, korder=k, h=h, beta=b, mu=m) for h, b, m in ((0.02, 4.0, 0.1), (0.05, 7.0, -0.3))]
    G, S, eps = ng.Herm(grids[0]), ng.Herm(grids[0]), ng.Func(grids[0])
    gen = torch.Generator(device="cuda").manual_seed(nf + nb)
    for H, s in ((G, 0.3), (S, 0.1 / nf)):
        for t in H.tensors().values():
            torch.view_as_real(t).normal_(0.0, s, generator=gen)
    row, T1 = n * (n + 1) // 2, grids[0].ntau + 1
    both = ng.Context(k)
    for g in grids + grids[:1]:
        own = ng.Context(k)
        out = []
        for ctx in (both, own):
            ctx.dyson_timestep(g, n, G, S, eps)
            assert ctx.status_sync()[1] == 0
            out.append([t.clone() for t in (G.ret[row:], G.les[row:], G.tv[n * T1:])])
        for x, y in zip(*out):
            assert torch.equal(x, y)
        own.close()
    both.close()
