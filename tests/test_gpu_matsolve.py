"""The two dense solvers of the Matsubara equation against each other: batches factorise one block per
problem (panels of 16, 8 or 4 columns by the number of unknowns), a few problems keep the inverse.  The
equation's condition number here is below 1e3 and each solver's backward error below N 2^-53 with
N <= 1622 unknowns, so the solutions agree to 1e3 * 1622 * 2 * 1.1e-16 = 4e-10 of the largest element in
the worst case."""
import pytest
import torch

pytestmark = pytest.mark.gpu
TOL = 4e-10


@pytest.fixture(scope="module")
def ng():
    import paper_1911_01211_gb300 as ng
    ng.load_library()
    return ng


@pytest.mark.parametrize("nf,ntau", [(1, 12), (1, 47), (1, 63), (2, 40), (4, 33), (8, 20), (1, 800), (2, 810)])
def test_batch_against_single(ng, nf, ntau):
    nb, k = 40, 5
    ctx = ng.Context(k)
    gen = torch.Generator(device="cuda").manual_seed(nf * 1000 + ntau)

    def grid(n):
        return ng.Grid(nt=2 * k + 2, ntau=ntau, nf=nf, nbatch=n, korder=k, h=0.05, beta=4.0, mu=0.1)

    def hermitian(n):
        a = torch.view_as_complex(torch.randn((n, nf, nf, 2), generator=gen, device="cuda", dtype=torch.float64))
        return 0.5 * (a + a.transpose(1, 2).conj())

    g = grid(nb)
    G, S, eps = ng.Herm(g), ng.Herm(g), ng.Func(g)
    ctx.green_from_H_const(g, S, hermitian(nb).cpu().numpy(), scale=0.3)
    eps.val[:] = hermitian(nb).permute(1, 2, 0)[None]
    ctx.dyson_mat(g, G, S, eps)
    assert ctx.status_sync() == (ng.NG_OK, 0)
    for kb in (0, nb - 1):
        g1 = grid(1)
        G1, S1, e1 = ng.Herm(g1), ng.Herm(g1), ng.Func(g1)
        S1.mat.copy_(S.mat[..., kb:kb + 1])
        e1.val.copy_(eps.val[..., kb:kb + 1])
        ctx.dyson_mat(g1, G1, S1, e1)
        assert ctx.status_sync() == (ng.NG_OK, 0)
        x, y = G.mat[..., kb], G1.mat[..., 0]
        assert ((x - y).abs().max() / x.abs().max()).item() < TOL
