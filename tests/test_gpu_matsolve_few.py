"""Matsubara solves of a few problems on either side of the line between the kept inverse (nb N^2 <= 4e5 for N = (ntau + 1) nf
unknowns, nf <= 4) and the LU spread over the GPU, against batches of 40 problems (LU, one block per problem).  The
equation's condition number here is below 1e3 and each solver's backward error below N 2^-53 with N <= 1300
unknowns, so the solutions agree to 1e3 * 1300 * 2 * 1.1e-16 = 3e-10 of the largest element in the worst case."""
import pytest
import torch

pytestmark = pytest.mark.gpu
TOL = 3e-10


@pytest.mark.parametrize("nf,ntau,few", [(1, 102, 37), (1, 105, 37), (1, 199, 10), (1, 200, 10), (2, 99, 10), (2, 100, 10), (4, 80, 3),
                                         (4, 78, 4), (1, 631, 1), (1, 632, 1), (1, 1260, 1), (8, 12, 1), (8, 40, 3)])
def test_few_against_batch(nf, ntau, few):
    import paper_1911_01211_gb300 as ng
    ng.load_library()
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
    g1 = grid(few)
    G1, S1, e1 = ng.Herm(g1), ng.Herm(g1), ng.Func(g1)
    S1.mat.copy_(S.mat[..., nb - few:])
    e1.val.copy_(eps.val[..., nb - few:])
    ctx.dyson_mat(g1, G1, S1, e1)
    assert ctx.status_sync() == (ng.NG_OK, 0)
    x, y = G.mat[..., nb - few:], G1.mat
    assert ((x - y).abs().amax((0, 1, 2)) <= TOL * x.abs().amax((0, 1, 2))).all()
    ctx.close()


def test_refined_solves_of_a_set_up():
    """A second-Born set-up above that line, whose solves keep the inverse for refinement: G^M afterwards against a solve for
    itself (LU) with the final self-energy, to the set-up's tolerance (a distance of 1e-12 summed over all elements,
    contracted once more) and the solvers' 3e-10 of the largest element."""
    import paper_1911_01211_gb300 as ng
    from paper_1911_01211_gb300 import workloads as wl
    ng.load_library()
    nk = 16
    w = wl.chain_kspace(nk=nk, nt=12, ntau=200, beta=4.0, h=0.05)
    g = ng.Grid(nt=w.nt, ntau=w.ntau, nf=1, nbatch=nk, korder=w.korder, h=w.h, beta=w.beta)
    ctx = ng.Context(w.korder)
    G, L, S = ng.Herm(g), ng.Herm(g, ldk=1), ng.Herm(g, ldk=1)
    e0, mf, U = ng.Func(g, values=torch.from_numpy(w.eps0)), ng.Func(g), ng.Func(g, scalar=True)
    U.val[:, 0, 0, 0] = torch.from_numpy(w.U.astype(complex))
    ctx.run_2b(g, G, L, S, e0, mf, U, corrector=w.corrector)
    G1 = ng.Herm(g)
    ctx.dyson_mat(g, G1, S, mf)
    assert ctx.status_sync() == (ng.NG_OK, 0)
    assert ((G.mat - G1.mat).abs().max() <= TOL * G1.mat.abs().max()).item()
    ctx.close()
