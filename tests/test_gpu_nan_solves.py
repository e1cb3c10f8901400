"""Dense solves of a problem whose matrix is NaN throughout, with the sign bit set and clear, beside finite problems:
the status is set, and the finite problems' results are bitwise those of a batch without it."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
NANS = [float("nan"), float(np.copysign(np.nan, -1.0))]


@pytest.fixture(scope="module")
def ng():
    import paper_1911_01211_gb300 as ng
    ng.load_library()
    return ng


def _case(ng, nb, nf, ntau, nt, k, bad, value):
    g = ng.Grid(nt=nt, ntau=ntau, nf=nf, nbatch=nb, korder=k, h=0.05, beta=4.0, mu=0.1)
    gen = torch.Generator(device="cuda").manual_seed(nf * 100 + ntau)
    G, S, eps = ng.Herm(g), ng.Herm(g), ng.Func(g)
    for t in S.tensors().values():
        torch.view_as_real(t).normal_(0.0, 0.1, generator=gen)
    a = torch.randn(eps.val.shape[1:], generator=gen, device="cuda", dtype=torch.float64)
    eps.val[:] = (a + a.transpose(0, 1))[None].to(eps.val.dtype)
    if bad is not None:
        for t in S.tensors().values():
            torch.view_as_real(t)[..., bad, :] = value
        torch.view_as_real(eps.val)[..., bad, :] = value
    return g, G, S, eps


# 40 problems: LU by panels, one block per problem; 3: the inverse over the whole GPU.  The last problem's matrix ends the
# workspace
@pytest.mark.parametrize("nb,nf,ntau", [(40, 1, 25), (40, 2, 20), (3, 1, 40), (3, 2, 15)])
@pytest.mark.parametrize("value", NANS)
@pytest.mark.parametrize("where", ["first", "last"])
def test_matsubara_and_start(ng, nb, nf, ntau, value, where):
    k, bad = 5, 0 if where == "first" else nb - 1
    ctx = ng.Context(k)
    out = []
    for b in (None, bad):
        g, G, S, eps = _case(ng, nb, nf, ntau, 2 * k + 2, k, b, value)
        ctx.dyson_mat(g, G, S, eps)
        ctx.dyson_start(g, G, S, eps)
        for n in range(k + 1, g.nt + 1):
            ctx.dyson_timestep(g, n, G, S, eps)
        flags = ctx.status_sync()[1]
        assert flags == 0 if b is None else flags & 1
        out.append(G)
    keep = [i for i in range(nb) if i != bad]
    for q in ("mat", "ret", "les", "tv"):
        x, y = getattr(out[0], q)[..., keep], getattr(out[1], q)[..., keep]
        assert torch.isfinite(torch.view_as_real(x)).all()
        assert torch.equal(x, y), q
    ctx.close()


@pytest.mark.parametrize("value", NANS)
def test_uneven_batch(ng, value):
    """Four orbital counts; the solves of the bad problem run on the warps of a block (40 x 40 for 8 orbitals)."""
    k, n, ntau = 5, 12, 12
    ctx = ng.Context(k)
    out = []
    for bad in (None, 0, 3):
        probs = [_case(ng, 1, nf, ntau, 12, k, 0 if i == bad else None, value) for i, nf in enumerate((8, 1, 2, 8, 4))]
        for i, p in enumerate(probs):
            gen = torch.Generator(device="cuda").manual_seed(i)
            for t in p[1].tensors().values():
                torch.view_as_real(t).normal_(0.0, 0.3, generator=gen)
        ctx.batch(*[[p[q] for p in probs] for q in range(4)]).step(n)
        flags = ctx.status_sync()[1]
        assert flags == 0 if bad is None else flags & 1
        out.append((bad, [p[1] for p in probs]))
    for bad, G in out[1:]:
        for i in range(5):
            if i != bad:
                for q in ("ret", "les", "tv"):
                    assert torch.equal(getattr(G[i], q), getattr(out[0][1][i], q)), (bad, i, q)
    ctx.close()
