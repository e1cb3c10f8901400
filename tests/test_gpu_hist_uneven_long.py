"""Digit-product steps of problems long enough that a task takes more than 16 tiles of the contraction (from 384
tiles on: nf (n + 1) > 6144), where the number of chunks falls from 24 to 23 as n grows, against the FP64 kernels of
the same library (NG_BULK_THREAD).

Tolerance: each sum has N <= 8 (n + ntau + 1) <= 7000 terms, the FP64 kernels round each addition to 2^-53 of a
partial sum below sum |terms|; for random terms sum |terms| is about sqrt(N) / 3 < 30 times the largest result,
so the two differ by at most 7000 * 30 * 2^-53 = 2.4e-11 of the largest element."""
import pytest
import torch

pytestmark = pytest.mark.gpu
TOL = 2.4e-11


@pytest.mark.parametrize("nf,n,nt,T,k", [(8, 768, 782, 33, 5), (8, 785, 785, 100, 4)])
def test_long_problem(nf, n, nt, T, k):
    import paper_1911_01211_gb300 as ng
    ng.load_library()
    g = ng.Grid(nt=nt, ntau=T, nf=nf, nbatch=1, korder=k, h=0.02, beta=4.0, mu=0.1)
    G, S, eps = ng.Herm(g), ng.Herm(g), ng.Func(g)
    gen = torch.Generator(device="cuda").manual_seed(n)
    for H, scale in ((G, 0.3), (S, 0.0125)):
        for t in H.tensors().values():
            torch.view_as_real(t).normal_(0.0, scale, generator=gen)
    e = torch.randn(eps.val.shape[:-1], dtype=torch.float64, device="cuda", generator=gen)
    eps.val[..., 0] = (e + e.transpose(1, 2)).to(eps.val.dtype)
    lo, hi, T1 = n * (n + 1) // 2, (n + 1) * (n + 2) // 2, T + 1
    ctx = ng.Context(k)
    out = []
    for mode in (ng.NG_BULK_THREAD, ng.NG_BULK_AUTO):
        ctx.set_bulk_split(mode)
        rows = G.ret[lo:hi], G.les[lo:hi], G.tv[n * T1:(n + 1) * T1]
        for r in rows:
            r.zero_()
        ctx.dyson_timestep(g, n, G, S, eps)
        assert ctx.status_sync()[1] == 0
        out.append([r.clone() for r in rows])
    for x, y in zip(*out):
        assert ((x - y).abs().max() / x.abs().max()).item() < TOL
    ctx.close()
