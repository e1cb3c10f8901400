"""Digit-product history sums (nf = 1) that are small beside the largest element of their 128 x 128 unit, element by
element against the FP64 kernels of the same library (NG_BULK_THREAD).

G falls by e^-x per time step along one axis and by e^-y per step of tau, the self-energy falls by e^-x per step
as well, all terms of a sum have one sign, and the last k rows of G and its Matsubara part are zero, so that an element
of the new slice is a history sum and nothing else; one component of the self-energy at a time is not zero.

Tolerance, relative to the element itself: at most N = n + ntau + 1 <= 800 terms of one sign; the FP64 kernels round
each of the two real products of a term and add it (2 N 2^-53), the digit products are off by at most 2^-45.8 of a
unit's sum and 2^-53 for each of the few units and factors: 1600 2^-53 + 2^-45.8 + 20 2^-53 = 2.0e-13."""
import pytest
import torch

pytestmark = pytest.mark.gpu
TOL = 2.0e-13


@pytest.fixture(scope="module")
def ng():
    import paper_1911_01211_gb300 as ng
    ng.load_library()
    return ng


def _fill(H, g, x, y, sign):
    """ret: -i a, les: i a, tv: i a with a = e^(-x |t - t'|) (e^(-x t - y tau) for tv), each problem on another scale."""
    dev = "cuda"
    scale = torch.exp2(-2.0 * (torch.arange(H.ldk, device=dev, dtype=torch.float64) % 20))
    for n in range(g.nt + 1):
        d = n - torch.arange(n + 1, device=dev, dtype=torch.float64)
        a = torch.exp(-x * d)[:, None, None, None] * scale
        lo, hi = n * (n + 1) // 2, (n + 1) * (n + 2) // 2
        H.ret[lo:hi] = -1j * a
        H.les[lo:hi] = 1j * a
        tau = torch.arange(g.ntau + 1, device=dev, dtype=torch.float64)
        if sign < 0:
            tau = g.ntau - tau
        H.tv[n * (g.ntau + 1):(n + 1) * (g.ntau + 1)] = 1j * torch.exp(-0.5 * x * n - y * tau)[:, None, None, None] * scale


@pytest.mark.parametrize("part", ["ret", "les", "tv"])
@pytest.mark.parametrize("nk,n,T,k,shared,x,y,sign", [(24, 500, 127, 5, True, 0.1, 0.3, 1), (20, 500, 140, 4, False, 0.3, 0.5, -1),
                                                      (17, 400, 300, 2, True, 1.0, 0.1, -1), (130, 200, 127, 5, False, 0.02, 1.0, 1)])
def test_each_element(ng, part, nk, n, T, k, shared, x, y, sign):
    g = ng.Grid(nt=n, ntau=T, nf=1, nbatch=nk, korder=k, h=0.02, beta=4.0)
    G, S, eps = ng.Herm(g), ng.Herm(g, ldk=1 if shared else None), ng.Func(g)
    _fill(G, g, x, y, sign)
    _fill(S, g, x, y, -sign)
    G.mat.zero_()
    S.mat.zero_()
    for q in ("ret", "les", "tv"):
        if q != part:
            getattr(S, q).zero_()
    lo, T1 = (n - k) * (n - k + 1) // 2, T + 1
    for t in (G.ret[lo:], G.les[lo:], G.tv[(n - k) * T1:]):
        t.zero_()
    ctx = ng.Context(k)
    out = []
    for mode in (ng.NG_BULK_THREAD, ng.NG_BULK_AUTO):
        ctx.set_bulk_split(mode)
        row = n * (n + 1) // 2
        ctx.dyson_timestep(g, n, G, S, eps)
        assert ctx.status_sync()[1] == 0
        out.append({"ret": G.ret[row:row + n - k].clone(), "les": G.les[row + 1:row + n - k].clone(), "tv": G.tv[n * T1:].clone()})
    worst = 0.0
    for q in out[0]:
        a, b = out[0][q], out[1][q]
        assert torch.equal(a == 0, b == 0), q
        big = a.abs()
        err = (a - b).abs()[big > 0] / big[big > 0]
        if err.numel():
            worst = max(worst, err.max().item())
    assert worst < TOL, worst
    ctx.close()
