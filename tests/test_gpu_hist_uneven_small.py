"""Digit-product sums of the uneven batch that are small beside the largest element on their scale (a weak coupling
between orbitals, a damped tail), element by element against the FP64 kernels of the same library (NG_BULK_THREAD).

G and Sigma are real positive matrices (1 on the diagonal, a coupling off it) times e^(-x (t - t')) (e^(-y tau) on the
left-mixing rows) and one phase per component, the last k rows of G and its Matsubara part are zero, one
component of Sigma at a time is not zero: an element of the new slice is a sum of terms of one sign, but for the product with
M_n^-1 = a_0 / h + h ..., whose off-diagonal part is below 1e-3 of the coupling.

Tolerance, relative to the element itself: N <= 8 (n + ntau + 1) <= 4100 terms; the FP64 kernels round two products a term
(2 N 2^-53), the digit products are off by at most 2^-45.8 of each task's sum: 9.2e-13 in all, 1e-12 with the factors."""
import pytest
import torch

pytestmark = pytest.mark.gpu
TOL = 1e-12


@pytest.fixture(scope="module")
def ng():
    import paper_1911_01211_gb300 as ng
    ng.load_library()
    return ng


def _fill(H, g, x, y, couple, sign):
    dev = "cuda"
    d = g.nf
    A = (torch.eye(d, device=dev, dtype=torch.float64) * (1.0 - couple) + couple)[None, :, :, None]
    for n in range(g.nt + 1):
        a = torch.exp(-x * (n - torch.arange(n + 1, device=dev, dtype=torch.float64)))[:, None, None, None] * A
        lo, hi = n * (n + 1) // 2, (n + 1) * (n + 2) // 2
        H.ret[lo:hi] = -1j * a
        H.les[lo:hi] = 1j * a
        tau = torch.arange(g.ntau + 1, device=dev, dtype=torch.float64)
        if sign < 0:
            tau = g.ntau - tau
        H.tv[n * (g.ntau + 1):(n + 1) * (g.ntau + 1)] = 1j * torch.exp(-0.5 * x * n - y * tau)[:, None, None, None] * A


@pytest.mark.parametrize("part", ["ret", "les", "tv"])
@pytest.mark.parametrize("n,T,k,x,y,couple,sign", [(400, 100, 5, 0.1, 0.2, 1e-9, 1), (300, 127, 3, 0.4, 0.5, 1e-3, -1),
                                                   (257, 60, 4, 0.01, 0.01, 1e-30, 1), (200, 70, 2, 0.05, 1.0, 0.0, -1)])
def test_each_element(ng, part, n, T, k, x, y, couple, sign):
    ctx = ng.Context(k)
    probs = []
    for i, nf in enumerate((1, 2, 4, 8)):
        g = ng.Grid(nt=n + i, ntau=T + 7 * i, nf=nf, nbatch=1, korder=k, h=0.02, beta=4.0)
        G, S, eps = ng.Herm(g), ng.Herm(g), ng.Func(g)
        _fill(G, g, x, y, couple, sign)
        _fill(S, g, x, y, couple, -sign)
        for q in ("ret", "les", "tv"):
            if q != part:
                getattr(S, q).zero_()
        lo, T1 = (n - k) * (n - k + 1) // 2, g.ntau + 1
        for t in (G.ret[lo:], G.les[lo:], G.tv[(n - k) * T1:]):
            t.zero_()
        probs.append((g, G, S, eps))
    b = ctx.batch(*[[p[q] for p in probs] for q in range(4)])
    out = []
    for mode in (ng.NG_BULK_THREAD, ng.NG_BULK_AUTO):
        ctx.set_bulk_split(mode)
        b.step(n)
        assert ctx.status_sync()[1] == 0
        row = n * (n + 1) // 2
        out.append([t.clone() for g, G, _, _ in probs
                    for t in (G.ret[row:row + n - k], G.les[row + 1:row + n - k], G.tv[n * (g.ntau + 1):(n + 1) * (g.ntau + 1)])])
    worst = 0.0
    for i, (x_, y_) in enumerate(zip(*out)):
        assert torch.equal(x_ == 0, y_ == 0), i
        big = x_.abs()
        err = (x_ - y_).abs()[big > 0] / big[big > 0]
        if err.numel():
            worst = max(worst, err.max().item())
    assert worst < TOL, worst
    ctx.close()
