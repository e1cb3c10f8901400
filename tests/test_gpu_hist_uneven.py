"""Steps of the uneven batch and of nf = 4, 8 whose history sums run as digit products on the tensor
cores, against the FP64 kernels of the same library (NG_BULK_THREAD, themselves pinned to the oracle):
edges of the 128-element tasks and 16 x 16 tiles for every orbital count, problems of different length
and orbital count side by side, zeros, scale growth and non-finite values.

Tolerance: each sum has N <= 8 (n + ntau + 1) <= 6000 terms, the FP64 kernels round each addition to 2^-53 of
a partial sum below sum |terms|; for random terms sum |terms| is about sqrt(N) / 3 < 30 times the largest
result, so the two differ by at most 6000 * 30 * 2^-53 = 2e-11 of the largest element."""
import pytest
import torch

pytestmark = pytest.mark.gpu
TOL = 2e-11


@pytest.fixture(scope="module")
def ng():
    import paper_1911_01211_gb300 as ng
    ng.load_library()
    return ng


def _random(H, seed, scale):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    for t in H.tensors().values():
        torch.view_as_real(t).normal_(0.0, scale, generator=gen)


def _problem(ng, seed, nf, nt, T, k):
    g = ng.Grid(nt=nt, ntau=T, nf=nf, nbatch=1, korder=k, h=0.02, beta=4.0, mu=0.1)
    G, S, eps = ng.Herm(g), ng.Herm(g), ng.Func(g)
    _random(G, seed, 0.3)
    _random(S, seed + 100, 0.1 / nf)
    e = torch.randn(eps.val.shape[:-1], dtype=torch.float64, device="cuda", generator=torch.Generator(device="cuda").manual_seed(seed))
    eps.val[..., 0] = (e + e.transpose(1, 2)).to(eps.val.dtype)
    return g, G, S, eps


def _slices(probs, n):
    out = []
    for g, G, _, _ in probs:
        T1, lo, hi = g.ntau + 1, n * (n + 1) // 2, (n + 1) * (n + 2) // 2
        out.append({"ret": G.ret[lo:hi], "les": G.les[lo:hi], "tv": G.tv[n * T1:(n + 1) * T1]} if n <= g.nt else {})
    return out


def _both(ng, ctx, probs, n, call):
    out = []
    for mode in (ng.NG_BULK_THREAD, ng.NG_BULK_AUTO):
        ctx.set_bulk_split(mode)
        for s in _slices(probs, n):
            for v in s.values():
                v.zero_()
        call()
        flags = ctx.status_sync()[1]
        out.append(([{q: v.clone() for q, v in s.items()} for s in _slices(probs, n)], flags))
    return out


def _check(a, b):
    for i, (x, y) in enumerate(zip(a, b)):
        for q in x:
            err = ((x[q] - y[q]).abs().max() / x[q].abs().max()).item()
            assert err < TOL, (i, q, err)


BATCH = [  # n, k, problems (nf, nt - n, ntau)
    (300, 5, [(1, 0, 300), (2, 3, 127), (4, 0, 128), (8, 1, 60), (8, 0, 33), (1, 7, 600)]),
    (257, 3, [(8, 0, 31), (4, 9, 300), (2, 0, 129), (1, 0, 255), (4, -100, 50)]),
    (128, 1, [(8, 0, 100), (2, 0, 500), (4, 0, 64)]),
    (420, 4, [(4, 0, 280), (2, 0, 64), (8, 0, 40)]),
]


@pytest.mark.parametrize("n,k,shape", BATCH)
@pytest.mark.parametrize("threads", [64, 256])
def test_batch_step(ng, n, k, shape, threads):
    probs = [_problem(ng, 10 * i + 1, nf, n + dn, T, k) for i, (nf, dn, T) in enumerate(shape)]
    ctx = ng.Context(k)
    b = ctx.batch(*[[p[q] for p in probs] for q in range(4)])
    (x, fx), (y, fy) = _both(ng, ctx, probs, n, lambda: b.step(n, threads=threads))
    assert fx == fy == 0
    _check(x, y)


@pytest.mark.parametrize("nf,n,T,k", [(8, 200, 75, 5), (4, 330, 200, 2), (8, 129, 127, 4)])
def test_timestep(ng, nf, n, T, k):
    p = _problem(ng, 3, nf, n, T, k)
    ctx = ng.Context(k)
    (x, fx), (y, fy) = _both(ng, ctx, [p], n, lambda: ctx.dyson_timestep(p[0], n, p[1], p[2], p[3]))
    assert fx == fy == 0
    _check(x, y)


@pytest.mark.parametrize("grow", [1.0, -1.0])
def test_scale_growth_and_zeros(ng, grow):
    """History that grows (or falls) by 2^60 along the rows, and a problem that is zero."""
    n, T, k = 300, 100, 5
    probs = [_problem(ng, 10 * i + 1, nf, n, T, k) for i, nf in enumerate((1, 2, 4, 8, 2))]
    for _, G, _, _ in probs:
        row = torch.cat([torch.full((j + 1,), float(j), device="cuda", dtype=torch.float64) for j in range(n + 1)])
        for t in (G.ret, G.les):
            t *= torch.exp2(grow * 0.2 * row)[:, None, None, None]
        G.tv *= torch.exp2(grow * 0.2 * torch.arange(n + 1, device="cuda").repeat_interleave(T + 1).double())[:, None, None, None]
    for t in probs[-1][1].tensors().values():
        t.zero_()
    ctx = ng.Context(k)
    b = ctx.batch(*[[p[q] for p in probs] for q in range(4)])
    (x, fx), (y, fy) = _both(ng, ctx, probs, n, lambda: b.step(n))
    assert fx == fy == 0
    _check(x[:-1], y[:-1])
    for q in x[-1]:
        assert torch.equal(x[-1][q], y[-1][q])


@pytest.mark.parametrize("where", ["ret", "les", "tv", "S"])
@pytest.mark.parametrize("value", [float("nan"), float("inf")])
def test_non_finite(ng, where, value):
    """A non-finite element spoils the items that read it and no others, and sets the status."""
    n, T, k = 300, 100, 5
    probs = [_problem(ng, 10 * i + 1, nf, n, T, k) for i, nf in enumerate((1, 2, 4, 8))]
    for g, G, S, _ in probs[1:]:
        at = {"ret": (G.ret, 100 * 101 // 2 + 30), "les": (G.les, 150 * 151 // 2 + 140), "tv": (G.tv, 130 * (T + 1) + 7),
              "S": (S.ret, n * (n + 1) // 2 + 60)}[where]
        at[0][at[1], 1, 0, 0] = value
    ctx = ng.Context(k)
    b = ctx.batch(*[[p[q] for p in probs] for q in range(4)])
    (x, fx), (y, fy) = _both(ng, ctx, probs, n, lambda: b.step(n))
    assert fx == fy == 1                      # the non-finite flag alone, both times
    for u, v in zip(x, y):
        for q in u:
            a, c = torch.isfinite(torch.view_as_real(u[q])).all(-1), torch.isfinite(torch.view_as_real(v[q])).all(-1)
            assert torch.equal(a, c)
            if a.any():
                assert ((u[q] - v[q])[a].abs().max() <= TOL * u[q][a].abs().max()).item()
