"""Time steps whose history sums run as digit products on the tensor cores (nf = 1, at least 8
problems, enough work), and steps with several lanes per item below that, against the FP64 kernels of the same library (NG_BULK_THREAD, themselves
pinned to the oracle): edges of the 128 x 128 units and 16 x 16 tiles, ragged problem groups, every
quadrature order, shared and per-problem row functions, scale growth inside a unit, zeros and
non-finite values.

Tolerance: each sum has at most n + ntau + 1 <= 1000 terms, the FP64 kernels round each addition to
2^-53 of a partial sum below sum |terms|; for the random data here sum |terms| is below 40 times the
largest result, so the two differ by at most 1000 * 40 * 2^-53 = 5e-12 of the largest element."""
import pytest
import torch

pytestmark = pytest.mark.gpu
TOL = 5e-12


@pytest.fixture(scope="module")
def ng():
    import paper_1911_01211_gb300 as ng
    ng.load_library()
    return ng


def _random(H, seed, scale):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    for t in H.tensors().values():
        torch.view_as_real(t).normal_(0.0, scale, generator=gen)


def _slice(G, g, n):
    T1 = g.ntau + 1
    lo, hi = n * (n + 1) // 2, (n + 1) * (n + 2) // 2
    return {"ret": G.ret[lo:hi], "les": G.les[lo:hi], "tv": G.tv[n * T1:(n + 1) * T1]}


def _both(ng, ctx, g, n, G, call):
    """The slice by the FP64 kernels and by the digit products, and their device status."""
    out = []
    for mode in (ng.NG_BULK_THREAD, ng.NG_BULK_AUTO):
        ctx.set_bulk_split(mode)
        for v in _slice(G, g, n).values():
            v.zero_()
        call()
        flags = ctx.status_sync()[1]
        out.append(({k: v.clone() for k, v in _slice(G, g, n).items()}, flags))
    return out


def _check(a, b):
    for k in a:
        x, y = a[k][:, 0, 0], b[k][:, 0, 0]
        # per problem: the scale of one must not hide another's error
        err = ((x - y).abs().amax(0) / x.abs().amax(0)).max().item()
        assert err < TOL, (k, err)


DYSON = [  # nk, n, ntau, k, shared
    (29, 384, 300, 5, True), (129, 129, 640, 4, True), (264, 13, 400, 5, True), (130, 128, 127, 3, False),
    (36, 400, 127, 2, False), (17, 600, 129, 1, True), (131, 144, 383, 5, False), (8, 770, 639, 5, True),
    # below the line: eight or four lanes per item, the boundary with one lane per problem (16 problems and
    # more); direct left-mixing source, then by FFT
    (16, 11, 12, 5, True), (33, 12, 25, 4, False), (47, 30, 16, 1, True), (31, 64, 40, 3, True), (70, 40, 100, 5, True),
    (300, 60, 30, 2, False), (129, 20, 300, 4, False), (20, 90, 600, 5, True),
]


@pytest.mark.parametrize("nk,n,T,k,shared", DYSON)
def test_dyson_step(ng, nk, n, T, k, shared):
    g = ng.Grid(nt=max(n, 2 * k + 2), ntau=T, nf=1, nbatch=nk, korder=k, h=0.02, beta=4.0, mu=0.1)
    G, S, eps = ng.Herm(g), ng.Herm(g, ldk=1 if shared else None), ng.Func(g)
    _random(G, 1, 0.3)
    _random(S, 2, 0.1)
    torch.view_as_real(eps.val)[..., 0].normal_()
    ctx = ng.Context(k)
    (a, fa), (b, fb) = _both(ng, ctx, g, n, G, lambda: ctx.dyson_timestep(g, n, G, S, eps))
    assert fa == fb == 0
    _check(a, b)


@pytest.mark.parametrize("nk,n,T,k,fs,ccs,sig", [(33, 384, 300, 5, False, False, 1), (65, 331, 90, 3, True, False, -1),
                                                 (31, 470, 33, 4, False, True, 1), (200, 20, 375, 5, True, True, 1)])
def test_vie2_step(ng, nk, n, T, k, fs, ccs, sig):
    g = ng.Grid(nt=n, ntau=T, nf=1, nbatch=nk, korder=k, h=0.02, beta=4.0, sig=sig)
    G, F, Fcc, Q = ng.Herm(g), ng.Herm(g, ldk=1 if fs else None), ng.Herm(g, ldk=1 if ccs else None), ng.Herm(g)
    for i, x in enumerate((G, F, Fcc, Q)):
        _random(x, 10 + i, 0.2)
    ctx = ng.Context(k)
    (a, fa), (b, fb) = _both(ng, ctx, g, n, G, lambda: ctx.vie2_timestep(g, n, G, F, Fcc, Q))
    assert fa == fb == 0
    _check(a, b)


@pytest.mark.parametrize("grow", [1.0, -1.0])
def test_scale_growth_and_zeros(ng, grow):
    """History that grows (or falls) by 2^60 along the rows, problems of very different size, and
    problems that are zero."""
    nk, n, T, k = 60, 300, 100, 5
    g = ng.Grid(nt=n, ntau=T, nf=1, nbatch=nk, korder=k, h=0.02, beta=4.0)
    G, S, eps = ng.Herm(g), ng.Herm(g, ldk=1), ng.Func(g)
    _random(G, 3, 0.3)
    _random(S, 4, 0.1)
    for t in (G.ret, G.les):
        row = torch.cat([torch.full((j + 1,), float(j), device="cuda", dtype=torch.float64) for j in range(n + 1)])
        t *= torch.exp2(grow * 0.3 * row)[:, None, None, None]
    G.tv *= torch.exp2(grow * 0.3 * torch.arange(n + 1, device="cuda").repeat_interleave(T + 1).double())[:, None, None, None]
    for t in G.tensors().values():
        t *= torch.exp2(10.0 * torch.arange(nk, device="cuda").double() - 300.0)
        t[..., 5] = 0
    ctx = ng.Context(k)
    (a, _), (b, _) = _both(ng, ctx, g, n, G, lambda: ctx.dyson_timestep(g, n, G, S, eps))
    for q in a:
        x, y = a[q][:, 0, 0], b[q][:, 0, 0]
        big = x.abs().amax(0)
        assert torch.isfinite(torch.view_as_real(y)).all()
        err = ((x - y).abs().amax(0) / torch.where(big > 0, big, torch.ones_like(big))).max().item()
        assert err < TOL, (q, err)


@pytest.mark.parametrize("where", ["ret", "les", "tv", "S"])
@pytest.mark.parametrize("value", [float("nan"), float("inf")])
def test_non_finite(ng, where, value):
    """A non-finite element spoils the items that read it and no others, and sets the status."""
    nk, n, T, k = 61, 300, 100, 5
    g = ng.Grid(nt=n, ntau=T, nf=1, nbatch=nk, korder=k, h=0.02, beta=4.0)
    G, S, eps = ng.Herm(g), ng.Herm(g), ng.Func(g)
    _random(G, 5, 0.3)
    _random(S, 6, 0.1)
    at = {"ret": (G.ret, 100 * 101 // 2 + 30), "les": (G.les, 150 * 151 // 2 + 140), "tv": (G.tv, 130 * (T + 1) + 7),
          "S": (S.ret, n * (n + 1) // 2 + 60)}[where]
    at[0][at[1], 0, 0, 3] = value
    ctx = ng.Context(k)
    (a, fa), (b, fb) = _both(ng, ctx, g, n, G, lambda: ctx.dyson_timestep(g, n, G, S, eps))
    assert fa == fb == 1                      # the non-finite flag alone, both times
    for q in a:
        x, y = a[q][:, 0, 0], b[q][:, 0, 0]
        fx, fy = torch.isfinite(torch.view_as_real(x)).all(-1), torch.isfinite(torch.view_as_real(y)).all(-1)
        assert torch.equal(fx, fy)
        d = torch.where(fx, (x - y).abs(), torch.zeros_like(x.abs()))
        s = torch.where(fx, x.abs(), torch.zeros_like(x.abs())).amax(0)
        # a problem without any finite element has nothing to compare
        assert (d.amax(0) <= TOL * torch.where(s > 0, s, torch.ones_like(s))).all()


@pytest.mark.parametrize("nk,shared", [(3, True), (64, True), (65, False)])
@pytest.mark.parametrize("T,k", [(4, 1), (12, 5), (13, 5), (24, 5), (25, 4), (40, 5), (127, 3)])
def test_fft_source_edges(ng, nk, shared, T, k):
    """The left-mixing row with its Matsubara source by FFT against the direct sums, where most or all
    columns lie next to an end of the tau axis; with the self-energy's spectra shared and not."""
    n = 2 * k + 3
    g = ng.Grid(nt=n, ntau=T, nf=1, nbatch=nk, korder=k, h=0.02, beta=4.0, mu=0.1)
    G, S, eps = ng.Herm(g), ng.Herm(g, ldk=1 if shared else None), ng.Func(g)
    _random(G, 7, 0.3)
    _random(S, 8, 1.0)
    ctx = ng.Context(k)
    ctx.set_bulk_split(ng.NG_BULK_THREAD)
    out = []
    for src in (ng.NG_TVSRC_DIRECT, ng.NG_TVSRC_AUTO):
        ctx.set_tv_source(src)
        ctx.dyson_timestep(g, n, G, S, eps)
        out.append({q: v.clone() for q, v in _slice(G, g, n).items()})
    _check(*out)


@pytest.mark.parametrize("nf,nk,n,T,k", [(2, 1, 40, 25, 5), (2, 3, 12, 33, 5), (2, 2, 97, 12, 4), (1, 1, 64, 40, 3), (1, 5, 33, 31, 5),
                                         (2, 1, 11, 12, 5)])
def test_warp_items(ng, nf, nk, n, T, k):
    """A warp per item, two per lesser item (one or a few problems, an odd and an even number of start-up
    warps before them, the first step inside the history), against a thread per item."""
    g = ng.Grid(nt=max(n, 2 * k + 2), ntau=T, nf=nf, nbatch=nk, korder=k, h=0.02, beta=4.0, mu=0.1)
    G, S, eps = ng.Herm(g), ng.Herm(g), ng.Func(g)
    _random(G, 1, 0.3)
    _random(S, 2, 0.1)
    torch.view_as_real(eps.val)[..., 0].normal_()
    ctx = ng.Context(k)
    out = []
    for mode in (ng.NG_BULK_THREAD, ng.NG_BULK_WARP):
        ctx.set_bulk_split(mode)
        for v in _slice(G, g, n).values():
            v.zero_()
        ctx.dyson_timestep(g, n, G, S, eps)
        assert ctx.status_sync()[1] == 0
        out.append({q: v.clone() for q, v in _slice(G, g, n).items()})
    for q in out[0]:
        x, y = out[0][q], out[1][q]
        assert ((x - y).abs().amax((0, 1, 2)) <= TOL * x.abs().amax((0, 1, 2))).all(), q
