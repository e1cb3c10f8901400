"""Steps whose digit-product workspace does not fit the device: the call takes the form it would take otherwise, gives its
result and leaves no message; the workspace is taken again by a later run for which there is room."""
import pytest
import torch

pytestmark = pytest.mark.gpu
TOL = 5e-12


def test_step_without_room():
    import paper_1911_01211_gb300 as ng
    ng.load_library()
    nk, n, T, k = 2048, 400, 100, 5     # the workspace takes about 240 MB
    g = ng.Grid(nt=n, ntau=T, nf=1, nbatch=nk, korder=k, h=0.02, beta=4.0, mu=0.1)
    G, S, eps = ng.Herm(g, zero=False), ng.Herm(g, ldk=1), ng.Func(g)
    gen = torch.Generator(device="cuda").manual_seed(1)
    for H, s in ((G, 0.3), (S, 0.1)):
        for t in H.tensors().values():
            torch.view_as_real(t).normal_(0.0, s, generator=gen)
    row = n * (n + 1) // 2
    ctx = ng.Context(k)
    ctx.set_bulk_split(ng.NG_BULK_THREAD)       # everything the FP64 kernels need is allocated here
    ctx.dyson_timestep(g, n, G, S, eps)
    ctx.set_bulk_split(ng.NG_BULK_AUTO)
    ctx.dyson_timestep(g, 2 * k + 1, G, S, eps)
    torch.cuda.synchronize()
    out = []
    free = torch.cuda.mem_get_info()[0]
    held = torch.empty(free - (160 << 20), dtype=torch.uint8, device="cuda")
    try:
        assert torch.cuda.mem_get_info()[0] < 200 << 20
        for _ in range(2):
            ctx.dyson_timestep(g, n, G, S, eps)
        assert ctx.status_sync() == (ng.NG_OK, 0)
        assert "allocation" not in ctx.lib.ng_last_error(ctx.h).decode()
        out.append([t[row:].clone() for t in (G.ret, G.les)])
        assert torch.cuda.mem_get_info()[0] < 200 << 20
    finally:
        del held
        torch.cuda.empty_cache()
    own = ng.Context(k)
    own.dyson_timestep(g, n, G, S, eps)          # with its workspace
    assert own.status_sync() == (ng.NG_OK, 0)
    for x, y in zip(out[0], (G.ret[row:], G.les[row:])):
        assert ((x - y).abs().amax((0, 1, 2)) <= TOL * x.abs().amax((0, 1, 2))).all()
    own.close()
    before = torch.cuda.mem_get_info()[0]
    ctx.dyson_timestep(g, n - 1, G, S, eps)      # an earlier step: asked again
    assert ctx.status_sync() == (ng.NG_OK, 0)
    assert before - torch.cuda.mem_get_info()[0] > 100 << 20
    ctx.close()
