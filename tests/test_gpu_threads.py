"""Two contexts in two host threads, each on a stream of its own, with problems whose kernels need different amounts of
shared memory (transforms of other lengths, LU panels of other sizes), called at the same time: every call succeeds
and gives what it gives alone."""
import threading

import pytest
import torch

pytestmark = pytest.mark.gpu


def _steps(ng, nk, n, T, nf, shared, reps, out, errors, meet=lambda: None):
    try:
        k = 5
        stream = torch.cuda.Stream()
        with torch.cuda.stream(stream):
            g = ng.Grid(nt=n, ntau=T, nf=nf, nbatch=nk, korder=k, h=0.02, beta=4.0, mu=0.1)
            gen = torch.Generator(device="cuda").manual_seed(nk)
            G, S, eps = ng.Herm(g), ng.Herm(g, ldk=1 if shared else None), ng.Func(g)
            for H, s in ((G, 0.3), (S, 0.1)):
                for t in H.tensors().values():
                    torch.view_as_real(t).normal_(0.0, s, generator=gen)
            ctx = ng.Context(k)
            ctx.set_bulk_split(ng.NG_BULK_THREAD)     # the source by FFT at every size
            for i in range(reps):
                meet()
                ctx.dyson_timestep(g, n, G, S, eps)
                if i % 100 == 0:
                    meet()
                    ctx.dyson_mat(g, G, S, eps)
            stream.synchronize()
            out.append([G.mat.clone(), G.tv[n * (T + 1):].clone()])
            ctx.close()
    except BaseException as e:          # noqa: BLE001 - reported by the main thread
        errors.append(e)
        meet()


def test_two_threads():
    import paper_1911_01211_gb300 as ng
    ng.load_library()
    cases = [(40, 12, 900, 1, True), (44, 12, 300, 1, True)]
    reps = 3000
    alone, errors = [], []
    for c in cases:
        _steps(ng, *c, reps, alone, errors)
    assert not errors, errors
    both = [[], []]
    barrier = threading.Barrier(2)

    def meet():
        if not errors:
            try:
                barrier.wait(60)
            except threading.BrokenBarrierError:
                pass

    threads = [threading.Thread(target=_steps, args=(ng, *c, reps, both[i], errors, meet)) for i, c in enumerate(cases)]
    for t in threads:
        t.start()
    for t in threads:
        t.join(300)
    assert not errors, errors
    for x, y in zip(alone, both):
        for a, b in zip(x, y[0]):
            assert torch.equal(a, b)
