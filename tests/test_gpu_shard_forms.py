"""ng_run_2b_sharded where the batch of a rank and the batch of one GPU would take other forms of a step on their own
(chunks of the boundary's sums, lanes or a warp per item, digit products from some step on, the kept inverse
or the LU of the set-up): G_k of every rank, Gloc and Sigma bitwise those of one ng_run_2b.  The ranks are host threads
(ThreadExchange), no kernel waits on another."""
import threading

import numpy as np
import pytest
import torch

from paper_1911_01211_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nk,nranks,nt,ntau,precision", [
    (250, 4, 24, 200, 0),   # digit products from n = 18 for all 250, later or not at all for 58 or 64; 38 chunks against 48
    (33, 2, 20, 30, 0),     # lanes per item against a warp per item; a rank of one k-point
    (97, 3, 18, 100, 1),    # FP32 copies: two problems a thread for 32 but not for 97
    (129, 5, 80, 300, 0),   # digit products from n = 75 on, on a rank of one k-point too
])
def test_ranks_equal_one_gpu(nk, nranks, nt, ntau, precision):
    import paper_1911_01211_gb300 as ng
    from paper_1911_01211_gb300.shard import ThreadExchange
    ng.load_library()
    w = wl.chain_kspace(nk=nk, nt=nt, ntau=ntau, beta=4.0, h=0.05)
    group = ThreadExchange.Group(nranks, timeout=300.0)
    out, errors = {}, []

    def run(r):
        b, c = (0, nk) if r is None else ng.shard_plan(nk, r, nranks, ng.Grid(nt=nt, ntau=ntau, nf=1, nbatch=nk, korder=w.korder,
                                                                              h=w.h, beta=w.beta))[:2]
        g = ng.Grid(nt=nt, ntau=ntau, nf=1, nbatch=c, korder=w.korder, h=w.h, beta=w.beta)
        ctx = ng.Context(w.korder)
        G, L, S = ng.Herm(g), ng.Herm(g, ldk=1), ng.Herm(g, ldk=1)
        e0 = ng.Func(g, values=torch.from_numpy(np.ascontiguousarray(w.eps0[..., b:b + c])))
        mf, U = ng.Func(g), ng.Func(g, scalar=True)
        U.val[:, 0, 0, 0] = torch.from_numpy(w.U.astype(complex))
        if r is None:
            its = ctx.run_2b(g, G, L, S, e0, mf, U, corrector=w.corrector, precision=precision)
        else:
            its = ctx.run_2b_sharded(g, G, L, S, e0, mf, U, ThreadExchange(group, nk, r, g), corrector=w.corrector,
                                     precision=precision)
        torch.cuda.synchronize()
        out[r] = (b, c, G, L, S, its)
        ctx.close()

    def rank_main(r):
        try:
            run(r)
        except BaseException as e:          # noqa: BLE001 - reported by the main thread
            errors.append(e)
            group.barrier.abort()

    run(None)
    threads = [threading.Thread(target=rank_main, args=(r,)) for r in range(nranks)]
    for t in threads:
        t.start()
    for t in threads:
        t.join(600)
    assert not errors, errors
    _, _, G, L, S, its = out.pop(None)
    for b, c, Gr, Lr, Sr, it in out.values():
        assert it == its
        for name in ("mat", "ret", "les", "tv"):
            assert torch.equal(getattr(Gr, name), getattr(G, name)[..., b:b + c]), name
            assert torch.equal(getattr(Lr, name), getattr(L, name)), name
            assert torch.equal(getattr(Sr, name), getattr(S, name)), name
