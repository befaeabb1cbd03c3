"""Calls whose kernels begin under the tail of the one before, between work of the caller on the
same stream that writes the inputs just before the call and overwrites them, and the outputs, just
behind it: issued eagerly and replayed from a graph captured on a stream forked from another."""
import pytest
import torch

from gpu_helpers import Runner
from paper_2606_07878_gb300 import still, synth

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


@pytest.mark.parametrize("H,d,D,t,N", [(2, 64, 512, 40, 700), (2, 256, 512, 130, 2048)])
def test_calls_order_with_the_callers_work(H, d, D, t, N):
    wl = synth.tiny_workload(H=H, d=d, D=D, n=2, F=256, N=N, heavy=2, ts=(t,))
    r = Runner(wl, t)
    try:
        ins = [synth.gen_kv(wl, 0, device=DEV, seed=i) for i in range(3)]
        want = [tuple(x.clone() for x in r.layer(0, K, V, t)[:2]) for K, V in ins]
        still.still_reserve_workspace(r.ctx, N, t)
        K, V = (torch.empty_like(x) for x in ins[0])
        Ck, Cv = r.out(t)
        got = [tuple(torch.empty_like(x) for x in w) for w in want]

        def calls(s):
            for (k, v), g in zip(ins, got):
                K.copy_(k)
                V.copy_(v)
                still.still_compact_layer(r.ctx, 0, K, V, t, Ck, Cv, stream=s)
                g[0].copy_(Ck)
                g[1].copy_(Cv)
                for x in (K, V, Ck, Cv):
                    x.fill_(float("nan"))

        def check():
            torch.cuda.synchronize()
            r.check_status()
            for w, g in zip(want, got):
                assert torch.equal(w[0], g[0]) and torch.equal(w[1], g[1])
                g[0].zero_()
                g[1].zero_()

        torch.cuda.synchronize()
        s = torch.cuda.Stream()
        with torch.cuda.stream(s):
            for _ in range(4):
                calls(s)
        check()
        other = torch.cuda.Stream()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=s):
            other.wait_stream(s)
            with torch.cuda.stream(other):
                calls(other)
            s.wait_stream(other)
        for _ in range(2):
            graph.replay()
            check()
    finally:
        r.close()


def _order(status, sets, bufs, outs, call):
    """call(stream) reads bufs and writes outs: on each set of inputs, written just before it and
    overwritten just behind it, it gives what it gives on an idle device, eager and replayed."""
    want = []
    for xs in sets:
        for b, x in zip(bufs, xs):
            b.copy_(x)
        torch.cuda.synchronize()
        call(None)
        torch.cuda.synchronize()
        status()
        want.append([o.clone() for o in outs])
    got = [[torch.zeros_like(o) for o in w] for w in want]

    def calls(s):
        for xs, g in zip(sets, got):
            for b, x in zip(bufs, xs):
                b.copy_(x)
            call(s)
            for a, o in zip(g, outs):
                a.copy_(o)
            for x in (*bufs, *outs):
                x.fill_(float("nan"))

    def check():
        torch.cuda.synchronize()
        status()
        for w, g in zip(want, got):
            for a, b in zip(w, g):
                assert torch.isfinite(a.float()).all() and torch.equal(a, b)
                b.zero_()

    s, other = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(s):
        for _ in range(4):
            calls(s)
    check()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=s):
        other.wait_stream(s)
        with torch.cuda.stream(other):
            calls(other)
        s.wait_stream(other)
    for _ in range(2):
        graph.replay()
        check()


@pytest.mark.parametrize("call", ["two_block", "beta", "folded", "ragged", "recompact"])
def test_every_sequence_orders_with_the_callers_work(call):
    H, d, D, n = 2, 64, 256, 2
    lens, ts = [700, 333, 90], [40, 60, 9]
    wl = synth.tiny_workload(H=H, d=d, D=D, n=n, F=0 if call == "two_block" else 256, N=700,
                             heavy=2, ts=(60,), n_blocks=2 if call == "two_block" else 1)
    r = Runner(wl, 60, cfg_over=dict(compactor_rope=0) if call == "folded" else None)
    try:
        still.still_reserve_workspace(r.ctx, 2000, 60)
        new = lambda rows: torch.empty((rows, H, d), dtype=torch.bfloat16, device=DEV)  # noqa: E731
        gen = lambda n, i: synth.gen_kv(wl, 0, N=n, device=DEV, seed=i)  # noqa: E731
        if call in ("ragged", "recompact"):
            total = sum(lens)
            cu = [0, 700, 1033, 1123]
            if call == "ragged":
                sets = [gen(total, i) for i in range(3)]
                bufs, outs = [new(total), new(total)], [new(sum(ts)), new(sum(ts))]
                go = lambda s: still.still_compact_layer_ragged(  # noqa: E731
                    r.ctx, 0, *bufs, cu, ts, *outs, stream=s)
            else:
                prev = [30, 20, 5]
                sets = [gen(sum(prev), i) + gen(total, 9 + i) for i in range(3)]
                bufs = [new(sum(prev)), new(sum(prev)), new(total), new(total)]
                length = [1000, 640, 160]
                rows = sum(still.still_budget(a + b, 32) for a, b in zip(length, lens))
                outs = [new(rows), new(rows)]
                go = lambda s: still.still_recompact_layer_ragged(  # noqa: E731
                    r.ctx, 0, *bufs[:2], [0, 30, 50, 55], length, *bufs[2:], cu, 32, *outs, stream=s)
        else:
            sets = [gen(700, i) for i in range(3)]
            bufs, outs = [new(700), new(700)], [new(60), new(60)]
            if call == "beta":
                w = torch.randn(D, generator=torch.Generator().manual_seed(1)) * 0.02
                still.still_set_beta_head(r.ctx, 0, w.to(torch.bfloat16).to(DEV), beta_max=4.0,
                                          mass_match=1)
                torch.cuda.synchronize()
                outs.append(torch.empty((60, H), device=DEV))
                go = lambda s: still.still_compact_layer_beta(  # noqa: E731
                    r.ctx, 0, *bufs, 60, *outs, stream=s)
            else:
                go = lambda s: still.still_compact_layer(r.ctx, 0, *bufs, 60, *outs,  # noqa: E731
                                                         stream=s)
        _order(r.check_status, sets, bufs, outs, go)
    finally:
        r.close()


@pytest.mark.parametrize("t,S", [(40, 20), (700, 1500)])  # one slot written directly, and the merge
def test_decode_orders_with_the_callers_work(t, S):
    L, nq, Hq, H, d = 3, 1, 8, 2, 128
    g = torch.Generator().manual_seed(5)
    rand = lambda *s: torch.randn(s, generator=g).to(torch.bfloat16).to(DEV)  # noqa: E731
    shapes = [(nq, Hq, d), (t, H, d), (t, H, d), (S, H, d), (S, H, d)] * L
    sets = [[rand(*s) for s in shapes] for _ in range(3)]
    bufs = [torch.empty_like(x) for x in sets[0]]
    outs = [torch.empty((nq, Hq, d), dtype=torch.bfloat16, device=DEV) for _ in range(L)]
    ctx = still.still_create(0)
    try:
        def go(s):
            q, Ck, Cv, Kf, Vf = ([bufs[5 * l + i] for l in range(L)] for i in range(5))
            still.still_attend_biased_stack(ctx, q, Ck, Cv, None, Kf, Vf, outs, stream=s)

        _order(lambda: None, sets, bufs, outs, go)
    finally:
        still.still_destroy(ctx)
