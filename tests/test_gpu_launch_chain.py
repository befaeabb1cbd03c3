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
