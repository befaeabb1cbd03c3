"""A compaction captured into a graph as the first call, or after one of another size: the captured
call takes GEMM forms and key-projection variants that no call has taken before, so each case runs
in a process of its own. The replay gives the bits of an eager call that follows."""
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

CODE = """
import sys
sys.path[:0] = [{root!r}, {tests!r}]
import torch
from gpu_helpers import Runner
from paper_2606_07878_gb300 import still, synth

(H, d, D, n, F, blocks, rope), first, size = {shape}, {first}, {size}
wl = synth.tiny_workload(H=H, d=d, D=D, n=n, F=F, N=max(x[0] for x in (first, size) if x), heavy=2,
                         ts=(size[1],), n_blocks=blocks)
t_max = max(x[1] for x in (first, size) if x)
r = Runner(wl, t_max, cfg_over=dict(compactor_rope=rope))
seg = lambda N: [(0, 1, N // 2), (N // 2 + 0.5, 1, N - N // 2)]
def call(N, t, segments, stream=None):
    K, V = synth.gen_kv(wl, 0, N=N, device="cuda:0", positions=synth.positions_from_segments(segments))
    Ck, Cv = r.out(t)
    go = lambda s=None: still.still_compact_layer(r.ctx, 0, K, V, t, Ck, Cv, segments, stream=s)
    return go, Ck, Cv
still.still_reserve_workspace(r.ctx, wl["N"] + 64, t_max)
if first:
    go, _, _ = call(*first, [(0, 1, first[0])])
    go()
    r.check_status()
go, Ck, Cv = call(*size, seg(size[0]))
torch.cuda.synchronize()
graph, s = torch.cuda.CUDAGraph(), torch.cuda.Stream()
with torch.cuda.graph(graph, stream=s):
    go(s)
for _ in range(2):
    Ck.zero_()
    Cv.zero_()
    graph.replay()
    torch.cuda.synchronize()
    r.check_status()
got = Ck.clone(), Cv.clone()
assert torch.isfinite(got[0].float()).all() and got[0].any() and got[1].any()
go()
r.check_status()
assert torch.equal(got[0], Ck) and torch.equal(got[1], Cv)
print("captured")
"""


@pytest.mark.parametrize("shape,first,size", [
    ((2, 64, 256, 4, 1024, 1, 1), (300, 9), (3000, 700)),   # split forms first, pairs captured
    ((2, 64, 256, 4, 1024, 1, 1), (3000, 700), (300, 9)),
    ((2, 64, 256, 4, 1024, 1, 1), None, (1000, 100)),
    ((2, 128, 512, 2, 0, 2, 1), (200, 5), (2500, 300)),     # two blocks
    ((4, 128, 512, 4, 256, 1, 0), (200, 5), (3001, 64)),    # folded key norms
    ((1, 256, 512, 2, 512, 1, 1), (200, 5), (2100, 400)),   # head dim 256
])
def test_capture_after_a_call_of_another_size(shape, first, size):
    import os
    tests = os.path.dirname(os.path.abspath(__file__))
    code = CODE.format(root=os.path.dirname(tests), tests=tests, shape=shape, first=first, size=size)
    p = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, timeout=300)
    assert p.returncode == 0 and "captured" in p.stdout, p.stderr[-3000:]
