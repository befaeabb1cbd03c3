"""The strip kernel's shares of KV-heads and its loads: token counts that end inside a tile, head
counts that do not divide into the shares, caches long enough for one share, rows that start off
a 16-byte boundary (element-wise loads) and value rows of more than one thread's items."""
import pytest
import torch

from gpu_helpers import Runner, assert_parity, oracle_layer
from paper_2606_07878_gb300 import still, synth

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


@pytest.mark.parametrize("H,d,N,rope", [
    (3, 64, 33, 1), (8, 128, 1000, 1), (3, 256, 2100, 1), (5, 64, 4999, 0), (2, 128, 10007, 1),
])
def test_strip_shares_and_unaligned_rows(H, d, N, rope):
    t = 16
    wl = synth.tiny_workload(H=H, d=d, D=512, n=1, F=0, N=N, heavy=2, ts=(t,))
    over = dict(compactor_rope=rope)
    r = Runner(wl, t, cfg_over=over)
    try:
        K, V = synth.gen_kv(wl, 0, device=DEV)
        Ck, Cv, _ = r.layer(0, K, V, t)
        rk, rv, _, _ = oracle_layer(wl, r.W[0], K, V, t, cfg_over=over)
        for name, ref, got in (("C_k", rk, Ck), ("C_v", rv, Cv)):
            assert_parity(ref, synth.bf16_to_f64(got), name)
        shifted = []
        for x in (K, V):  # the same rows, one element past a 16-byte boundary, odd row pitch
            buf = torch.zeros(N * (H * d + 3) + 1, dtype=x.dtype, device=DEV)
            view = buf[1:].view(N, H * d + 3)[:, : H * d].view(N, H, d)
            view.copy_(x)
            shifted.append(view)
        C2k, C2v = r.out(t)
        still.still_compact_layer(r.ctx, 0, shifted[0], shifted[1], t, C2k, C2v)
        r.check_status()
        assert torch.equal(C2k, Ck) and torch.equal(C2v, Cv)
    finally:
        r.close()
