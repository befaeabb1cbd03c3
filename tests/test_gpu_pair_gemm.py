"""Latent sublayers and folded key norms wide enough for the GEMM on CTA pairs (tiles of 256 x 160,
192 or 256) against the oracle: an odd number of row tiles, rows and columns that end inside a
tile, and several waves."""
import pytest

from gpu_helpers import PAIRS, SINGLE, Runner, assert_parity, oracle_layer
from paper_2606_07878_gb300 import synth

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


@pytest.mark.parametrize("H,d,D,n,F,t,pairs", [
    (2, 64, 512, 4, 4096, 641, ["ffn1"]),       # 11 row tiles (odd), FFN of 16 column tiles
    (1, 128, 256, 16, 2880, 700, ["sa_proj"]),  # rows that end inside a tile, 32 column tiles
    (4, 64, 256, 8, 3072, 520, ["sa_scores", "sa_pv", "ffn1"]),  # 32 batches
    (2, 64, 256, 4, 2880, 1300, ["ffn1"]),      # FFN width that ends inside a tile
])
def test_wide_latent_sublayers_match_oracle(H, d, D, n, F, t, pairs):
    wl = synth.tiny_workload(H=H, d=d, D=D, n=n, F=F, N=max(768, t), heavy=2, ts=(t,))
    r = Runner(wl, t)
    try:
        K, V = synth.gen_kv(wl, 0, device=DEV)
        Ck, Cv, _ = r.layer(0, K, V, t)
        for cls in pairs:
            assert r.gemm(cls) == (PAIRS, 256, 1), cls
        rk, rv, _, _ = oracle_layer(wl, r.W[0], K, V, t)
        for name, ref, got in (("C_k", rk, Ck), ("C_v", rv, Cv)):
            assert_parity(ref, synth.bf16_to_f64(got), name)
    finally:
        r.close()


@pytest.mark.parametrize("d,D,N,want", [
    (128, 512, 3001, (PAIRS, 160, 1)),   # 320 columns of key norms
    (64, 256, 3001, (SINGLE, 256, 1)),   # 192 columns, three waves
    (64, 256, 5501, (PAIRS, 192, 1)),    # five, an odd number of row tiles
])
def test_folded_key_norms_match_oracle(d, D, N, want):
    t = 48
    wl = synth.tiny_workload(H=4, d=d, D=D, n=4, F=0, N=N, heavy=2, ts=(t,))
    over = dict(compactor_rope=0)
    r = Runner(wl, t, cfg_over=over)
    try:
        K, V = synth.gen_kv(wl, 0, device=DEV)
        Ck, Cv, _ = r.layer(0, K, V, t)
        assert r.gemm("keyproj") == want
        rk, rv, _, _ = oracle_layer(wl, r.W[0], K, V, t, cfg_over=dict(compactor_rope=False))
        for name, ref, got in (("C_k", rk, Ck), ("C_v", rv, Cv)):
            assert_parity(ref, synth.bf16_to_f64(got), name)
    finally:
        r.close()
