"""Latent sublayers whose GEMMs have few tiles (split along K inside clusters, 64- or 256-column
tiles) against the oracle: row counts around a tile, one K iteration per CTA and many, column
counts that end inside a tile, FFN and heads included, and the largest tile counts that split."""
import pytest

from gpu_helpers import PAIRS, SPLIT, Runner, assert_parity, oracle_layer
from paper_2606_07878_gb300 import synth

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


@pytest.mark.parametrize("H,d,D,n,F,t,other", [
    (1, 64, 256, 1, 64, 1, {}),        # one row, one tile, one K iteration a pass
    (1, 64, 256, 2, 192, 129, {}),     # FFN width that ends inside a tile, rows one past a tile
    (2, 128, 512, 1, 0, 63, {}),       # no FFN
    (1, 256, 512, 2, 448, 40, {}),     # head dim 256: output heads of 512 columns
    (3, 64, 256, 4, 1024, 300, {}),    # 8 row tiles: up to the count at which tiles stop splitting
    (5, 128, 256, 3, 320, 257, {"sa_scores": PAIRS}),  # 90 tiles of scores
    (1, 64, 512, 1, 0, 2304, {"sa_scores": PAIRS}),   # q / k projection: 72 tiles
    (1, 64, 512, 1, 0, 2433, {"sa_proj": PAIRS, "sa_scores": PAIRS}),  # 80 tiles
])
def test_small_latent_sublayers_match_oracle(H, d, D, n, F, t, other):
    wl = synth.tiny_workload(H=H, d=d, D=D, n=n, F=F, N=max(320, t), heavy=2, ts=(t,))
    r = Runner(wl, t)
    try:
        K, V = synth.gen_kv(wl, 0, device=DEV)
        Ck, Cv, _ = r.layer(0, K, V, t)
        classes = ["vo", "sa_proj", "sa_v", "sa_scores", "sa_pv", "sa_out", "heads"]
        for cls in classes + (["ffn1", "ffn2"] if F else []):
            form, width, ranks = r.gemm(cls)
            assert form == other.get(cls, SPLIT) and (form != SPLIT or ranks >= 2), cls
        Ck2, Cv2, _ = r.layer(0, K, V, t)
        assert (Ck == Ck2).all() and (Cv == Cv2).all()  # sums in a fixed order
        rk, rv, _, _ = oracle_layer(wl, r.W[0], K, V, t)
        for name, ref, got in (("C_k", rk, Ck), ("C_v", rv, Cv)):
            assert_parity(ref, synth.bf16_to_f64(got), name)
    finally:
        r.close()
