"""One-pass scores at head dim 256 whose rows keep few, many or too many heavy keys, so that the
CTAs of the repair hold lists of every length and rows that are recomputed beside rows that are
not: row counts that end inside a CTA, several key splits, and one query row."""
import pytest

from gpu_helpers import Runner, assert_parity, oracle_layer
from paper_2606_07878_gb300 import still, synth

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


@pytest.mark.parametrize("D,n,H,t,N,logit_scale", [
    (512, 1, 1, 1, 700, 64.0),
    (512, 2, 2, 101, 2900, 16.0),
    (768, 1, 3, 45, 1500, 48.0),
    (2048, 1, 1, 130, 2100, 96.0),
])
def test_repair_matches_oracle(D, n, H, t, N, logit_scale):
    wl = synth.tiny_workload(d=256, D=D, n=n, F=512, H=H, N=N, heavy=2, ts=(t,))
    r = Runner(wl, t, cfg_over=dict(logit_scale=logit_scale))
    try:
        K, V = synth.gen_kv(wl, 0, device=DEV)
        still.still_profile_enable(r.ctx, True)
        still.still_profile_enable_classes(r.ctx, [])
        Ck, Cv, _ = r.layer(0, K, V, t)
        assert still.still_profile_read(r.ctx)["repair"][0] > 0
        still.still_profile_enable(r.ctx, False)
        Ck2, Cv2, _ = r.layer(0, K, V, t)
        assert (Ck == Ck2).all() and (Cv == Cv2).all()
        rk, rv, _, _ = oracle_layer(wl, r.W[0], K, V, t, cfg_over=dict(logit_scale=logit_scale))
        for name, ref, got in (("C_k", rk, Ck), ("C_v", rv, Cv)):
            assert_parity(ref, synth.bf16_to_f64(got), name)
    finally:
        r.close()
