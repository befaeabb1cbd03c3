"""Key projection (App. A, cross-attention keys) at the edges of its tiles, bands and position
tables, through a whole layer against the oracle: token counts around the 256-token tile pairs and
the 4096-token bands, cached positions whose segments start anywhere, step unevenly or lie on
fractions, and every head dimension."""
import numpy as np
import pytest

from gpu_helpers import Runner, assert_parity, oracle_layer
from paper_2606_07878_gb300 import synth

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


def _wl(d, D, N):
    return synth.tiny_workload(d=d, D=D, N=N, heavy=2, ts=(24,))


@pytest.mark.parametrize("d,D,segments", [
    (64, 256, [(0, 1, 255)]), (64, 256, [(0, 1, 257)]), (128, 512, [(3, 1, 4097)]),
    (256, 512, [(0, 1, 513)]),
    # previous compact slots on fractions, then new tokens that meet no multiple of 32
    (128, 256, [(0, 37.25, 21), (783, 1, 300)]),
    # a short leading segment, a wide step, then a longer run on half positions
    (64, 512, [(5, 1, 33), (100, 2, 50), (1000.5, 1, 200)]),
    # a backward segment and one position repeated
    (64, 256, [(90, -1, 70), (200, 0, 5), (300, 1, 65)]),
])
def test_layer_matches_oracle_at_key_edges(d, D, segments):
    N = sum(c for _, _, c in segments)
    wl = _wl(d, D, N)
    t = 24
    pos = synth.positions_from_segments(segments)
    r = Runner(wl, t)
    try:
        K, V = synth.gen_kv(wl, 0, device=DEV, positions=pos)
        Ck, Cv, _ = r.layer(0, K, V, t, segments)
        rk, rv, _, _ = oracle_layer(wl, r.W[0], K, V, t, kpos=pos.numpy())
        for name, ref, got in (("C_k", rk, Ck), ("C_v", rv, Cv)):
            assert_parity(ref, synth.bf16_to_f64(got), name)
    finally:
        r.close()
