"""Biased decode attention (App. B, "Bias semantics in attention") at the edges of its kernel:
batches of 32 / 16 / 8 entries (d = 64 / 128 / 256) that end inside either part, row blocks of 4
and 8 query rows that are full or not, one slot (written directly) and several (merged)."""
import math

import numpy as np
import pytest
import torch

from oracle import still_oracle as O
from paper_2606_07878_gb300 import still

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


def _bf16(shape, seed):
    g = torch.Generator().manual_seed(seed)
    return torch.randn(shape, generator=g).to(torch.bfloat16).to(DEV)


@pytest.mark.parametrize("d,nq,Hq,H,t,S", [
    (64, 1, 1, 1, 1, 0), (64, 1, 5, 1, 33, 31), (64, 3, 6, 2, 0, 65),      # G = 1, 5, 9
    (128, 1, 8, 2, 16, 16), (128, 3, 12, 4, 17, 15), (128, 2, 32, 4, 129, 1000),  # G = 4, 9, 16
    (256, 1, 8, 1, 7, 9), (256, 1, 4, 2, 8, 0), (256, 8, 8, 1, 700, 333),  # G = 8, 2, 64
])
def test_decode_edges_match_oracle(d, nq, Hq, H, t, S):
    q = _bf16((nq, Hq, d), 1)
    Ck, Cv = _bf16((t, H, d), 2), _bf16((t, H, d), 3)
    Kf, Vf = _bf16((S, H, d), 4), _bf16((S, H, d), 5)
    beta = torch.randn((t, H), generator=torch.Generator().manual_seed(6)).to(DEV)
    out = torch.full((nq, Hq, d), float("nan"), dtype=torch.bfloat16, device=DEV)
    ctx = still.still_create(0)
    try:
        still.still_attend_biased(ctx, q, Ck, Cv, beta if t else None, Kf, Vf, out)
        torch.cuda.synchronize()
    finally:
        still.still_destroy(ctx)
    f = lambda x: x.double().cpu().numpy()
    ref = np.empty((nq, Hq, d))
    for i in range(Hq):
        h = i // (Hq // H)
        ref[:, i] = O.biased_attention(f(q)[:, i], f(Ck)[:, h], f(Cv)[:, h], f(beta)[:, h],
                                       f(Kf)[:, h], f(Vf)[:, h], 1 / math.sqrt(d))
    # bf16 output, 8 significant bits: rounding moves a value by at most 2^-8 of itself. The fp32
    # sums and exponentials before it stay below 2^-14 of the largest |V| (about 4).
    assert np.all(np.abs(f(out) - ref) <= 2.0 ** -8 * np.abs(ref) + 4 * 2.0 ** -14)


@pytest.mark.parametrize("d", [64, 128, 256])
def test_infinite_value_stays_in_its_dimension(d):
    """A short last batch repeats loads of the last entry: its infinite value must enter once."""
    t, S = 3, 5
    q, Ck, Cv = _bf16((1, 4, d), 1), _bf16((t, 1, d), 2), _bf16((t, 1, d), 3)
    Kf, Vf = _bf16((S, 1, d), 4), _bf16((S, 1, d), 5)
    Vf[S - 1, 0, 11] = float("inf")
    out = torch.empty((1, 4, d), dtype=torch.bfloat16, device=DEV)
    ctx = still.still_create(0)
    try:
        still.still_attend_biased(ctx, q, Ck, Cv, None, Kf, Vf, out)
        torch.cuda.synchronize()
    finally:
        still.still_destroy(ctx)
    inf = torch.zeros(d, dtype=torch.bool, device=DEV)
    inf[11] = True
    assert torch.all(torch.isposinf(out[..., inf])) and torch.all(torch.isfinite(out[..., ~inf]))
