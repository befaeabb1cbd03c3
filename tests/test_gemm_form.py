"""CPU checks of the rule that picks a GEMM's kernel form, tile width and CTAs per tile, on tables of
devices filled with given residency."""
import ctypes

import pytest

from paper_2606_07878_gb300 import still

SINGLE, PAIRS, SPLIT = 1, 2, 3
PLAIN, CHUNK_SUMS, HALF_SUMS, NORMS, HEADS, HEADS128 = range(6)
# clusters of 1 .. 8 CTAs that can be resident (index 0 unused)
GB300 = (152, [0, 0, 76, 46, 36, 28, 23, 15, 15])  # as cudaOccupancyMaxActiveClusters gives them
UNEVEN = (152, [0, 0, 75, 46, 36, 28, 23, 15, 15])  # GPCs that leave two single SMs over
SMALL = (40, [0, 0, 20, 13, 10, 8, 6, 5, 4])
NO_CLUSTERS = (152, [0] * 9)


def form(kind, M, N, batch, iters, device=GB300):
    sms, resident = device
    out = (ctypes.c_int32 * 3)()
    ok = still.lib().still_internal_gemm_form(kind, M, N, batch, iters, sms,
                                              (ctypes.c_int32 * 9)(*resident), out)
    assert ok, (kind, M, N)
    return tuple(out)


def tiles(M, N, batch, width):
    return -(-M // 128) * -(-N // width) * batch


@pytest.mark.parametrize("device", [GB300, SMALL, NO_CLUSTERS])
@pytest.mark.parametrize("kind", [PLAIN, CHUNK_SUMS, HALF_SUMS, NORMS, HEADS, HEADS128])
def test_forms_are_possible_ones(kind, device):
    sms, resident = device
    for M in (1, 128, 129, 641, 1280, 9728, 20000):
        for N in (32, 64, 192, 256, 320, 1024, 8192):
            for batch in (1, 5, 64):
                for iters in (1, 2, 3, 8, 24, 96):
                    f, width, ranks = form(kind, M, N, batch, iters, device)
                    at = (M, N, batch, iters, f, width, ranks)
                    if f == SPLIT:
                        n = tiles(M, N, batch, width)
                        assert 2 <= ranks <= min(8, iters), at
                        assert n <= resident[ranks] and n <= sms // 2, at  # all at once
                        assert kind != HALF_SUMS, at       # its sums need whole tiles in one CTA
                        assert width in {HEADS: (256,), HEADS128: (128,)}.get(kind, (64, 256)), at
                    else:
                        assert ranks == 1
                    if f == PAIRS:
                        assert kind in (PLAIN, HALF_SUMS, NORMS), at
                        assert width in ((160, 192) if kind == NORMS else (256,)), at
                    if f == SINGLE:
                        assert width == (128 if kind == HEADS128 else 256), at


@pytest.mark.parametrize("device,most", [(GB300, 76), (UNEVEN, 75), (SMALL, 20), (NO_CLUSTERS, 0)])
@pytest.mark.parametrize("kind", [PLAIN, CHUNK_SUMS, NORMS, HEADS])
def test_tiles_split_up_to_the_resident_pairs(kind, device, most):
    split = [m for m in range(1, 90) if form(kind, 128 * m, 256, 1, 16, device)[0] == SPLIT]
    assert split == list(range(1, most + 1))


@pytest.mark.parametrize("kind", [PLAIN, CHUNK_SUMS, NORMS, HEADS])
def test_column_tiles_and_batches_count_as_row_tiles(kind):
    assert form(kind, 128 * 25, 768, 1, 16)[0] == SPLIT
    assert form(kind, 128 * 25, 768 + 1, 1, 16)[0] != SPLIT
    assert form(kind, 128 * 5, 256, 15, 16)[0] == SPLIT
    assert form(kind, 128 * 5 + 1, 256, 15, 16)[0] != SPLIT
    # one K iteration cannot be split; two can
    assert form(kind, 128, 256, 1, 1)[0] != SPLIT
    assert form(kind, 128, 256, 1, 2)[2] == 2


def test_few_tiles_take_narrow_columns_and_more_ctas():
    assert form(PLAIN, 128, 256, 1, 8)[:2] == (SPLIT, 64)
    assert form(PLAIN, 256, 1024, 1, 32)[:2] == (SPLIT, 64)
    assert form(PLAIN, 1004, 1024, 1, 128) == (SPLIT, 256, 4)


def test_pairs_where_their_waves_are_shorter():
    # 4 x 1024 rows, d_l = 1024: 128 tiles on 152 SMs, or 64 pairs on 76 clusters of two
    assert form(PLAIN, 4096, 1024, 1, 32) == (PAIRS, 256, 1)
    # P v of t = 617, d_l = 2048: 5 m-tiles are 3 pairs, the last half empty
    assert form(PLAIN, 617, 2048, 128, 30)[0] == SINGLE
    # sums of squares per tile half do not split
    assert form(HALF_SUMS, 600, 256, 8, 8)[0] == PAIRS
    assert form(HEADS, 4096, 512, 4, 64)[0] == SINGLE  # no 2-SM form


def test_key_norms_take_the_faster_form():
    """The folded key norms of 4 KV-heads of 8 cross heads: the faster of the two measured forms at
    every measured token count (equal at 2,048 tokens of K_p = 192)."""
    for tokens in (896, 1024, 1152, 1280, 2688, 8192):
        assert form(NORMS, tokens, 320, 32, 15) == (PAIRS, 160, 1), tokens
    for tokens, want in [(1024, SINGLE), (2048, SINGLE), (2432, SINGLE), (4864, PAIRS), (8192, PAIRS)]:
        got = form(NORMS, tokens, 192, 32, 9)
        assert got == ((PAIRS, 192, 1) if want == PAIRS else (SINGLE, 256, 1)), (tokens, got)


@pytest.mark.parametrize("N,width", [(320, 160), (192, 192)])
def test_key_norm_tiles_hold_no_padding(N, width):
    for tokens in range(64, 20000, 97):
        for batch in (1, 4, 16, 64):
            f, w, _ = form(NORMS, tokens, N, batch, 3 * N // 64)
            assert f != PAIRS or w == width, (tokens, batch)
