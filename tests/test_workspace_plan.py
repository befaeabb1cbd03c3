"""CPU checks of the workspace plan: what a call takes, what a reservation takes, and that a call
fits every limit that holds its buffers with one sum-of-squares partial per 128 columns."""
import ctypes

import pytest

from paper_2606_07878_gb300 import still

MIB = 1 << 20
OUT = ctypes.c_int64 * 5


@pytest.fixture(scope="module")
def lib():
    L = still.lib()
    L.still_internal_reserve.restype = ctypes.c_size_t
    return L


def _cfg(H, d, D, n, F, t_max):
    return still.make_config(H, d, D, n, F, t_max, 1e6)


SPLIT = 76  # tiles that the device splits


def plan(lib, cfg, N, t, limit, split=SPLIT):
    """(bytes, pairs per cross-attention group, KV-heads and self heads per self-attention group,
    partials per vector), or None when the limit is too small."""
    out = OUT()
    ok = lib.still_internal_plan(ctypes.byref(cfg), split, 0, 0, ctypes.c_int64(N), t,
                                 ctypes.c_double(0), ctypes.c_double(N - 1),
                                 ctypes.c_size_t(limit), out)
    return tuple(out) if ok else None


def _a256(x):
    return (x + 255) // 256 * 256


def smallest_need(H, d, D, n, F, N, t):
    """Bytes of a call's buffers (one block, queries precomputed, compactor RoPE) in its smallest
    groups: one (h, i) pair, and one KV-head with one self head at a time."""
    up = lambda x, a: (x + a - 1) // a * a  # noqa: E731
    Np, tp, ldt, G = up(N, 64), up(t, 64), up(t, 4), (N - 1) // 32 + 2
    fixed = sum(map(_a256, [
        H * N * 3 * d * 2, H * 2 * d * 2 * Np * 2, (G + 32) * D * 4, D // 2 * 4, Np * 8,
        t * d // 2 * 8, H * t * 2 * n * 2 * d * 2, H * t * D * 4, H * t * 2 * D * 2,
        H * t * n * D * 4, H * t * D * 4, H * t * D * 4, H * t * max(F, 1) * 4, H * t * D * 4]))
    splits, cand = 16, 0
    if d == 256 and 512 <= D <= 2048:  # one-pass scores: candidate keys and logits
        cand = 2 * _a256(t * 32 * 4) * splits
    pair = (_a256(N * 4 * D) + _a256(N * 4 * (2 * (D // 256) + 1)) + _a256(t * 4 * D)
            + (_a256(t * 8) + _a256(t * 2 * d * 4)) * splits + cand)
    bank = (_a256(2 * n * t * 4 * D) + _a256(4 * 2 * n * t * (2 * (D // 256) + 1))
            + _a256(n * D * tp * 4))
    head = t * ldt * 4 + t * tp * 4
    one_head = bank + head + 1024
    return fixed + max(pair, one_head) + 256


@pytest.mark.parametrize("H,d,D,n,F,N,t", [
    (1, 64, 256, 4, 1024, 1856, 1597),   # past the last latent count with finer sums
    (1, 128, 256, 4, 0, 1697, 1616),
    (1, 128, 512, 8, 0, 5115, 639),      # the scratch holds it with coarse sums only
    (2, 256, 2048, 4, 0, 293, 241),
])
def test_calls_that_fit_the_fixed_scratch(lib, H, d, D, n, F, N, t):
    assert smallest_need(H, d, D, n, F, N, t) <= 64 * MIB
    got = plan(lib, _cfg(H, d, D, n, F, t), N, t, 64 * MIB)
    assert got is not None and got[0] <= 64 * MIB


@pytest.mark.parametrize("H,d,D,n,F", [(1, 64, 256, 4, 1024), (2, 64, 256, 1, 0),
                                       (2, 128, 1024, 2, 2048), (1, 256, 512, 2, 512)])
def test_a_limit_that_holds_the_buffers_is_enough(lib, H, d, D, n, F):
    for N in (40, 257, 1000, 4097):
        for t in (1, 17, 129, 300, 640, 1217, 4000):
            if t > N:
                continue
            cfg = _cfg(H, d, D, n, F, t)
            need = smallest_need(H, d, D, n, F, N, t)
            got = plan(lib, cfg, N, t, need)
            assert got is not None and got[0] <= need, (N, t, need)
            # not half as much: the restatement is the plan's own size, not a loose bound
            assert plan(lib, cfg, N, t, need // 2) is None, (N, t)


def test_finer_sums_cost_no_group(lib):
    """A limit between the needs with coarse and with finer sums keeps the coarse ones' groups."""
    H, d, D, n, F, N, t = 4, 64, 256, 4, 1024, 1024, 200
    cfg = _cfg(H, d, D, n, F, t)
    seen = set()
    last = None
    for limit in range(MIB, 40 * MIB, 65536):
        p = plan(lib, cfg, N, t, limit)
        if p is None:
            assert last is None  # a larger limit never refuses what a smaller one took
            continue
        assert p[0] <= limit
        if last is not None:
            assert p[1:4] >= last[1:4]  # nor makes smaller groups
        seen.add(p[4])
        last = p
    assert last[2] == H and last[4] == D // 32 and seen <= {2 * (D // 256), D // 32}


@pytest.mark.parametrize("H,d,D,n,F", [(2, 64, 256, 4, 1024), (1, 64, 256, 1, 0),
                                       (8, 128, 1024, 8, 4096)])
def test_reservation_serves_every_smaller_call(lib, H, d, D, n, F):
    limit = 48 << 30
    for t_max in (1, 40, 650, 1300, 4000, 5500):
        N = max(6000, t_max)
        cfg = _cfg(H, d, D, n, F, t_max)
        bytes_ = lib.still_internal_reserve(ctypes.byref(cfg), SPLIT, 0, 0, ctypes.c_int64(N), t_max,
                                            ctypes.c_size_t(limit))
        assert bytes_ > 0
        for t in range(1, t_max + 1, max(1, t_max // 200)):
            assert plan(lib, cfg, N, t, limit)[0] <= bytes_, (t_max, t)


def test_finer_sums_end_where_the_device_stops_splitting(lib):
    """2 n d_l / 256 = 4 column tiles: the last latent count whose row tiles times 4 still split,
    for whole and for cut-down devices."""
    H, d, D, n = 2, 64, 256, 2
    for split in (76, 75, 74, 33, 8, 4, 3, 0):
        rows = split // 4 * 128
        for t in {1, max(1, rows // H), rows // H + 1, 700}:
            tiles = -(-H * t // 128) * 4
            cfg = _cfg(H, d, D, n, 512, t)
            parts = plan(lib, cfg, 3000, t, 48 << 30, split)[4]
            assert parts == (D // 32 if tiles <= split else 2 * (D // 256)), (split, t, tiles)
