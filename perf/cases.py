"""The work that users of the Still compactor have it do, as cases that can be timed and compared.

Every case goes through the public entry points of paper_2606_07878_gb300.still. Inputs are the
synthetic caches and random-init weights of paper_2606_07878_gb300.synth (keys with outlier
channels, rotated by the base model's RoPE at their cache positions, bf16), drawn from the seed.
`exact` restates the compactor in 64-bit torch and uses none of the library's code.
"""
from __future__ import annotations

import math

import torch

from paper_2606_07878_gb300 import still, synth

DEVICE = "cuda:0"

# Compactor shapes: H KV-heads of head dim d, width D, n heads, FFN hidden F, blocks, compactor
# RoPE. `most` and `least` bound the cached tokens of a drawn case.
FAMILIES = {
    # a small base model's cache: every launch is short
    "small": dict(H=2, d=64, D=256, n=4, F=1024, theta=1e4, heavy=4, least=256, most=32768),
    # Qwen-7B-shaped
    "qwen7b": dict(H=4, d=128, D=1024, n=8, F=4096, theta=1e6, heavy=4, least=1024, most=32768),
    # Qwen-8B-shaped
    "qwen8b": dict(H=8, d=128, D=1024, n=8, F=4096, theta=1e6, heavy=1, least=1024, most=32768),
    # Gemma-shaped
    "gemma": dict(H=8, d=256, D=2048, n=16, F=8192, theta=1e6, heavy=3, least=2048, most=32768),
    # the paper's canonical compactor on a Qwen3-4B-shaped cache: two blocks, one head, no FFN
    "canonical": dict(H=8, d=128, D=256, n=1, F=0, theta=1e6, heavy=1, n_blocks=2, least=512,
                      most=65536),
    # Qwen-7B-shaped without compactor RoPE: the key projection folds into the queries
    "norope": dict(H=4, d=128, D=1024, n=8, F=4096, theta=1e6, heavy=4, compactor_rope=0,
                   least=1024, most=32768),
}


def listed():
    return [
        # one layer of a short prompt: latency and launches
        dict(name="layer_small_1k", kind="layer", family="small", N=1024, t=128),
        # three sequences at their own passes of the lookahead schedule, 1024-token chunks
        dict(name="lookahead_canonical_3x1k", kind="lookahead", family="canonical", B=3, c=8,
             t=128, first_pass=5),
        # a stack call: the step that a served model makes per document
        dict(name="stack_qwen7b_8k_8x", kind="stack", family="qwen7b", L=4, N=8192, t=1024),
        # one layer with the per-slot bias head, odd sizes
        dict(name="beta_qwen7b_odd", kind="beta", family="qwen7b", N=8003, t=251),
        # a long document at a high ratio (few latents, the cache streams through)
        dict(name="layer_qwen8b_32k_200x", kind="layer", family="qwen8b", N=32768, t=164),
        # the same document at a low ratio (the contractions dominate)
        dict(name="layer_qwen8b_32k_16x", kind="layer", family="qwen8b", N=32768, t=2048),
        # the long-context headline: one of 48 identical layers at 128k tokens
        dict(name="layer_gemma_128k_200x", kind="layer", family="gemma", N=131072, t=655),
        # the same compactor on a mid-size document of odd length
        dict(name="layer_gemma_12k_odd", kind="layer", family="gemma", N=12345, t=617),
        # the paper's canonical two-block compactor at 64k tokens, 50x
        dict(name="layer_canonical_64k_50x", kind="layer", family="canonical", N=65536, t=1311),
        # the ablation without compactor RoPE (folded key path)
        dict(name="layer_norope_8k_8x", kind="layer", family="norope", N=8192, t=1024),
        # iterative serving: compact caches plus 8192 fresh tokens each, re-compacted at 32x
        dict(name="recompact_qwen8b_3seq", kind="recompact", family="qwen8b", lens="9001,20480,31007",
             new=8192, ratio=32),
        # a decode step over compact caches: 36 layers, one token, 32 query heads
        dict(name="decode_36x1_t1311", kind="decode", L=36, nq=1, Hq=32, H=8, d=128, t=1311,
             S=4096, beta=True),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["layer", "layer", "layer", "stack", "beta", "lookahead", "recompact",
                       "decode", "decode"])
    if kind == "decode":
        d = rng.choice([64, 128, 128, 256])
        H = rng.choice([2, 4, 8])
        group = rng.choice([1, 2, 4, 8])
        return dict(kind=kind, L=rng.choice([1, 1, 8, 28, 36, 48]), nq=rng.choice([1, 1, 2, 4]),
                    Hq=H * group, H=H, d=d, t=_log(rng, 16, 4096), S=_log(rng, 1, 8192),
                    beta=rng.random() < 0.5)
    if kind == "lookahead":
        family = rng.choice(["small", "canonical", "qwen8b"])
        t = _log(rng, 16, 256)
        return dict(kind=kind, family=family, B=rng.randint(1, 4), c=rng.choice([8, 16, 32]), t=t,
                    first_pass=rng.randint(0, 40))
    if kind == "recompact":
        family = rng.choice(["small", "qwen7b", "qwen8b"])
        lens = [_log(rng, 2048, 32768) for _ in range(rng.randint(1, 4))]
        return dict(kind=kind, family=family, lens=",".join(map(str, lens)),
                    new=_log(rng, 1024, 8192), ratio=rng.choice([16, 32, 50]))
    family = rng.choice(["small", "qwen7b", "qwen8b", "gemma", "canonical", "norope"])
    f = FAMILIES[family]
    N = _log(rng, f["least"], f["most"])
    t = max(1, min(N, int(round(N / math.exp(rng.uniform(math.log(8), math.log(200)))))))
    if kind == "stack":
        return dict(kind=kind, family=family, L=rng.randint(2, 3), N=min(N, 16384),
                    t=min(t, 2048))
    return dict(kind=kind, family=family, N=N, t=t)


# ------------------------------------------------------------------------------ states

class Context:
    """A library context that is destroyed with the state that holds it."""

    def __init__(self):
        self.handle = still.still_create(0)

    def __del__(self):
        if self.handle is not None:
            still.still_destroy(self.handle)
            self.handle = None


def _workload(case):
    return FAMILIES[case["family"]]


def _lens(case):
    return [int(x) for x in case["lens"].split(",")]


def _budget(n, ratio):  # round half up
    return (2 * n + ratio) // (2 * ratio)


def _recompact_plan(case):
    """Per sequence: previous slots, previous logical length, new tokens, new slots."""
    return [(max(1, _budget(n, case["ratio"])), n, case["new"],
             max(1, _budget(n + case["new"], case["ratio"]))) for n in _lens(case)]


def _t_max(case):
    if case["kind"] == "recompact":
        return max(p[3] for p in _recompact_plan(case))
    return case["t"]


def _weights(case, layer, seed):
    return synth.gen_weights(_workload(case), layer, _t_max(case), DEVICE, seed=seed)


def _cache(case, layer, n, seed, positions=None, stream=0):
    return synth.gen_kv(_workload(case), layer, n, DEVICE, seed=seed + 1, positions=positions,
                        stream=stream)


def _inputs(case, seed):
    """The tensors of a case: weights per layer and caches (or the decode tensors)."""
    kind = case["kind"]
    if kind == "decode":
        g = torch.Generator(device=DEVICE)
        g.manual_seed(seed)

        def rand(*shape):
            return torch.randn(shape, generator=g, device=DEVICE).to(torch.bfloat16)

        L, H, d = case["L"], case["H"], case["d"]
        s = dict(q=[rand(case["nq"], case["Hq"], d) for _ in range(L)],
                 Ck=[rand(case["t"], H, d) for _ in range(L)],
                 Cv=[rand(case["t"], H, d) for _ in range(L)],
                 Kf=[rand(case["S"], H, d) for _ in range(L)],
                 Vf=[rand(case["S"], H, d) for _ in range(L)], beta=None)
        if case["beta"]:
            s["beta"] = [torch.randn((case["t"], H), generator=g, device=DEVICE) for _ in range(L)]
        return s
    if kind == "lookahead":
        B, n = case["B"], case["c"] * case["t"]
        passes = [case["first_pass"] + 3 * b for b in range(B)]
        kv = [_cache(case, 0, n, seed, stream=b,
                     positions=torch.arange(n, dtype=torch.float64) + passes[b] * n)
              for b in range(B)]
        return dict(W=[_weights(case, 0, seed)], passes=passes,
                    K=torch.cat([k for k, _ in kv]), V=torch.cat([v for _, v in kv]))
    if kind == "recompact":
        prev, new = [], []
        for b, (tp, length, nn, _) in enumerate(_recompact_plan(case)):
            at = torch.linspace(0, length - 1, tp, dtype=torch.float64)
            prev.append(_cache(case, 0, tp, seed, stream=2 * b, positions=at))
            new.append(_cache(case, 0, nn, seed, stream=2 * b + 1,
                              positions=length + torch.arange(nn, dtype=torch.float64)))
        return dict(W=[_weights(case, 0, seed)],
                    Kp=torch.cat([k for k, _ in prev]), Vp=torch.cat([v for _, v in prev]),
                    Kn=torch.cat([k for k, _ in new]), Vn=torch.cat([v for _, v in new]))
    L = case.get("L", 1)
    kv = [_cache(case, l, case["N"], seed) for l in range(L)]
    s = dict(W=[_weights(case, l, seed) for l in range(L)], K=[k for k, _ in kv],
             V=[v for _, v in kv])
    if kind == "beta":
        g = torch.Generator(device=DEVICE)
        g.manual_seed(seed + 2)
        w = torch.randn(_workload(case)["D"], generator=g, device=DEVICE)
        s["wbeta"] = (w * 0.02).to(torch.bfloat16)
    return s


def prepare(case, seed):
    wl = _workload(case) if "family" in case else None
    s = dict(_inputs(case, seed), case=case, ctx=Context())
    ctx = s["ctx"].handle
    if case["kind"] == "decode":
        s["out"] = [torch.empty_like(q) for q in s["q"]]
        return s
    for l, W in enumerate(s.pop("W")):
        still.still_load_layer_weights(ctx, l, still.config_from_workload(wl, _t_max(case)), W)
    if case["kind"] == "beta":  # saturated and mass matched, as a serving engine would consume it
        still.still_set_beta_head(ctx, 0, s["wbeta"], beta_max=4.0, mass_match=1)
        s["beta"] = torch.empty((case["t"], wl["H"]), device=DEVICE)
    if case["kind"] == "recompact":
        plan = _recompact_plan(case)
        cum = lambda xs: [sum(xs[:i]) for i in range(len(xs) + 1)]  # noqa: E731
        s["cu_prev"], s["cu_new"] = cum([p[0] for p in plan]), cum([p[2] for p in plan])
        s["prev_len"] = [p[1] for p in plan]
        rows = sum(p[3] for p in plan)
    elif case["kind"] == "lookahead":
        rows = case["B"] * case["t"]
    else:
        rows = case["t"]
    new = lambda: torch.empty((rows, wl["H"], wl["d"]), dtype=torch.bfloat16,  # noqa: E731
                              device=DEVICE)
    L = case.get("L", 1)
    s["Ck"], s["Cv"] = [new() for _ in range(L)], [new() for _ in range(L)]
    return s


def run(state):
    case, ctx = state["case"], state["ctx"].handle
    kind = case["kind"]
    if kind == "decode":
        still.still_attend_biased_stack(ctx, state["q"], state["Ck"], state["Cv"], state["beta"],
                                        state["Kf"], state["Vf"], state["out"])
        return state["out"]
    Ck, Cv = state["Ck"], state["Cv"]
    if kind == "layer":
        still.still_compact_layer(ctx, 0, state["K"][0], state["V"][0], case["t"], Ck[0], Cv[0])
    elif kind == "stack":
        still.still_compact_stack(ctx, state["K"], state["V"], case["t"], Ck, Cv)
    elif kind == "beta":
        still.still_compact_layer_beta(ctx, 0, state["K"][0], state["V"][0], case["t"], Ck[0],
                                       Cv[0], state["beta"])
        return [Ck, Cv, state["beta"]]
    elif kind == "lookahead":
        still.still_lookahead_compact_layer(ctx, 0, state["K"], state["V"], state["passes"],
                                            case["c"], case["t"], Ck[0], Cv[0])
    else:
        still.still_recompact_layer_ragged(ctx, 0, state["Kp"], state["Vp"], state["cu_prev"],
                                           state["prev_len"], state["Kn"], state["Vn"],
                                           state["cu_new"], case["ratio"], Ck[0], Cv[0])
    return [Ck, Cv]


# ------------------------------------------------------------------------------ work, tolerance

def _sequences(case):
    """(tokens, slots) of every layer and sequence that one pass compacts."""
    if case["kind"] == "recompact":
        return [(tp + nn, t) for tp, _, nn, t in _recompact_plan(case)]
    if case["kind"] == "lookahead":
        return [(case["c"] * case["t"], case["t"])] * case["B"]
    return [(case["N"], case["t"])] * case.get("L", 1)


def _layer_flops(f, N, t):
    """Algorithmic flops of one layer: W_V W_O and the first block's queries precomputed, the
    keys projected unless there is no compactor RoPE (then queries and norms fold W_K)."""
    H, d, D, n, F = f["H"], f["d"], f["D"], f["n"], f["F"]
    B, kw = f.get("n_blocks", 1), 2 * d
    total = 4.0 * t * H * D * d
    for b in range(B):
        if f.get("compactor_rope", 1):
            total += 2.0 * N * H * kw * n * D + 2.0 * t * N * H * n * D
        else:
            total += 2.0 * N * H * n * kw * kw + 2.0 * t * N * H * n * kw
        if b > 0:
            total += 2.0 * t * H * D * n * D
        total += 2.0 * t * N * H * n * kw + 2.0 * t * H * n * kw * D  # P X, then W_V W_O
        total += 6.0 * t * H * D * n * D + 4.0 * t * t * H * n * D + 2.0 * t * H * n * D * D
        total += 4.0 * t * H * D * F
    return total


def work(case):
    if case["kind"] == "decode":
        rows = case["t"] + case["S"]
        kv = 2 * rows * case["H"] * case["d"] * 2
        if case["beta"]:
            kv += 4 * case["t"] * case["H"]
        qo = 2 * case["nq"] * case["Hq"] * case["d"] * 2
        return {"bytes": case["L"] * (kv + qo),
                "flops": case["L"] * 4.0 * case["nq"] * case["Hq"] * case["d"] * rows}
    f = _workload(case)
    seqs = _sequences(case)
    row = 2 * 2 * f["H"] * f["d"]  # bytes of a K and a V row
    weights = sum(2 * math.prod(s) for s in synth.weight_shapes(
        f["H"], f["d"], f["D"], f["n"], f["F"], _t_max(case), f.get("n_blocks", 1)).values())
    return {"bytes": sum(row * (N + t) for N, t in seqs) + weights * case.get("L", 1),
            "flops": sum(_layer_flops(f, N, t) for N, t in seqs)}


def tolerance(case):
    # Outputs are bf16: against 64 bits every case measures 1.7e-3, the rounding of the outputs
    # themselves. Four times that between two implementations.
    if case["kind"] == "decode":
        return {"rel": 7e-3, "max": 2e-2}  # 32-bit sums: single values move by one bf16 step
    # The logits d_l cos(q, k) of the latent self-attention amplify a changed rounding upstream
    # in single rows: up to 0.02 x RMS in one block, 0.03 in two.
    two = _workload(case).get("n_blocks", 1) > 1
    return {"rel": 7e-3, "max": 0.12 if two else 0.08}


# ------------------------------------------------------------------------------ 64-bit values

EXACT_MOST_FLOPS = 1.6e13  # more than this takes too long in 64 bits


def _angles(pos, width, base):
    m = torch.arange(width // 2, dtype=torch.float64, device=DEVICE)
    return pos.to(device=DEVICE, dtype=torch.float64)[:, None] * base ** (-2.0 * m / width)


def _rotate(x, pos, base, sign=1.0):
    h = x.shape[-1] // 2
    ang = sign * _angles(pos, x.shape[-1], base)
    c, s = torch.cos(ang), torch.sin(ang)
    a, b = x[:, :h], x[:, h:]
    return torch.cat([a * c - b * s, a * s + b * c], dim=-1)


def _rms(x):
    return x / torch.sqrt((x * x).mean(-1, keepdim=True) + 1e-6)


def _unit(x):
    return x / x.norm(dim=-1, keepdim=True).clamp_min(1e-12)


def _spread(lo, hi, t):
    if t == 1:
        return torch.full((1,), lo, dtype=torch.float64)
    return torch.linspace(lo, hi, t, dtype=torch.float64)


def _exact_head(f, W, Kh, Vh, Z, pos):
    """One KV-head in 64 bits: (C_k, C_v, Z_out)."""
    D, n, theta = f["D"], f["n"], f["theta"]
    rope = f.get("compactor_rope", 1)
    t = Z.shape[0]
    out_pos = _spread(float(pos.min()), float(pos.max()), t)
    X = torch.cat([_rotate(Kh.double(), pos, theta, -1.0), Vh.double()], dim=-1)
    Z = Z.double()
    for b in range(f.get("n_blocks", 1)):
        def w(name):
            return W[name if b == 0 else "%s@%d" % (name, b)]

        Zn = _rms(Z)
        add = torch.zeros_like(Z)
        for i in range(n):
            c = slice(i * D, (i + 1) * D)
            q = _unit(Zn @ w("Wq")[:, c].double() + w("bq")[c].double())
            k = _unit(X @ w("Wk")[:, c].double() + w("bk")[c].double())
            if rope:
                q, k = _rotate(q, out_pos, 10.0), _rotate(k, pos, 10.0)
            PX = torch.softmax(D * (q @ k.T), dim=-1) @ X
            add += (PX @ w("Wv")[:, c].double()) @ w("Wo")[c].double()
        Z = Z + add
        Zn = _rms(Z)
        add = torch.zeros_like(Z)
        for i in range(n):
            c = slice(i * D, (i + 1) * D)
            q = _unit(Zn @ w("Sq")[:, c].double() + w("sbq")[c].double())
            k = _unit(Zn @ w("Sk")[:, c].double() + w("sbk")[c].double())
            P = torch.softmax(D * (q @ k.T), dim=-1)
            add += (P @ (Zn @ w("Sv")[:, c].double())) @ w("So")[c].double()
        Z = Z + add
        if f["F"]:
            Z = Z + torch.nn.functional.gelu(_rms(Z) @ w("W1").double()) @ w("W2").double()
    Ck = _rotate(Z @ W["Wkey"].double(), out_pos, theta)
    return Ck, Z @ W["Wval"].double(), Z


def _exact_seq(f, W, K, V, pos, t):
    heads = [_exact_head(f, W, K[:, h], V[:, h], W["Z"][h, :t], pos) for h in range(f["H"])]
    return [torch.stack([h[j] for h in heads], dim=1) for j in range(3)]


def exact(case, seed):
    if work(case)["flops"] > EXACT_MOST_FLOPS:
        return None
    s = _inputs(case, seed)
    if case["kind"] == "decode":
        group, outs = case["Hq"] // case["H"], []
        for l in range(case["L"]):
            K = torch.cat([s["Ck"][l], s["Kf"][l]]).double().repeat_interleave(group, dim=1)
            V = torch.cat([s["Cv"][l], s["Vf"][l]]).double().repeat_interleave(group, dim=1)
            logits = torch.einsum("qhd,nhd->qhn", s["q"][l].double(), K) / math.sqrt(case["d"])
            if s["beta"] is not None:
                b = s["beta"][l].double().repeat_interleave(group, dim=1).T
                logits[:, :, :case["t"]] += b[None]
            outs.append(torch.einsum("qhn,nhd->qhd", torch.softmax(logits, dim=-1), V))
        return outs
    f = _workload(case)
    if case["kind"] == "lookahead":
        n, t = case["c"] * case["t"], case["t"]
        got = [_exact_seq(f, s["W"][0], s["K"][b * n:(b + 1) * n], s["V"][b * n:(b + 1) * n],
                          torch.arange(n, dtype=torch.float64) + p * n, t)
               for b, p in enumerate(s["passes"])]
    elif case["kind"] == "recompact":
        got, a0, b0 = [], 0, 0
        for tp, length, nn, t in _recompact_plan(case):
            pos = torch.cat([_spread(0.0, length - 1.0, tp),
                             length + torch.arange(nn, dtype=torch.float64)])
            K = torch.cat([s["Kp"][a0:a0 + tp], s["Kn"][b0:b0 + nn]])
            V = torch.cat([s["Vp"][a0:a0 + tp], s["Vn"][b0:b0 + nn]])
            got.append(_exact_seq(f, s["W"][0], K, V, pos, t))
            a0, b0 = a0 + tp, b0 + nn
    else:
        pos = torch.arange(case["N"], dtype=torch.float64)
        got = [_exact_seq(f, W, K, V, pos, case["t"]) for W, K, V in zip(s["W"], s["K"], s["V"])]
        if case["kind"] == "beta":
            Zout = got[0][2]
            b = 4.0 * torch.tanh(Zout @ s["wbeta"].double() / 4.0)
            return [[got[0][0]], [got[0][1]], b + math.log(case["N"] / case["t"])]
        return [[g[0] for g in got], [g[1] for g in got]]
    return [[torch.cat([g[0] for g in got])], [torch.cat([g[1] for g in got])]]
