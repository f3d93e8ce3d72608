"""Timed cases of the library's public entry points, with 64-bit references.

Each case is one pass of what a closed-loop policy has the library do: one linear, the linears
of a decoder or vision block, whole transformer layers recorded as one chain, attention, the
norm and rotary steps, or packing a weight matrix. Inputs are synthetic (weights ~N(0, 0.02),
activations ~N(0, 1) in bf16), made on the GPU from the seed alone; the sizes are those of
`workloads` and generic odd ones.

`listed()` gives the named cases, `draw(rng)` another one of the same ranges, `prepare(case,
seed)` what a program holds before the call (packed weights, activations, outputs, recorded
chain), `run(state)` one pass, `work(case)` the bytes and operations it cannot do without,
`tolerance(case)` how far two correct implementations may be apart, and `exact(case, seed)`
the outputs in 64 bits from plain torch.
"""
from __future__ import annotations

import math

import torch

import paper_2607_02501_gb300 as emb

FORMATS = {"q8_0": emb.EMB_Q8_0, "q6_0": emb.EMB_Q6_0, "q4_0": emb.EMB_Q4_0}
BLOCK_BYTES = {"q8_0": 34, "q6_0": 26, "q4_0": 18}  # packed bytes per 32 weights
PACK = {"q8_0": emb.emb_quantize_q8_0, "q6_0": emb.emb_quantize_q6_0, "q4_0": emb.emb_quantize_q4_0}
GATED = {"geglu": emb.EMB_EPI_GEGLU, "swiglu": emb.EMB_EPI_SWIGLU}
ROPE_BASE = 10000.0
EPS = 1e-6


# ----------------------------------------------------------------------------- the cases

def listed():
    return [
        # one projection of an action-token decode step, called by itself: launch latency
        {"name": "linear_q8_m1", "kind": "linear", "fmt": "q8_0", "M": 1, "N": 2048, "K": 2048,
         "precise": False},
        # a projection with ragged sizes in every dimension for a handful of tokens
        {"name": "linear_q4_m17_odd", "kind": "linear", "fmt": "q4_0", "M": 17, "N": 1000, "K": 1184,
         "precise": False},
        # the linears of one 2B decode step in the 8-bit format, recorded as one chain
        {"name": "decode_q8_2b", "kind": "decoder", "fmt": "q8_0", "M": 1, "D": 2048, "Q": 2048, "KV": 256,
         "F": 16384, "layers": 18, "act": "none", "recorded": True, "outliers": 0.0},
        # whole 7B layers of one decode step in the 4-bit format over a 280-token prefix
        {"name": "layers_q4_7b_m1", "kind": "layers", "fmt": "q4_0", "M": 1, "D": 4096, "H": 32, "Hk": 32,
         "d": 128, "F": 11008, "prefix": 280, "layers": 8, "act": "swiglu", "outliers": 0.01},
        # 2B linears in the 6-bit format for four token streams at a time
        {"name": "decode_q6_2b_m4", "kind": "decoder", "fmt": "q6_0", "M": 4, "D": 2048, "Q": 2048, "KV": 256,
         "F": 16384, "layers": 4, "act": "none", "recorded": True, "outliers": 0.0},
        # one denoising step of the action expert: 18 whole layers for a 50-token chunk over
        # the 816-token prefix cache
        {"name": "expert_step_m50", "kind": "layers", "fmt": "q8_0", "M": 50, "D": 1024, "H": 8, "Hk": 1,
         "d": 128, "F": 4096, "prefix": 816, "layers": 18, "act": "geglu", "outliers": 0.0},
        # prefix prefill of the 2B backbone (3 x 256 image + 48 text tokens), two layers' linears
        {"name": "prefill_q8_2b_m816", "kind": "decoder", "fmt": "q8_0", "M": 816, "D": 2048, "Q": 2048,
         "KV": 256, "F": 16384, "layers": 2, "act": "geglu", "recorded": False, "outliers": 0.0},
        # prefix prefill of the 7B backbone (256 image + 24 text tokens), two layers' linears
        {"name": "prefill_q4_7b_m280", "kind": "decoder", "fmt": "q4_0", "M": 280, "D": 4096, "Q": 4096,
         "KV": 4096, "F": 11008, "layers": 2, "act": "swiglu", "recorded": False, "outliers": 0.01},
        # the vision tower's linears on three images, six of its layers
        {"name": "vit_q8_m768", "kind": "vit", "fmt": "q8_0", "M": 768, "D": 1152, "F": 4608, "layers": 6},
        # the prefix tokens attending to one another during prefill
        {"name": "attention_m816", "kind": "attention", "M": 816, "H": 8, "Hk": 1, "d": 128, "n0": 0, "n1": 816},
        # the norm and rotary steps of one prefill layer, called one by one
        {"name": "norm_rope_m816", "kind": "norm_rope", "M": 816, "D": 2048, "H": 8, "Hk": 1, "d": 256, "pos0": 0},
        # packing one matrix while a model is loaded
        {"name": "pack_q4_22016x4096", "kind": "pack", "fmt": "q4_0", "N": 22016, "K": 4096},
    ]


def _log(rng, lo, hi, step=1):
    """A multiple of `step` spread over the logarithm of lo .. hi."""
    v = math.exp(rng.uniform(math.log(lo), math.log(hi + step)))
    return min(hi // step * step, max(-(-lo // step) * step, int(v) // step * step))


def draw(rng):
    """Another case of the listed ranges. Sizes go from one token and narrow layers to the
    largest listed ones, odd ones among them (K in multiples of the 32-weight block, 64 for
    the 6-bit format's larger token counts)."""
    kind = rng.choice(["linear", "linear", "decoder", "decoder", "layers", "vit", "attention", "norm_rope", "pack"])
    fmt = rng.choice(sorted(FORMATS))
    k_step = 64 if fmt == "q6_0" else 32
    if kind == "linear":
        M = _log(rng, 1, 900)
        K = _log(rng, 128, 16384, k_step)
        N = _log(rng, 64, max(65, min(32768, (1 << 27) // K)))
        return {"kind": kind, "fmt": fmt, "M": M, "N": N, "K": K, "precise": rng.random() < 0.15}
    if kind in ("decoder", "vit"):
        M = rng.choice([1, 1, _log(rng, 2, 4), _log(rng, 5, 64), _log(rng, 65, 820)])
        D = _log(rng, 512, 4096, 64)
        if kind == "vit":
            return {"kind": kind, "fmt": fmt, "M": max(M, 16), "D": D, "F": min(16384, 4 * D),
                    "layers": rng.randint(1, 2 if D > 2048 else 4)}
        F = _log(rng, 2 * D, min(16384, 8 * D), 64)
        return {"kind": kind, "fmt": fmt, "M": M, "D": D, "Q": D, "KV": rng.choice([D, max(64, D // 8 // 64 * 64)]),
                "F": F, "layers": rng.randint(1, 2 if M > 64 else 6), "act": rng.choice(["none", "geglu", "swiglu"]),
                "recorded": rng.random() < 0.5, "outliers": rng.choice([0.0, 0.01])}
    if kind == "layers":
        d = rng.choice([64, 128])
        Hk = rng.choice([1, 2, 8])
        H = Hk * rng.choice([1, 4, 8] if Hk < 8 else [1, 2, 4])
        return {"kind": kind, "fmt": fmt, "M": rng.choice([1, _log(rng, 2, 64), _log(rng, 20, 120)]),
                "D": _log(rng, 1024, 3072, 64), "H": H, "Hk": Hk, "d": d, "F": _log(rng, 2048, 8192, 64),
                "prefix": _log(rng, 64, 1200), "layers": rng.randint(2, 8), "act": rng.choice(["geglu", "swiglu"]),
                "outliers": 0.0}
    if kind == "attention":
        Hk = rng.choice([1, 2, 4, 8])
        H = Hk * rng.choice([1, 2, 4, 8] if Hk < 8 else [1, 2])
        return {"kind": kind, "M": _log(rng, 1, 850), "H": H, "Hk": Hk, "d": rng.choice([64, 128]),
                "n0": rng.choice([0, _log(rng, 16, 1200)]), "n1": _log(rng, 1, 850)}
    if kind == "norm_rope":
        return {"kind": kind, "M": _log(rng, 1, 900), "D": _log(rng, 256, 4096, 8), "H": rng.choice([4, 8, 16, 32]),
                "Hk": rng.choice([1, 2, 4]), "d": rng.choice([64, 72, 128, 256]), "pos0": rng.randint(0, 2000)}
    K = _log(rng, 256, 16384, 32)
    return {"kind": "pack", "fmt": fmt, "N": _log(rng, 64, min(32768, (1 << 26) // K)), "K": K}


# ----------------------------------------------------------------------------- inputs

def _gen(seed, index):
    return torch.Generator(device="cuda").manual_seed((seed * 1000003 + index * 7919 + 17) % (1 << 62))


def _weight(N, K, seed, index, outliers=0.0):
    """fp32 W [N][K] ~ N(0, 0.02); a share `outliers` of the entries is eight times larger."""
    g = _gen(seed, index)
    w = torch.randn(N, K, generator=g, device="cuda").mul_(0.02)
    if outliers > 0:
        w *= 1.0 + 7.0 * (torch.rand(N, K, generator=g, device="cuda") < outliers)
    return w


def _normal(shape, seed, index, dtype=torch.bfloat16, scale=1.0, shift=0.0):
    return torch.randn(*shape, generator=_gen(seed, index), device="cuda").mul_(scale).add_(shift).to(dtype)


def _decoder_linears(case):
    """(name, N, K) of one decoder layer; gate and up are one matrix of interleaved rows when gated."""
    D, Q, KV, F = case["D"], case["Q"], case["KV"], case["F"]
    gu = [("gate", F, D), ("up", F, D)] if case["act"] == "none" else [("gate_up", 2 * F, D)]
    return [("q", Q, D), ("k", KV, D), ("v", KV, D), ("o", D, Q), *gu, ("down", D, F)]


def _vit_linears(case):
    D, F = case["D"], case["F"]
    return [("qkv", 3 * D, D), ("o", D, D), ("fc1", F, D), ("fc2", D, F)]


def _layer_linears(case):
    D, q, kv, F = case["D"], case["H"] * case["d"], case["Hk"] * case["d"], case["F"]
    return [("q", q, D), ("k", kv, D), ("v", kv, D), ("o", D, q), ("gate_up", 2 * F, D), ("down", D, F)]


def _packed(case, N, K, seed, index):
    return emb.quantize(FORMATS[case["fmt"]], _weight(N, K, seed, index, case.get("outliers", 0.0)))


def _group_input(name):
    """The linears of one group read the same activation."""
    return {"k": "q", "v": "q", "up": "gate"}.get(name, name)


def _chain_plan(case):
    """Per linear of a decoder or vision chain: (layer, name, N, K, epilogue, index of its
    weights and input). With `act`, q/k/v and the gated product are bf16, o and down add into
    the residual; otherwise every output is fp32."""
    fused = case.get("act", "none") != "none"
    linears = _vit_linears(case) if case["kind"] == "vit" else _decoder_linears(case)
    epi = {"q": emb.EMB_EPI_BF16, "k": emb.EMB_EPI_BF16, "v": emb.EMB_EPI_BF16, "o": emb.EMB_EPI_ADD,
           "gate_up": GATED.get(case.get("act")), "down": emb.EMB_EPI_ADD}
    plan = []
    for layer in range(case["layers"]):
        for j, (name, N, K) in enumerate(linears):
            plan.append((layer, name, N, K, epi[name] if fused else emb.EMB_EPI_F32, layer * 16 + j))
    return plan


def _chain_inputs(case, seed):
    """Activation of every group of the chain, by (layer, group). A fused chain's down
    projection reads the gated product instead."""
    X = {}
    for layer, name, _, K, epi, index in _chain_plan(case):
        key = (layer, _group_input(name))
        if key not in X and not (name == "down" and epi == emb.EMB_EPI_ADD):
            X[key] = _normal((case["M"], K), seed, 100000 + index)
    return X


def _residual(case, seed):
    return _normal((case["M"], case["D"]), seed, 200000, torch.float32, 2.0)


def _layer_gains(case, layer, seed):
    return [_normal((case["D"],), seed, 300000 + 2 * layer + j, torch.float32, 0.1, 1.0) for j in (0, 1)]


def _layer_cache(case, layer, seed):
    n = case["Hk"] * case["d"]
    return [_normal((case["prefix"], n), seed, 400000 + 2 * layer + j) for j in (0, 1)]


def _attention_inputs(case, seed):
    q, kv = case["H"] * case["d"], case["Hk"] * case["d"]
    shapes = [(case["M"], q), (case["n0"], kv), (case["n0"], kv), (case["n1"], kv), (case["n1"], kv)]
    return [_normal(s, seed, 500000 + i) if s[0] else None for i, s in enumerate(shapes)]


def _norm_rope_inputs(case, seed):
    M, d = case["M"], case["d"]
    return (_normal((M, case["D"]), seed, 600000, torch.float32, 2.0),
            _normal((case["D"],), seed, 600001, torch.float32, 0.1, 1.0),
            _normal((M, case["H"] * d), seed, 600002), _normal((M, case["Hk"] * d), seed, 600003))


# ----------------------------------------------------------------------------- one pass

def prepare(case, seed):
    return {"linear": _prepare_linear, "decoder": _prepare_chain, "vit": _prepare_chain, "layers": _prepare_layers,
            "attention": _prepare_attention, "norm_rope": _prepare_norm_rope, "pack": _prepare_pack}[case["kind"]](case, seed)


def run(state):
    return state["run"](state)


def _prepare_linear(case, seed):
    M, N, K = case["M"], case["N"], case["K"]
    W, X = _packed(case, N, K, seed, 0), _normal((M, K), seed, 100000)
    Y = torch.empty(M, N, dtype=torch.float32, device="cuda")
    state = {"W": W, "X": X, "Y": Y, "fmt": FORMATS[case["fmt"]], "M": M, "N": N, "K": K, "run": _run_linear}
    if case["precise"]:  # an option of the layer calls
        state["layers"] = emb.make_layers([(state["fmt"], W, N, K, X, Y, emb.EMB_EPI_F32 | emb.EMB_PRECISE_OPERAND)])
    return state


def _run_linear(s):
    if "layers" in s:
        emb.emb_qlayer_seq(s["layers"], s["M"])
    else:
        emb.emb_qmatmul(s["fmt"], s["W"], s["X"], s["Y"], s["M"], s["N"], s["K"])
    return s["Y"]


def _prepare_chain(case, seed):
    M, plan = case["M"], _chain_plan(case)
    X = _chain_inputs(case, seed)
    R0 = R = None
    if any(epi == emb.EMB_EPI_ADD for *_, epi, _ in plan):
        R0 = _residual(case, seed)
        R = torch.empty_like(R0)
    # the outputs of one type share one buffer, as a step that moves them with one copy has it
    sizes = {torch.float32: 0, torch.bfloat16: 0}
    spans = []
    for _, _, N, _, epi, _ in plan:
        kind = torch.float32 if epi == emb.EMB_EPI_F32 else torch.bfloat16
        n = 0 if epi == emb.EMB_EPI_ADD else M * (N if epi in (emb.EMB_EPI_F32, emb.EMB_EPI_BF16) else N // 2)
        spans.append((kind, sizes[kind], n))
        sizes[kind] += -(-n // 64) * 64
    arena = {kind: torch.zeros(n, dtype=kind, device="cuda") for kind, n in sizes.items() if n}
    specs, gated = [], {}
    for (layer, name, N, K, epi, index), (kind, at, n) in zip(plan, spans):
        Y = R if epi == emb.EMB_EPI_ADD else arena[kind][at:at + n]
        if name == "gate_up":
            gated[layer] = Y
        x = gated[layer] if name == "down" and layer in gated else X[(layer, _group_input(name))]
        specs.append((FORMATS[case["fmt"]], _packed(case, N, K, seed, index), N, K, x, Y, epi))
    state = {"specs": specs, "M": M, "R0": R0, "R": R, "arena": list(arena.values()), "run": _run_chain}
    if case.get("recorded", True):
        state["chain"] = emb.RecordedChain(specs, M)
    else:
        state["layers"] = emb.make_layers(specs)
        state["ws"] = emb.chain_workspace(state["layers"], M)
    return state


def _run_chain(s):
    if s["R"] is not None:
        s["R"].copy_(s["R0"])
    if "chain" in s:
        s["chain"].launch()
    else:
        emb.emb_qlayer_seq(s["layers"], s["M"], s["ws"], 0 if s["ws"] is None else s["ws"].numel())
    return s["arena"] + ([s["R"]] if s["R"] is not None else [])


def _prepare_layers(case, seed):
    M, D, H, Hk, d, F, P = (case[k] for k in ("M", "D", "H", "Hk", "d", "F", "prefix"))
    fmt, L = FORMATS[case["fmt"]], case["layers"]
    bf = lambda *shape: torch.zeros(*shape, dtype=torch.bfloat16, device="cuda")
    R0 = _residual(case, seed)
    R = torch.empty_like(R0)
    h, q, a, g = bf(M, D), bf(M, H * d), bf(M, H * d), bf(M, F)
    k, v = bf(L, M, Hk * d), bf(L, M, Hk * d)
    keep = [R0, R, h, q, a, g, k, v]
    stream = torch.cuda.Stream()
    weights = [[_packed(case, N, K, seed, layer * 16 + j) for j, (_, N, K) in enumerate(_layer_linears(case))]
               for layer in range(L)]
    gains = [_layer_gains(case, layer, seed) for layer in range(L)]
    caches = [_layer_cache(case, layer, seed) for layer in range(L)]
    stream.wait_stream(torch.cuda.current_stream())
    rec = emb.Recording(stream, keep=keep + weights + gains + caches)
    with torch.cuda.stream(stream), rec:
        for layer in range(L):
            Wq, Wk, Wv, Wo, Wgu, Wd = weights[layer]
            K0, V0 = caches[layer]
            emb.emb_rmsnorm(R, gains[layer][0], h, EPS)
            emb.emb_qlayer_seq_chained([(fmt, Wq, H * d, D, h, q, emb.EMB_EPI_BF16),
                                        (fmt, Wk, Hk * d, D, h, k[layer], emb.EMB_EPI_BF16),
                                        (fmt, Wv, Hk * d, D, h, v[layer], emb.EMB_EPI_BF16)], M)
            emb.emb_rope_qk(q, H, k[layer], Hk, d, P, ROPE_BASE)
            emb.emb_attention(q, K0, V0, k[layer], v[layer], a, H, Hk, d, 1.0 / math.sqrt(d))
            emb.emb_qlayer_seq_chained([(fmt, Wo, D, H * d, a, R, emb.EMB_EPI_ADD)], M)
            emb.emb_rmsnorm(R, gains[layer][1], h, EPS)
            emb.emb_qlayer_seq_chained([(fmt, Wgu, 2 * F, D, h, g, GATED[case["act"]])], M)
            emb.emb_qlayer_seq_chained([(fmt, Wd, D, F, g, R, emb.EMB_EPI_ADD)], M)
    torch.cuda.current_stream().wait_stream(stream)
    return {"rec": rec, "R0": R0, "R": R, "k": k, "v": v, "run": _run_layers}


def _run_layers(s):
    s["R"].copy_(s["R0"])
    s["rec"].launch()
    return [s["R"], s["k"], s["v"]]


def _prepare_attention(case, seed):
    Q, K0, V0, K1, V1 = _attention_inputs(case, seed)
    return {"in": (Q, K0, V0, K1, V1), "O": torch.empty_like(Q), "H": case["H"], "Hk": case["Hk"], "d": case["d"],
            "run": _run_attention}


def _run_attention(s):
    emb.emb_attention(*s["in"], s["O"], s["H"], s["Hk"], s["d"], 1.0 / math.sqrt(s["d"]))
    return s["O"]


def _prepare_norm_rope(case, seed):
    x, gamma, q, k = _norm_rope_inputs(case, seed)
    return {"x": x, "gamma": gamma, "q": q, "k": k, "y": torch.empty_like(x, dtype=torch.bfloat16),
            "H": case["H"], "Hk": case["Hk"], "d": case["d"], "pos0": case["pos0"], "run": _run_norm_rope}


def _run_norm_rope(s):
    # q and k are rotated in place; a further pass rotates them again
    emb.emb_rmsnorm(s["x"], s["gamma"], s["y"], EPS)
    emb.emb_rope_qk(s["q"], s["H"], s["k"], s["Hk"], s["d"], s["pos0"], ROPE_BASE)
    return [s["y"], s["q"], s["k"]]


def _prepare_pack(case, seed):
    N, K = case["N"], case["K"]
    return {"W": _weight(N, K, seed, 0), "out": emb.empty_qweight(FORMATS[case["fmt"]], N, K),
            "pack": PACK[case["fmt"]], "N": N, "K": K, "run": _run_pack}


def _run_pack(s):
    s["pack"](s["W"], s["N"], s["K"], s["out"])
    return s["out"]


# ----------------------------------------------------------------------------- work

def _output_bytes(epi, M, N):
    return {emb.EMB_EPI_F32: 4, emb.EMB_EPI_BF16: 2, emb.EMB_EPI_ADD: 8}.get(epi, 1) * M * N


def work(case):
    """Each input read once and each output written once; two operations per multiply-add."""
    kind, M = case["kind"], case.get("M", 0)
    if kind == "pack":
        n = case["N"] * case["K"]
        return {"bytes": 4 * n + n // 32 * BLOCK_BYTES[case["fmt"]], "flops": 0}
    if kind == "attention":
        n, q, kv = case["n0"] + case["n1"], case["H"] * case["d"], case["Hk"] * case["d"]
        return {"bytes": 2 * (2 * M * q + 2 * n * kv), "flops": 4 * M * q * n}
    if kind == "norm_rope":
        D, qk = case["D"], (case["H"] + case["Hk"]) * case["d"]
        return {"bytes": 6 * M * D + 4 * D + 4 * M * qk, "flops": 4 * M * D + 3 * M * qk}
    per = BLOCK_BYTES[case["fmt"]]
    if kind == "linear":
        N, K = case["N"], case["K"]
        return {"bytes": N * K // 32 * per + 2 * M * K + 4 * M * N, "flops": 2 * M * N * K}
    if kind == "layers":
        D, F, L, n = case["D"], case["F"], case["layers"], case["prefix"] + M
        q, kv = case["H"] * case["d"], case["Hk"] * case["d"]
        weights = sum(N * K for _, N, K in _layer_linears(case))
        # weights, gains and caches of every layer, the chunk's keys and values out, the residual in and out
        return {"bytes": L * (weights // 32 * per + 8 * D + 4 * n * kv) + 8 * M * D,
                "flops": L * (2 * M * weights + 4 * M * q * n)}
    bytes_, flops, read = 0, 0, set()
    for layer, name, N, K, epi, _ in _chain_plan(case):
        key = (layer, _group_input(name))
        bytes_ += N * K // 32 * per + _output_bytes(epi, M, N) + (0 if key in read else 2 * M * K)
        read.add(key)
        flops += 2 * M * N * K
    return {"bytes": bytes_, "flops": flops}


# ----------------------------------------------------------------------------- tolerance

def tolerance(case):
    """About four times the error against `exact` seen on one GB300, by what rounds the output:
    fp32 sums of exact products 8e-8 (stated as 1e-6, for sums in any order), products of weights
    held as bf16 hi + lo pairs (K < 1024, precise) below 2^-16, bf16 operands or one bf16 result
    1.7e-3, a bf16 result of bf16 operands feeding a further linear 3.1e-3, whole layers 3.8e-3
    (18 of the action expert) and 8.6e-3 (8 of the 7B backbone, whose outliers amplify)."""
    kind, M = case["kind"], case.get("M", 0)
    if kind == "pack":
        return "exact"
    if kind == "layers":
        return {"rel": 3e-2 if case["outliers"] else 1.5e-2}
    if kind in ("attention", "norm_rope"):
        return {"rel": 7e-3}
    if case.get("act", "none") != "none":
        return {"rel": 1.2e-2}
    if M <= 4:
        return {"rel": 1e-6}
    if kind == "linear" and (case["precise"] or case["K"] < 1024):
        return {"rel": 3e-5}
    return {"rel": 7e-3}


# ----------------------------------------------------------------------------- 64-bit values

def _dequantised(fmt, W):
    """The packed weights' values in 64 bits: each 32-weight block's scale and codes by the
    format's definition (one correctly rounded fp32 division, one fp16 rounding of the scale,
    ties of the codes away from zero)."""
    N, K = W.shape
    w = W.view(N, K // 32, 32)
    mag = w.abs()
    top = mag.amax(-1)
    if fmt == "q8_0":
        num, div, lo, hi = top, 127.0, -127.0, 127.0
    else:  # the signed weight of largest magnitude, the first one on ties
        half = 8.0 if fmt == "q4_0" else 32.0
        place = torch.where(mag == top.unsqueeze(-1), torch.arange(32, device=W.device), 32).amin(-1, keepdim=True)
        num, div, lo, hi = w.gather(-1, place).squeeze(-1), -half, -half, half - 1
    d = (num / torch.full_like(num, div)).to(torch.float16).float().unsqueeze(-1)
    t = torch.where(d == 0, torch.zeros_like(w), w / torch.where(d == 0, torch.ones_like(d), d)).double()
    q = (t.sign() * (t.abs() + 0.5).floor()).clamp_(lo, hi)
    return (q * d.double()).view(N, K)


def _matmul(case, x, N, K, seed, index):
    return x @ _dequantised(case["fmt"], _weight(N, K, seed, index, case.get("outliers", 0.0))).T


def _gate(act, y):
    gate, up = y[:, 0::2], y[:, 1::2]
    if act == "swiglu":
        return gate * torch.sigmoid(gate) * up
    return 0.5 * gate * (1.0 + torch.tanh(math.sqrt(2.0 / math.pi) * (gate + 0.044715 * gate ** 3))) * up


def _norm(x, gamma):
    eps = float(torch.tensor(EPS, dtype=torch.float32))
    return x / torch.sqrt((x * x).mean(-1, keepdim=True) + eps) * gamma.double()


def _rotate(x, heads, d, pos0):
    M = x.shape[0]
    i = torch.arange(d // 2, dtype=torch.float64, device=x.device)
    angle = (pos0 + torch.arange(M, dtype=torch.float64, device=x.device))[:, None, None] * ROPE_BASE ** (-2.0 * i / d)
    c, s = torch.cos(angle), torch.sin(angle)
    a, b = x.view(M, heads, d).split(d // 2, -1)
    return torch.cat([a * c - b * s, b * c + a * s], -1).reshape(M, heads * d)


def _attend(Q, K, V, H, Hk, d):
    M, n = Q.shape[0], K.shape[0]
    q = Q.view(M, Hk, H // Hk, d).permute(1, 2, 0, 3).reshape(Hk, -1, d)
    k, v = K.view(n, Hk, d).transpose(0, 1), V.view(n, Hk, d).transpose(0, 1)
    p = torch.softmax(q @ k.transpose(1, 2) * float(torch.tensor(1.0 / math.sqrt(d), dtype=torch.float32)), -1)
    return (p @ v).view(Hk, H // Hk, M, d).permute(2, 0, 1, 3).reshape(M, H * d)


def exact(case, seed):
    kind, M = case["kind"], case.get("M", 0)
    if kind == "pack":
        return None  # bytes, compared as such
    if kind == "linear":
        return _matmul(case, _normal((M, case["K"]), seed, 100000).double(), case["N"], case["K"], seed, 0)
    if kind == "attention":
        Q, K0, V0, K1, V1 = _attention_inputs(case, seed)
        join = lambda a, b: torch.cat([t.double() for t in (a, b) if t is not None])
        return _attend(Q.double(), join(K0, K1), join(V0, V1), case["H"], case["Hk"], case["d"])
    if kind == "norm_rope":
        x, gamma, q, k = _norm_rope_inputs(case, seed)
        return [_norm(x.double(), gamma), _rotate(q.double(), case["H"], case["d"], case["pos0"]),
                _rotate(k.double(), case["Hk"], case["d"], case["pos0"])]
    return _exact_layers(case, seed) if kind == "layers" else _exact_chain(case, seed)


def _exact_chain(case, seed):
    M, X = case["M"], _chain_inputs(case, seed)
    R, gated, parts = None, {}, {}
    for layer, name, N, K, epi, index in _chain_plan(case):
        x = gated[layer] if name == "down" and layer in gated else X[(layer, _group_input(name))].double()
        y = _matmul(case, x, N, K, seed, index)
        if epi == emb.EMB_EPI_ADD:
            R = (_residual(case, seed).double() if R is None else R) + y
            continue
        if name == "gate_up":
            y = gated[layer] = _gate(case["act"], y)
        pad = torch.zeros(-y.numel() % 64, dtype=torch.float64, device="cuda")
        parts.setdefault(epi == emb.EMB_EPI_F32, []).append(torch.cat([y.reshape(-1), pad]))
    return [torch.cat(parts[f32]) for f32 in (True, False) if f32 in parts] + ([R] if R is not None else [])


def _exact_layers(case, seed):
    M, H, Hk, d, P = (case[k] for k in ("M", "H", "Hk", "d", "prefix"))
    linears = _layer_linears(case)
    R, ks, vs = _residual(case, seed).double(), [], []
    for layer in range(case["layers"]):
        mm = lambda j, x: _matmul(case, x, linears[j][1], linears[j][2], seed, layer * 16 + j)
        gains, (K0, V0) = _layer_gains(case, layer, seed), _layer_cache(case, layer, seed)
        h = _norm(R, gains[0])
        q, k, v = (mm(j, h) for j in range(3))
        q, k = _rotate(q, H, d, P), _rotate(k, Hk, d, P)
        a = _attend(q, torch.cat([K0.double(), k]), torch.cat([V0.double(), v]), H, Hk, d)
        R = R + mm(3, a)
        R = R + mm(5, _gate(case["act"], mm(4, _norm(R, gains[1]))))
        ks.append(k)
        vs.append(v)
    return [R, torch.stack(ks), torch.stack(vs)]
