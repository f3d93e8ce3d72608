"""The layer steps around the linears against the oracle: RMSNorm, rotary embedding and
grouped-head attention over a prefix cache plus the chunk's own keys, element by element on
seeded inputs (ragged and maximum sizes, grouped, multi-query and per-head key/value heads,
one or many key splits); then one whole action-expert layer (norm, q/k/v, rotary, attention,
o + residual, norm, GeGLU gate/up, down + residual) recorded as one chain and replayed, each
step checked against the oracle from the bits the GPU produced before it."""
import math

import numpy as np
import pytest
import torch

import oracle
import paper_2607_02501_gb300 as emb
from tests.gpu_util import bits_of, launches
from workloads import activation_bits_np, weight_np

pytestmark = pytest.mark.gpu


def _bf16_dev(a):
    return torch.from_numpy(np.asarray(a, dtype=np.float32)).to(torch.bfloat16).cuda()


def _vals(t):
    return t.float().cpu().numpy().astype(np.float64)


def _check(out, ref, bound, what):
    assert np.isfinite(out).all(), f"{what}: non-finite output"
    bad = np.abs(out - ref) > bound
    assert not bad.any(), (f"{what}: {int(bad.sum())} of {bad.size} outside, first "
                           f"{np.argwhere(bad)[:4].tolist()} err={np.abs(out - ref)[bad][:4]} "
                           f"bound={bound[bad][:4]}")


@pytest.mark.parametrize("M,D", [(1, 1024), (50, 1024), (816, 2048), (3, 8), (7, 4104), (2, 65536)])
def test_rmsnorm_parity(cuda_device, M, D):
    rng = np.random.default_rng(M * 7 + D)
    x = (rng.standard_normal((M, D)) * 3).astype(np.float32)
    g = (1.0 + 0.1 * rng.standard_normal(D)).astype(np.float32)
    y = torch.full((M, D), float("nan"), dtype=torch.bfloat16, device="cuda")
    emb.emb_rmsnorm(torch.from_numpy(x).cuda(), torch.from_numpy(g).cuda(), y, 1e-6)
    torch.cuda.synchronize()
    ref, bound = oracle.rmsnorm_reference(x, g, 1e-6)
    _check(_vals(y), ref, bound, f"rmsnorm M={M} D={D}")


@pytest.mark.parametrize("M,H,d,pos0,base", [(50, 8, 128, 816, 10000.0), (1, 1, 64, 0, 10000.0),
                                             (816, 8, 256, 0, 10000.0), (3, 5, 2, 7, 500.0),
                                             (50, 1, 128, 816, 10000.0), (9, 3, 64, 100000, 1e6)])
def test_rope_parity(cuda_device, M, H, d, pos0, base):
    rng = np.random.default_rng(M + H * 3 + d)
    xb = oracle.bf16_round(rng.standard_normal((M, H * d)) * 2)
    x = _bf16_dev(xb)
    emb.emb_rope(x, H, d, pos0, base)
    torch.cuda.synchronize()
    ref, bound = oracle.rope_reference(xb, H, d, pos0, base)
    _check(_vals(x), ref, bound, f"rope M={M} H={H} d={d} pos0={pos0}")


@pytest.mark.parametrize("M,H,Hk,d", [(50, 8, 1, 128), (7, 3, 5, 64), (1, 1, 1, 2)])
def test_rope_qk_is_two_ropes_in_one_launch(cuda_device, M, H, Hk, d):
    rng = np.random.default_rng(M + H + Hk + d)
    qb = oracle.bf16_round(rng.standard_normal((M, H * d)))
    kb = oracle.bf16_round(rng.standard_normal((M, Hk * d)))
    q1, k1, q2, k2 = _bf16_dev(qb), _bf16_dev(kb), _bf16_dev(qb), _bf16_dev(kb)
    emb.emb_rope_qk(q1, H, k1, Hk, d, 816, 10000.0)
    emb.emb_rope(q2, H, d, 816, 10000.0)
    emb.emb_rope(k2, Hk, d, 816, 10000.0)
    torch.cuda.synchronize()
    assert torch.equal(q1.view(torch.int16), q2.view(torch.int16))
    assert torch.equal(k1.view(torch.int16), k2.view(torch.int16))
    for t, xb, heads in ((q1, qb, H), (k1, kb, Hk)):
        ref, bound = oracle.rope_reference(xb, heads, d, 816, 10000.0)
        _check(_vals(t), ref, bound, f"rope_qk heads={heads}")


# (M, H, Hk, d, n0, n1): the action expert over the 816-token prefix; grouped heads with
# two kv heads and no cache; 16 heads of one kv head (two CTAs of 8 heads); one kv head per
# query head; a single key; many keys at one query (eight key splits); a ragged last tile
ATTN = [(50, 8, 1, 128, 816, 50), (3, 4, 2, 64, 0, 5), (1, 16, 1, 128, 100, 0),
        (7, 8, 8, 64, 130, 1), (2, 1, 1, 128, 1, 0), (1, 8, 1, 128, 4000, 3),
        (5, 2, 1, 64, 63, 66)]


def _attn_inputs(M, H, Hk, d, n0, n1, seed):
    rng = np.random.default_rng(seed)
    r = lambda *s: oracle.bf16_round(rng.standard_normal(s))
    return r(M, H * d), r(n0, Hk * d), r(n0, Hk * d), r(n1, Hk * d), r(n1, Hk * d)


def _run_attention(Qb, K0b, V0b, K1b, V1b, H, Hk, d, scale):
    dev = lambda a: _bf16_dev(a) if a.shape[0] else None
    Q, K0, V0, K1, V1 = _bf16_dev(Qb), dev(K0b), dev(V0b), dev(K1b), dev(V1b)
    O = torch.full((Qb.shape[0], H * d), float("nan"), dtype=torch.bfloat16, device="cuda")
    emb.emb_attention(Q, K0, V0, K1, V1, O, H, Hk, d, scale)
    torch.cuda.synchronize()
    return O


@pytest.mark.parametrize("M,H,Hk,d,n0,n1", ATTN)
def test_attention_parity(cuda_device, M, H, Hk, d, n0, n1):
    ins = _attn_inputs(M, H, Hk, d, n0, n1, M + H + n0 + n1)
    scale = 1.0 / math.sqrt(d)
    O = _run_attention(*ins, H, Hk, d, scale)
    ref, bound = oracle.attention_reference(*ins, H, Hk, d, scale)
    _check(_vals(O), ref, bound, f"attention M={M} H={H} Hk={Hk} d={d} n={n0}+{n1}")
    assert emb.emb_device_status() == emb.EMB_OK


def test_attention_is_deterministic_and_ignores_the_split_of_cache_and_chunk(cuda_device):
    M, H, Hk, d = 50, 8, 1, 128
    Qb, K0b, V0b, K1b, V1b = _attn_inputs(M, H, Hk, d, 816, 50, 3)
    a = _run_attention(Qb, K0b, V0b, K1b, V1b, H, Hk, d, 0.0883883)
    b = _run_attention(Qb, K0b, V0b, K1b, V1b, H, Hk, d, 0.0883883)
    assert torch.equal(a.view(torch.int16), b.view(torch.int16))
    # the same keys given as one list: the same keys in the same order, same tiles and splits
    c = _run_attention(Qb, np.concatenate([K0b, K1b]), np.concatenate([V0b, V1b]),
                       K1b[:0], V1b[:0], H, Hk, d, 0.0883883)
    assert torch.equal(a.view(torch.int16), c.view(torch.int16))


def test_action_expert_layer_recorded(cuda_device):
    """One action-expert layer at M = 50 over an 816-token prefix cache, as one recorded
    chain: h = norm(r); q, k, v = W_qkv h (bf16); rotary on q, k at positions 816..865;
    a = attention(q | prefix k, v + chunk k, v); r += W_o a; h2 = norm(r);
    g = GeGLU(W_gu h2) (interleaved rows); r += W_d g. Checked step by step."""
    M, D, H, Hk, d, F, P = 50, 1024, 8, 1, 128, 4096, 816
    fmt = emb.EMB_Q8_0
    rng = np.random.default_rng(77)
    Ws = {"q": weight_np(H * d, D, 1), "k": weight_np(Hk * d, D, 2), "v": weight_np(Hk * d, D, 3),
          "o": weight_np(D, H * d, 4), "gu": weight_np(2 * F, D, 5), "d": weight_np(D, F, 6)}
    imgs = {k: emb.quantize(fmt, torch.from_numpy(w).cuda()) for k, w in Ws.items()}
    g1 = (1.0 + 0.1 * rng.standard_normal(D)).astype(np.float32)
    g2 = (1.0 + 0.1 * rng.standard_normal(D)).astype(np.float32)
    R0 = (rng.standard_normal((M, D)) * 2).astype(np.float32)
    K0b = oracle.bf16_round(rng.standard_normal((P, Hk * d)))
    V0b = oracle.bf16_round(rng.standard_normal((P, Hk * d)))
    dev = {"g1": torch.from_numpy(g1).cuda(), "g2": torch.from_numpy(g2).cuda(),
           "R": torch.from_numpy(R0.copy()).cuda(), "K0": _bf16_dev(K0b), "V0": _bf16_dev(V0b)}
    bf = lambda *s: torch.full(s, float("nan"), dtype=torch.bfloat16, device="cuda")
    h, q, k, v, a, h2, gg = bf(M, D), bf(M, H * d), bf(M, Hk * d), bf(M, Hk * d), bf(M, H * d), bf(M, D), bf(M, F)
    scale = 1.0 / math.sqrt(d)
    s = torch.cuda.Stream()

    def part1(stream, seq=emb.emb_qlayer_seq, one_rope=False):
        emb.emb_rmsnorm(dev["R"], dev["g1"], h, 1e-6, stream=stream)
        seq([(fmt, imgs["q"], H * d, D, h, q, emb.EMB_EPI_BF16),
                            (fmt, imgs["k"], Hk * d, D, h, k, emb.EMB_EPI_BF16),
                            (fmt, imgs["v"], Hk * d, D, h, v, emb.EMB_EPI_BF16)], M, stream=stream)
        if one_rope:
            emb.emb_rope_qk(q, H, k, Hk, d, P, 10000.0, stream=stream)
        else:
            emb.emb_rope(q, H, d, P, 10000.0, stream=stream)
            emb.emb_rope(k, Hk, d, P, 10000.0, stream=stream)
        emb.emb_attention(q, dev["K0"], dev["V0"], k, v, a, H, Hk, d, scale, stream=stream)
        seq([(fmt, imgs["o"], D, H * d, a, dev["R"], emb.EMB_EPI_ADD)], M, stream=stream)

    def part2(stream, seq=emb.emb_qlayer_seq):
        emb.emb_rmsnorm(dev["R"], dev["g2"], h2, 1e-6, stream=stream)
        seq([(fmt, imgs["gu"], 2 * F, D, h2, gg, emb.EMB_EPI_GEGLU)], M, stream=stream)
        seq([(fmt, imgs["d"], D, F, gg, dev["R"], emb.EMB_EPI_ADD)], M, stream=stream)

    # eager, with the residual kept between the halves, checked step by step against the
    # oracle, each step from the bits the GPU produced before it
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s):
        part1(s)
        s.synchronize()
        R1 = dev["R"].clone()
        part2(s)
    torch.cuda.synchronize()
    assert emb.emb_device_status() == emb.EMB_OK

    ref, bound = oracle.rmsnorm_reference(R0, g1, 1e-6)
    _check(_vals(h), ref, bound, "norm 1")
    hb = bits_of(h)
    Y, B = oracle.qmatmul(fmt, oracle.quantize(fmt, Ws["v"]), hb, Hk * d, D)
    r_, b_ = oracle.epilogue_reference(oracle.EPI_BF16, Y, B)
    _check(_vals(v), r_, b_, "v projection")
    # q and k were rotated in place: the rotation of the projection's bf16 result, where a
    # bf16 input within pre_b of the reference moves each rotated element by at most the
    # sum of its pair's input errors
    half = d // 2
    for name, buf, heads in (("q", q, H), ("k", k, Hk)):
        Y, B = oracle.qmatmul(fmt, oracle.quantize(fmt, Ws[name]), hb, heads * d, D)
        pre, pre_b = oracle.epilogue_reference(oracle.EPI_BF16, Y, B)
        rot, rot_b = oracle.rope_reference(pre, heads, d, P, 10000.0)
        spread = np.empty_like(pre_b)
        for hh in range(heads):
            e = pre_b[:, hh * d:hh * d + half] + pre_b[:, hh * d + half:(hh + 1) * d]
            spread[:, hh * d:hh * d + half] = e
            spread[:, hh * d + half:(hh + 1) * d] = e
        _check(_vals(buf), rot, rot_b + spread * (1 + 2.0 ** -8), f"{name} projection + rotary")
    ref, bound = oracle.attention_reference(_vals(q), K0b, V0b, _vals(k), _vals(v), H, Hk, d, scale)
    _check(_vals(a), ref, bound, "attention")
    Y, B = oracle.qmatmul(fmt, oracle.quantize(fmt, Ws["o"]), bits_of(a), D, H * d)
    r_, b_ = oracle.epilogue_reference(oracle.EPI_ADD, Y, B, R0)
    R1n = R1.cpu().numpy()
    _check(R1n.astype(np.float64), r_, b_, "o + residual")
    ref, bound = oracle.rmsnorm_reference(R1n, g2, 1e-6)
    _check(_vals(h2), ref, bound, "norm 2")
    Y, B = oracle.qmatmul(fmt, oracle.quantize(fmt, Ws["gu"]), bits_of(h2), 2 * F, D)
    r_, b_ = oracle.epilogue_reference(oracle.EPI_GEGLU, Y, B)
    _check(_vals(gg), r_, b_, "gate/up GeGLU")
    Y, B = oracle.qmatmul(fmt, oracle.quantize(fmt, Ws["d"]), bits_of(gg), D, F)
    r_, b_ = oracle.epilogue_reference(oracle.EPI_ADD, Y, B, R1n)
    _check(dev["R"].cpu().numpy().astype(np.float64), r_, b_, "down + residual")

    # the whole layer recorded as one chain, its linears through emb_qlayer_seq_chained (the
    # first launch of each call overlapping the layer step before it): nothing runs while
    # recording, and a replay gives the eager run's bits
    eager = [t.clone() for t in (h, q, k, v, a, h2, gg, dev["R"])]
    dev["R"].copy_(torch.from_numpy(R0))
    for t in (h, q, k, v, a, h2, gg):
        t.fill_(float("nan"))
    torch.cuda.synchronize()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s):
        rec = emb.Recording(s)
        with rec:
            part1(s, emb.emb_qlayer_seq_chained, one_rope=True)
            part2(s, emb.emb_qlayer_seq_chained)
    torch.cuda.synchronize()
    assert torch.isnan(h.float()).all() and torch.equal(dev["R"].cpu(), torch.from_numpy(R0))
    for _ in range(2):
        dev["R"].copy_(torch.from_numpy(R0))
        torch.cuda.synchronize()
        rec.launch(s)
        torch.cuda.synchronize()
        for t, e in zip((h, q, k, v, a, h2, gg, dev["R"]), eager):
            assert torch.equal(t.view(torch.int16) if t.dtype == torch.bfloat16 else t.view(torch.int32),
                               e.view(torch.int16) if e.dtype == torch.bfloat16 else e.view(torch.int32))
    rec.close()
    assert emb.emb_device_status() == emb.EMB_OK


# every kernel and split count of the attention plan, at its edges: keys shared out to the warps
# (one 16-row block exactly and one row more, a last tile that leaves warps without keys, 1 to 16
# splits) and rows shared out (a single tile, 1 to 8 splits, ragged last row block and tile)
ATTN_PLANS = [(1, 32, 32, 128, 280, 1), (16, 1, 1, 64, 0, 33), (17, 1, 1, 128, 5, 60), (16, 8, 1, 128, 816, 16),
              (1, 8, 1, 64, 4090, 3), (300, 8, 8, 64, 0, 300), (120, 8, 2, 128, 1000, 120), (130, 8, 2, 64, 300, 1),
              (816, 8, 1, 128, 0, 700), (400, 16, 4, 64, 500, 400), (280, 32, 32, 128, 0, 65), (17, 1, 1, 64, 5, 90),
              (16, 2, 2, 128, 0, 80), (3, 4, 4, 64, 0, 66), (34, 32, 32, 128, 0, 7), (50, 16, 8, 64, 819, 100)]


@pytest.mark.parametrize("M,H,Hk,d,n,warps,splits", [
    (34, 32, 32, 128, 7, 1, 1), (152, 32, 4, 128, 16, 1, 1), (1, 1, 1, 64, 64, 1, 1), (17, 1, 1, 64, 95, 4, 1),
    (16, 2, 2, 128, 80, 4, 2), (50, 16, 8, 64, 919, 4, 4), (1, 32, 32, 128, 281, 4, 8), (50, 8, 1, 128, 866, 4, 8),
    (1, 8, 1, 128, 4001, 4, 16), (38, 32, 4, 128, 3282, 1, 8), (24, 32, 4, 128, 4000, 1, 16), (816, 8, 1, 128, 816, 1, 2), (280, 32, 32, 128, 280, 1, 1)])
def test_attention_plan(cuda_device, M, H, Hk, d, n, warps, splits):
    """How many warps share a row's keys and how many key splits a call takes on 152 SMs."""
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        return
    t = lambda rows, heads: torch.empty(rows, heads * d, dtype=torch.bfloat16, device="cuda")
    Q, K, V, O = t(M, H), t(n, Hk), t(n, Hk), t(M, H)
    (kernel, args, grid), = launches(lambda: emb.emb_attention(Q, None, None, K, V, O, H, Hk, d, 0.1))
    assert (kernel, args, grid[2]) == ("attention_kernel", (d, warps), splits)


@pytest.mark.parametrize("M,H,Hk,d,n0,n1", ATTN_PLANS)
@pytest.mark.parametrize("gain", [1.0, 30.0])
def test_attention_plans(cuda_device, M, H, Hk, d, n0, n1, gain):
    """gain 30: scores in the hundreds, so one key takes nearly all the weight, the running
    maximum moves between tiles and splits, and most weights underflow to zero."""
    ins = _attn_inputs(M, H, Hk, d, n0, n1, M + H + n0 + n1 + 1)
    scale = gain / math.sqrt(d)
    O = _run_attention(*ins, H, Hk, d, scale)
    ref, bound = oracle.attention_reference(*ins, H, Hk, d, scale)
    _check(_vals(O), ref, bound, f"attention M={M} H={H} Hk={Hk} d={d} n={n0}+{n1} gain={gain}")
    again = _run_attention(*ins, H, Hk, d, scale)
    assert torch.equal(O.view(torch.int16), again.view(torch.int16))
    assert emb.emb_device_status() == emb.EMB_OK


# the pairs per thread follow from head_dim (half divisible by 8, 4, 2, 1) and from the size
@pytest.mark.parametrize("M,H,Hk,d,pos0", [(300, 8, 1, 256, 5), (900, 5, 3, 72, 100), (2000, 7, 2, 20, 1 << 20),
                                           (3000, 3, 1, 6, 7), (1, 2, 1, 16, 0), (40, 4, 4, 512, 100000)])
def test_rope_access_widths(cuda_device, M, H, Hk, d, pos0):
    rng = np.random.default_rng(M + H + d)
    qb = oracle.bf16_round(rng.standard_normal((M, H * d)))
    kb = oracle.bf16_round(rng.standard_normal((M, Hk * d)))
    q, k = _bf16_dev(qb), _bf16_dev(kb)
    emb.emb_rope_qk(q, H, k, Hk, d, pos0, 10000.0)
    torch.cuda.synchronize()
    for t, xb, heads in ((q, qb, H), (k, kb, Hk)):
        ref, bound = oracle.rope_reference(xb, heads, d, pos0, 10000.0)
        _check(_vals(t), ref, bound, f"rope d={d} heads={heads}")


# the thread counts and register shares of the norm: few and many tokens, rows around one, two and
# four groups per thread, rows longer than a CTA keeps in registers, a mostly empty last wave
@pytest.mark.parametrize("M,D", [(152, 8200), (153, 8200), (304, 16392), (760, 4104), (761, 4104), (761, 10248), (1100, 4104),
                                 (3, 512), (304, 520), (305, 1024), (400, 1032), (305, 2048), (320, 4104), (1, 2056),
                                 (2, 4096), (5, 4104), (310, 16384), (2, 16392)])
def test_rmsnorm_thread_counts(cuda_device, M, D):
    rng = np.random.default_rng(M + D)
    x = (rng.standard_normal((M, D)) * 2).astype(np.float32)
    g = (1.0 + 0.1 * rng.standard_normal(D)).astype(np.float32)
    y = torch.full((M, D), float("nan"), dtype=torch.bfloat16, device="cuda")
    emb.emb_rmsnorm(torch.from_numpy(x).cuda(), torch.from_numpy(g).cuda(), y, 1e-6)
    torch.cuda.synchronize()
    ref, bound = oracle.rmsnorm_reference(x, g, 1e-6)
    _check(_vals(y), ref, bound, f"rmsnorm M={M} D={D}")


# (M, H, Hk, d, n, first and end of the keys that are not finite): keys shared out to the warps, one
# split (all keys of a warp: those of the second tile are too few to reach it), two (all of a warp) and more
# (a whole split of eight and of sixteen); rows shared out, one split of one tile (some, one, all) and of more (one
# tile, one key) and two (a whole split); every key
ATTN_NOT_FINITE = [(1, 1, 1, 64, 100, 48, 64), (16, 2, 2, 128, 80, 16, 32), (16, 2, 2, 128, 80, 64, 80),
                   (1, 1, 1, 64, 64, 48, 64), (1, 1, 1, 128, 33, 32, 33), (16, 2, 2, 128, 64, 0, 16),
                   (3, 4, 2, 64, 40, 0, 40), (1, 32, 32, 128, 281, 0, 35), (1, 8, 1, 128, 4001, 250, 501),
                   (300, 8, 8, 64, 300, 64, 128), (300, 8, 8, 64, 300, 299, 300), (816, 8, 1, 128, 700, 0, 350),
                   (816, 8, 1, 128, 700, 350, 700), (300, 8, 8, 64, 300, 0, 300)]


@pytest.mark.parametrize("M,H,Hk,d,n,lo,hi", ATTN_NOT_FINITE)
def test_attention_keys_that_are_not_finite(cuda_device, M, H, Hk, d, n, lo, hi):
    """Keys lo .. hi - 1 of the last key/value head are NaN, give scores of +inf, or of -inf: the
    softmax is NaN, NaN, and the one over the other keys. Other heads keep their bits."""
    Qb, _, _, Kb, Vb = _attn_inputs(M, H, Hk, d, 0, n, M + H + n + lo)
    Qb[:, ::d] = np.abs(Qb[:, ::d]) + 0.5  # the sign of the first product of a score is the key's
    scale = 1.0 / math.sqrt(d)
    none = np.zeros((0, Hk * d))
    first = (H - H // Hk) * d  # output columns of the heads that read the last key/value head
    clean = _run_attention(Qb, none, none, Kb, Vb, H, Hk, d, scale)
    for bad in (np.nan, np.inf, -np.inf):
        K = Kb.copy()
        K[lo:hi, (Hk - 1) * d] = bad
        O = _run_attention(Qb, none, none, K, Vb, H, Hk, d, scale)
        assert torch.equal(O[:, :first].view(torch.int16), clean[:, :first].view(torch.int16)), bad
        got = _vals(O)[:, first:]
        if bad != -np.inf or hi - lo == n:
            assert np.isnan(got).all(), f"{bad}: {int((~np.isnan(got)).sum())} of {got.size} not NaN"
        else:
            keep = np.r_[0:lo, hi:n]
            ref, bound = oracle.attention_reference(Qb, none, none, Kb[keep], Vb[keep], H, Hk, d, scale)
            _check(got, ref[:, first:], bound[:, first:], "keys of score -inf")


# the last position of first-order correction and the first beyond it; then ever larger angles
@pytest.mark.parametrize("M,H,d,pos0,base", [(95, 3, 64, 4000, 1e4), (97, 3, 64, 4000, 1e4), (9, 3, 64, 100000, 1e4),
                                             (700, 4, 256, 1 << 20, 1e4), (5, 2, 128, 16000000, 1e4),
                                             (9, 3, 72, (1 << 24) - 9, 5e5), (4, 2, 6, (1 << 24) - 4, 0.5)])
def test_rope_large_positions(cuda_device, M, H, d, pos0, base):
    """The angle's residual beyond its fp32 value reaches a radian at the largest: cosine and
    sine stay within the oracle's 2^-21, which shows where a rotated element is near zero."""
    rng = np.random.default_rng(pos0 + d)
    xb = oracle.bf16_round(rng.standard_normal((M, H * d)))
    x = _bf16_dev(xb)
    emb.emb_rope(x, H, d, pos0, base)
    torch.cuda.synchronize()
    ref, bound = oracle.rope_reference(xb, H, d, pos0, base)
    _check(_vals(x), ref, bound, f"rope M={M} H={H} d={d} pos0={pos0} base={base}")
