"""emb_qmatmul against the oracle: GEMV (M <= 4 and most layers up to 16), chunk (M = 17..64)
and tcgen05 GEMM paths on shapes spanning several tiles with ragged tails in every dimension."""
import numpy as np
import pytest
import torch

import oracle
import paper_2607_02501_gb300 as emb
from tests.gpu_util import check_close, route, run_case, to_dev_bf16
from workloads import activation_bits_np, weight_np

pytestmark = pytest.mark.gpu

FMTS = [emb.EMB_Q8_0, emb.EMB_Q4_0]

# (1, 130, 16384), (1, 300, 11008) and (1, 1300, 7168) take the Q8_0 register kernel that
# loads a thread's whole row share before the wait (1 to 4 passes, ragged last pass);
# (1, 64, 40960) has rows longer than four passes and streams them one unit ahead.
GEMV_SHAPES = [(1, 1, 32), (1, 8, 64), (1, 136, 96), (1, 256, 2048), (1, 2048, 2048),
               (1, 130, 16384), (1, 300, 11008), (1, 1300, 7168), (1, 64, 40960),
               (1, 4096, 1152), (2, 200, 4608), (3, 129, 1024), (4, 1000, 2080)]

GEMM_SHAPES = [(5, 128, 1024), (7, 136, 96), (16, 8, 32), (49, 256, 2048), (50, 1024, 1024),
               (51, 264, 1152), (64, 384, 256), (127, 128, 1088), (129, 640, 2048),
               (255, 136, 512), (257, 256, 1024), (280, 512, 4096), (500, 300, 320),
               (768, 256, 1152), (816, 384, 2048)]


@pytest.mark.parametrize("fmt", FMTS)
@pytest.mark.parametrize("M,N,K", GEMV_SHAPES)
def test_gemv_parity(cuda_device, fmt, M, N, K):
    Y, Yref, B, _, _ = run_case(fmt, M, N, K, seed=M * 7 + N + K)
    check_close(Y, Yref, B, f"gemv fmt={fmt} M={M} N={N} K={K}")


@pytest.mark.parametrize("fmt", FMTS)
@pytest.mark.parametrize("M,N,K", GEMM_SHAPES)
def test_gemm_parity(cuda_device, fmt, M, N, K):
    Y, Yref, B, _, _ = run_case(fmt, M, N, K, seed=M * 13 + N + K)
    check_close(Y, Yref, B, f"gemm fmt={fmt} M={M} N={N} K={K}")


@pytest.mark.parametrize("M,N,K", [(1, 384, 2048), (3, 384, 2048), (50, 384, 2048),
                                   (280, 384, 2048), (1, 1300, 7168)])
def test_deterministic(cuda_device, M, N, K):
    W = torch.from_numpy(weight_np(N, K, 3)).cuda()
    X = to_dev_bf16(activation_bits_np(M, K, 4))
    for fmt in FMTS:
        img = emb.quantize(fmt, W)
        Y1 = emb.qmatmul(fmt, img, X, N)
        Y2 = emb.qmatmul(fmt, img, X, N)
        torch.cuda.synchronize()
        assert torch.equal(Y1.view(torch.int32), Y2.view(torch.int32))


def test_outliers_q4_0(cuda_device):
    """1% of weights x8 (the 7B configuration's outlier pattern) at both paths."""
    N, K = 512, 4096
    rng = np.random.default_rng(77)
    W = weight_np(N, K, 78)
    W[rng.random((N, K)) < 0.01] *= 8
    for M in (1, 280):
        Xb = activation_bits_np(M, K, 79)
        img = emb.quantize(emb.EMB_Q4_0, torch.from_numpy(W).cuda())
        Y = emb.qmatmul(emb.EMB_Q4_0, img, to_dev_bf16(Xb), N).cpu().numpy()
        Yref, B = oracle.qmatmul(emb.EMB_Q4_0, oracle.quantize(emb.EMB_Q4_0, W), Xb, N, K)
        check_close(Y, Yref, B, f"outliers M={M}")


def test_extreme_activations(cuda_device):
    """bf16 activations spanning 2^-60..2^40 plus zeros of both signs, where a handful of
    terms dominate sum|w x|: the GEMV (exact products) and the split-operand GEMM
    (K < 1024, operand error 2^-16) must meet the bound for such inputs too."""
    from workloads import bf16_bits_np
    rng = np.random.default_rng(91)
    for M, N, K in ((1, 256, 1024), (64, 256, 512)):
        W = weight_np(N, K, 90)
        x = (rng.standard_normal((M, K)) * np.exp2(rng.integers(-60, 40, size=(M, K)))).astype(np.float32)
        x[:, ::17] = 0.0
        x[:, 5::23] = -0.0
        Xb = bf16_bits_np(x)
        for fmt in FMTS:
            img = emb.quantize(fmt, torch.from_numpy(W).cuda())
            Y = emb.qmatmul(fmt, img, to_dev_bf16(Xb), N).cpu().numpy()
            Yref, B = oracle.qmatmul(fmt, oracle.quantize(fmt, W), Xb, N, K)
            check_close(Y, Yref, B, f"extreme x M={M} fmt={fmt}")


def test_y_fully_overwritten(cuda_device):
    N, K = 200, 512
    W = torch.from_numpy(weight_np(N, K, 5)).cuda()
    for M in (1, 70):
        X = to_dev_bf16(activation_bits_np(M, K, 6))
        for fmt in FMTS:
            img = emb.quantize(fmt, W)
            Y0 = emb.qmatmul(fmt, img, X, N)
            Y1 = torch.full((M, N), float("nan"), device="cuda")
            emb.qmatmul(fmt, img, X, N, out=Y1)
            torch.cuda.synchronize()
            assert torch.equal(Y0, Y1)


# Layers of at least 12 MB of packed weights take the staged GEMV at M = 1 (long rows the ring or
# tensor-core kernel, more tokens the tensor-core kernel): ragged row counts (partial last tile), K
# not a multiple of the warps' K slices.
STAGED_SHAPES = [(1, 24593, 1056), (2, 6151, 4128), (3, 6151, 4096), (4, 12301, 2048),
                 (1, 1543, 16384), (1, 12289, 2048), (2, 12289, 2048), (1, 6151, 4096)]


@pytest.mark.parametrize("fmt", FMTS)
@pytest.mark.parametrize("M,N,K", STAGED_SHAPES)
def test_staged_gemv_parity(cuda_device, fmt, M, N, K):
    Y, Yref, B, _, _ = run_case(fmt, M, N, K, seed=M * 5 + N + K)
    check_close(Y, Yref, B, f"staged gemv fmt={fmt} M={M} N={N} K={K}")


@pytest.mark.parametrize("fmt", FMTS)
def test_staged_gemv_fused_group(cuda_device, fmt):
    """Two matrices sharing X in one launch (gate/up): tiles of both in one CTA's run."""
    M, K, Ns = 1, 2048, (12289, 12291)
    Xb = activation_bits_np(M, K, 31)
    X = to_dev_bf16(Xb)
    specs, host = [], []
    for i, N in enumerate(Ns):
        W = weight_np(N, K, 40 + i)
        img = emb.quantize(fmt, torch.from_numpy(W).cuda())
        Y = torch.full((M, N), float("nan"), dtype=torch.float32, device="cuda")
        specs.append((fmt, img, N, K, X, Y))
        host.append(W)
    emb.emb_qlayer_seq(specs, M)
    torch.cuda.synchronize()
    first = [sp[5].clone() for sp in specs]
    emb.emb_qlayer_seq(specs, M)
    torch.cuda.synchronize()
    for a, sp in zip(first, specs):
        assert torch.equal(a.view(torch.int32), sp[5].view(torch.int32))   # deterministic
    for (f, img, N, _, _, Y), W in zip(specs, host):
        Yref, B = oracle.qmatmul(fmt, oracle.quantize(fmt, W), Xb, N, K)
        check_close(Y.cpu().numpy(), Yref, B, f"fused staged N={N}")


# Problems with at least 152 output tiles (128 weight rows x up to 256 tokens): several
# waves of CTAs, tiles that straddle a ragged N, M and K (partial 64-k step and partial
# 256-k raw stage), and a fused pair. Checked element by element against the oracle.
MANY_TILE_SHAPES = [(208, 19461, 1056), (417, 6531, 2080), (816, 4864, 1024), (280, 11008, 1024)]


@pytest.mark.parametrize("fmt", FMTS)
@pytest.mark.parametrize("M,N,K", MANY_TILE_SHAPES)
def test_many_tile_gemm_parity(cuda_device, fmt, M, N, K):
    Y, Yref, B, _, _ = run_case(fmt, M, N, K, seed=M * 3 + N + K)
    check_close(Y, Yref, B, f"many-tile gemm fmt={fmt} M={M} N={N} K={K}")


@pytest.mark.parametrize("fmt", FMTS)
def test_many_tile_gemm_fused_pair_and_determinism(cuda_device, fmt):
    M, K, Ns = 280, 1024, (11008, 11001)   # two token tiles per CTA (as Llama-7B gate/up)
    Xb = activation_bits_np(M, K, 61)
    X = to_dev_bf16(Xb)
    specs, host = [], []
    for i, N in enumerate(Ns):
        W = weight_np(N, K, 62 + i)
        img = emb.quantize(fmt, torch.from_numpy(W).cuda())
        Y = torch.full((M, N), float("nan"), dtype=torch.float32, device="cuda")
        specs.append((fmt, img, N, K, X, Y))
        host.append(W)
    emb.emb_qlayer_seq(specs, M)
    torch.cuda.synchronize()
    first = [sp[5].clone() for sp in specs]
    emb.emb_qlayer_seq(specs, M)
    torch.cuda.synchronize()
    for a, sp in zip(first, specs):
        assert torch.equal(a.view(torch.int32), sp[5].view(torch.int32))
    for (f, img, N, _, _, Y), W in zip(specs, host):
        Yref, B = oracle.qmatmul(fmt, oracle.quantize(fmt, W), Xb, N, K)
        check_close(Y.cpu().numpy(), Yref, B, f"fused many-tile N={N}")


# Wide layers at 280..561 tokens where one CTA computes two token tiles from each
# dequantised weight tile: several waves, ragged N, the last token tile partly past M
# (420 = 2 x 224 - 28 with the widest pair tiles, 561 = 4 x 144 - 15), K not a multiple
# of the 256-k raw stage.
PAIR_SHAPES = [(420, 30000, 1024), (561, 19000, 1056), (300, 40000, 1024), (280, 23000, 2080)]


@pytest.mark.parametrize("fmt", FMTS)
@pytest.mark.parametrize("M,N,K", PAIR_SHAPES)
def test_token_pair_gemm_parity(cuda_device, fmt, M, N, K):
    Y, Yref, B, _, _ = run_case(fmt, M, N, K, seed=M * 13 + N + K)
    check_close(Y, Yref, B, f"token-pair gemm fmt={fmt} M={M} N={N} K={K}")


# 5..64 tokens with K >= 1024 (the action-chunk range): ragged token tails, ragged N, K
# that is not a multiple of the 64-k step or the 256-k raw stage, and long rows.
ACTION_CHUNK_SHAPES = [(5, 136, 1024), (8, 200, 1056), (9, 77, 2048), (16, 300, 1024), (17, 129, 1056),
                   (33, 64, 4128), (50, 1000, 1024), (50, 130, 4096), (64, 257, 2080)]


@pytest.mark.parametrize("fmt", FMTS)
@pytest.mark.parametrize("M,N,K", ACTION_CHUNK_SHAPES)
def test_action_chunk_parity(cuda_device, fmt, M, N, K):
    Y, Yref, B, _, _ = run_case(fmt, M, N, K, seed=M * 11 + N + K)
    check_close(Y, Yref, B, f"action-chunk fmt={fmt} M={M} N={N} K={K}")


@pytest.mark.parametrize("fmt", FMTS)
def test_action_chunk_fused_group_and_determinism(cuda_device, fmt):
    M, K, Ns = 50, 1024, (1024, 128, 128)
    Xb = activation_bits_np(M, K, 71)
    X = to_dev_bf16(Xb)
    specs, host = [], []
    for i, N in enumerate(Ns):
        W = weight_np(N, K, 72 + i)
        img = emb.quantize(fmt, torch.from_numpy(W).cuda())
        Y = torch.full((M, N), float("nan"), dtype=torch.float32, device="cuda")
        specs.append((fmt, img, N, K, X, Y))
        host.append(W)
    emb.emb_qlayer_seq(specs, M)
    torch.cuda.synchronize()
    first = [sp[5].clone() for sp in specs]
    emb.emb_qlayer_seq(specs, M)
    torch.cuda.synchronize()
    for a, sp in zip(first, specs):
        assert torch.equal(a.view(torch.int32), sp[5].view(torch.int32))
    for (f, img, N, _, _, Y), W in zip(specs, host):
        Yref, B = oracle.qmatmul(fmt, oracle.quantize(fmt, W), Xb, N, K)
        check_close(Y.cpu().numpy(), Yref, B, f"fused action-chunk N={N}")


def test_precise_operand_flag_few_dominant_terms(cuda_device):
    """The tensor-core GEMM at K >= 1024 stages bf16(w') (relative error <= 2^-8 per
    weight, bf16's unit roundoff): with activations where a single term dominates sum|w x|
    (one-hot rows), the output error reaches that rounding and so exceeds the 1e-3 * S
    bound for some outputs; the documented (2^-8 + 2^-12) * S + 1e-6 bound holds. With EMB_PRECISE_OPERAND the same layer runs
    with the two-operand weights and meets 1e-3 * S + 1e-6 everywhere."""
    fmt, M, N, K = emb.EMB_Q8_0, 64, 256, 2048
    W = weight_np(N, K, 95)
    img = emb.quantize(fmt, torch.from_numpy(W).cuda())
    ks = (np.arange(M) * 37) % K
    Xb = np.zeros((M, K), dtype=np.uint16)
    Xb[np.arange(M), ks] = 0x3F80                       # e_k: one term per output
    Xb[:, (ks + 1) % K] = 0x3380                        # plus one 2^-24 term (negligible)
    X = to_dev_bf16(Xb)
    Yref, B = oracle.qmatmul(fmt, oracle.quantize(fmt, W), Xb, N, K)
    S = (B - 1e-6) / 1e-3
    Yd = torch.empty(M, N, device="cuda")
    Yp = torch.empty(M, N, device="cuda")
    emb.emb_qlayer_seq([(fmt, img, N, K, X, Yd)], M)
    emb.emb_qlayer_seq([(fmt, img, N, K, X, Yp, emb.EMB_EPI_F32 | emb.EMB_PRECISE_OPERAND)], M)
    torch.cuda.synchronize()
    err_d = np.abs(Yd.cpu().numpy().astype(np.float64) - Yref)
    assert (err_d <= (2.0 ** -8 + 2.0 ** -12) * S + 1e-6).all()
    assert (err_d > B).any()            # the single-operand form is not within 1e-3 here
    check_close(Yp.cpu().numpy(), Yref, B, "EMB_PRECISE_OPERAND")


# the tensor-core GEMV's edges: a single row, row tiles one short and one over, a 32-weight row, an
# odd block count, a ragged last 256-k chunk, one and several chunks per warp, sixteen warps per CTA
# (long rows, few tiles), several row tiles per CTA; eight tokens, and both ends of the
# sixteen-token variant (the one-token shapes take the other kernels: below are those that do not)
TC_SHAPES = [(3, 1, 64), (3, 15, 32), (4, 17, 96), (6, 33, 352), (8, 300, 2048), (9, 16, 2080), (16, 31, 256),
             (13, 257, 4160), (1, 100, 4096), (1, 5000, 4128), (8, 70, 16384), (16, 2433, 5056), (7, 9000, 1088)]


@pytest.mark.parametrize("fmt", FMTS + [emb.EMB_Q6_0])
@pytest.mark.parametrize("M,N,K", TC_SHAPES)
def test_tensor_core_gemv_has_exact_products(cuda_device, fmt, M, N, K):
    """Products of codes and activations are exact, so only fp32 sums round: 32 products per block
    (2^-23 of their magnitudes each, as tensor-core sums may truncate), the scaled block sums and
    the warps' sums, K / 32 + 32 additions of 2^-24: no bf16 rounding of a weight (2^-9) fits."""
    if fmt == emb.EMB_Q6_0 and K % 64:
        K += 32
    W = weight_np(N, K, M + N + K)
    Xb = activation_bits_np(M, K, M + N + K + 1)
    img = emb.quantize(fmt, torch.from_numpy(W).cuda())
    X = to_dev_bf16(Xb)
    Yref, B = oracle.qmatmul(fmt, oracle.quantize(fmt, W), Xb, N, K)
    S = (B - 1e-6) / 1e-3
    bound = (32 * 2.0 ** -23 + (K // 32 + 32) * 2.0 ** -24) * S + 1e-9
    Y = torch.full((M, N), float("nan"), device="cuda")
    emb.emb_qmatmul(fmt, img, X, Y, M, N, K)
    again = torch.full_like(Y, float("nan"))
    emb.emb_qmatmul(fmt, img, X, again, M, N, K)
    torch.cuda.synchronize()
    assert torch.equal(Y.view(torch.int32), again.view(torch.int32))
    err = np.abs(Y.cpu().numpy().astype(np.float64) - Yref)
    assert (err <= bound).all(), f"{int((err > bound).sum())} of {err.size} outside, worst {float((err / bound).max()):.2f}"
    # a gated and an adding epilogue of the same sums
    if N % 2 == 0:
        H = torch.full((M, N // 2), float("nan"), dtype=torch.bfloat16, device="cuda")
        emb.emb_qlayer_seq([(fmt, img, N, K, X, H, emb.EMB_EPI_SWIGLU)], M)
        ref, b = oracle.epilogue_reference(oracle.EPI_SWIGLU, Yref, bound)
        assert (np.abs(H.float().cpu().numpy().astype(np.float64) - ref) <= b).all()
    R = torch.ones(M, N, device="cuda")
    emb.emb_qlayer_seq([(fmt, img, N, K, X, R, emb.EMB_EPI_ADD)], M)
    assert torch.equal(R, torch.ones_like(R) + Y)
    assert emb.emb_device_status() == emb.EMB_OK


# the tensor-core GEMV at one token (long rows of Q4_0 and Q6_0): sixteen warps and few rows, eight
# warps in one round with ragged last tiles, several rounds; with compensated totals from K = 6208
# (eight warps) and 16448 (sixteen) on
TC_ONE_TOKEN = [(emb.EMB_Q4_0, 1000, 4128), (emb.EMB_Q6_0, 1000, 4160), (emb.EMB_Q4_0, 4096, 4096),
                (emb.EMB_Q6_0, 4100, 4096), (emb.EMB_Q4_0, 4090, 11008), (emb.EMB_Q6_0, 4096, 11008),
                (emb.EMB_Q4_0, 6144, 5120), (emb.EMB_Q6_0, 6144, 5120), (emb.EMB_Q4_0, 1100, 16448)]


@pytest.mark.parametrize("fmt,N,K", TC_ONE_TOKEN)
def test_tensor_core_gemv_at_one_token(cuda_device, fmt, N, K):
    assert route(fmt, 1, N, K)[0] == "gemv_tc_kernel"
    test_tensor_core_gemv_has_exact_products(cuda_device, fmt, 1, N, K)


# its two-warp instance: many tiles of short rows, one to six, nine and ten chunks (ragged, fewer than two),
# a ragged last tile, just past the least number of tiles, several tiles per CTA
TC_TWO_WARPS = [(2, 4881, 96), (4, 5003, 512), (3, 14610, 544), (4, 14600, 1536), (2, 32768, 1280),
                (3, 14610, 2336)]


@pytest.mark.parametrize("fmt", FMTS + [emb.EMB_Q6_0])
@pytest.mark.parametrize("M,N,K", TC_TWO_WARPS)
def test_tensor_core_gemv_two_warps(cuda_device, fmt, M, N, K):
    if fmt == emb.EMB_Q6_0 and K % 64:
        K += 32
    kernel, args, _ = route(fmt, M, N, K)
    if M > 2:  # (two tokens of short rows mostly take the register kernel)
        assert kernel == "gemv_tc_kernel" and args[2] == 2
    test_tensor_core_gemv_has_exact_products(cuda_device, fmt, M, N, K)


@pytest.mark.parametrize("fmt", FMTS + [emb.EMB_Q6_0])
def test_shapes_take_the_kernels_they_are_named_for(cuda_device, fmt):
    k64 = lambda K: K + 32 if fmt == emb.EMB_Q6_0 and K % 64 else K
    for M, N, K in TC_SHAPES:
        if M > 3:
            assert route(fmt, M, N, k64(K))[0] == "gemv_tc_kernel", (M, N, K)
    for M, N, K in CHUNK_SHAPES:
        # not: few long rows (the GEMM's K splits), a second round of a few CTAs
        other = (M, N, K) in ((64, 130, 16384), (64, 33, 4160), (50, 5000, 1280))
        assert route(fmt, M, N, k64(K))[0] == ("gemm_tc_kernel" if other else "gemm_chunk_kernel"), (M, N, K)
    for M, N, K in SHORT_ROW_SHAPES:
        assert route(fmt, M, N, k64(K))[0] == "gemm_tc_kernel", (M, N, K)
    for N, K in LONG_ROW_SHAPES:
        for M in (2, 4):
            if N > 512:  # two tokens of few row tiles, and four of very few: the register kernel
                assert route(fmt, M, N, K)[0] == "gemv_tc_kernel", (M, N, K)


# the chunk kernel's edges: 17, 32, 33 and 64 tokens; one row tile, one short and one over, several
# per CTA; K of four chunks exactly, with a ragged last one, odd block counts
CHUNK_SHAPES = [(17, 16, 1024), (32, 15, 2048), (33, 300, 1056), (50, 1280, 1024), (64, 33, 4160), (50, 5000, 1280),
                (24, 6000, 1120), (64, 130, 16384), (40, 2048, 2080)]
# long rows: the longest of a layer of the workloads, a ragged last tile and chunk, one token group; several
# row tiles per CTA with one token group and with both in a CTA; 64 tokens and one row more than two tiles
CHUNK_MORE_SHAPES = [(50, 2048, 16384), (33, 1930, 8256), (20, 4000, 11008), (24, 7000, 1120), (50, 9500, 1024),
                     (64, 33, 2080)]


@pytest.mark.parametrize("fmt", FMTS + [emb.EMB_Q6_0])
@pytest.mark.parametrize("M,N,K", CHUNK_SHAPES)
def test_chunk_gemm_is_the_bf16_operand_product(cuda_device, fmt, M, N, K):
    """Y against the fp64 product of the bf16-rounded weights (the operand of every GEMM path at
    K >= 1024): only fp32 sums round, K + 64 additions of up to 2^-23 of the terms' magnitudes
    (tensor-core sums may truncate)."""
    if fmt == emb.EMB_Q6_0 and K % 64:
        K += 32
    W = weight_np(N, K, M + N + K)
    Xb = activation_bits_np(M, K, M + N + K + 1)
    ref_img = oracle.quantize(fmt, W)
    img = emb.quantize(fmt, torch.from_numpy(W).cuda())
    w = (oracle.dequant_bf16(fmt, ref_img, N, K).astype(np.uint32) << 16).view(np.float32).astype(np.float64)
    x = (Xb.astype(np.uint32) << 16).view(np.float32).astype(np.float64)
    Yref, S = x @ w.T, np.abs(x) @ np.abs(w).T
    bound = (K + 64) * 2.0 ** -23 * S + 1e-9
    X = to_dev_bf16(Xb)
    Y = torch.full((M, N), float("nan"), device="cuda")
    emb.emb_qmatmul(fmt, img, X, Y, M, N, K)
    again = torch.full_like(Y, float("nan"))
    emb.emb_qmatmul(fmt, img, X, again, M, N, K)
    assert torch.equal(Y.view(torch.int32), again.view(torch.int32))
    err = np.abs(Y.cpu().numpy().astype(np.float64) - Yref)
    assert (err <= bound).all(), f"{int((err > bound).sum())} of {err.size} outside, worst {float((err / bound).max()):.2f}"
    R = torch.ones(M, N, device="cuda")
    emb.emb_qlayer_seq([(fmt, img, N, K, X, R, emb.EMB_EPI_ADD)], M)
    assert torch.equal(R, torch.ones_like(R) + Y)
    H = torch.full((M, N), float("nan"), dtype=torch.bfloat16, device="cuda")
    emb.emb_qlayer_seq([(fmt, img, N, K, X, H, emb.EMB_EPI_BF16)], M)
    assert torch.equal(H, Y.to(torch.bfloat16))
    if N % 2 == 0:
        G = torch.full((M, N // 2), float("nan"), dtype=torch.bfloat16, device="cuda")
        emb.emb_qlayer_seq([(fmt, img, N, K, X, G, emb.EMB_EPI_GEGLU)], M)
        ref, b = oracle.epilogue_reference(oracle.EPI_GEGLU, Yref, bound)
        assert (np.abs(G.float().cpu().numpy().astype(np.float64) - ref) <= b).all()
    assert emb.emb_device_status() == emb.EMB_OK


@pytest.mark.parametrize("fmt", FMTS + [emb.EMB_Q6_0])
@pytest.mark.parametrize("M,N,K", CHUNK_MORE_SHAPES)
def test_chunk_gemm_long_rows_and_rounds(cuda_device, fmt, M, N, K):
    if fmt == emb.EMB_Q6_0 and K % 64:
        K += 32
    assert route(fmt, M, N, K)[0] == "gemm_chunk_kernel"
    test_chunk_gemm_is_the_bf16_operand_product(cuda_device, fmt, M, N, K)


# short rows whose launch leaves SMs idle take more token tiles of 96 and more tokens instead of a K
# split: tiles that end exactly at M and ragged ones (97, 193, 577, 1030, 1537), the last one row short
# of or one over a tile, a K of 4.1 raw stages; long rows of few tiles keep the split (97 x 300)
SHORT_ROW_SHAPES = [(768, 1152, 1152), (577, 1000, 1056), (97, 300, 2112), (193, 130, 1056), (1030, 1100, 1088),
                    (1537, 900, 1312), (128, 8192, 1024), (65, 40, 1024)]


@pytest.mark.parametrize("fmt", FMTS + [emb.EMB_Q6_0])
@pytest.mark.parametrize("M,N,K", SHORT_ROW_SHAPES)
def test_short_row_gemm_is_the_bf16_operand_product(cuda_device, fmt, M, N, K):
    test_chunk_gemm_is_the_bf16_operand_product(cuda_device, fmt, M, N, K)


# the tensor-core GEMV's compensated totals: the last K without and the first with them at eight warps
# (tiles of two CTAs per SM) and sixteen (one tile per SM), ragged last chunks, few rows
LONG_ROW_SHAPES = [(4900, 6144), (4900, 6208), (4096, 11008), (300, 16384), (300, 16448), (33, 32768), (2600, 14336)]


@pytest.mark.parametrize("fmt", FMTS + [emb.EMB_Q6_0])
@pytest.mark.parametrize("M", [2, 4])
@pytest.mark.parametrize("N,K", LONG_ROW_SHAPES)
def test_long_row_gemv_error_does_not_grow_with_k(cuda_device, fmt, M, N, K):
    """Exact products; the roundings on a term's way are those of its MMA (16 terms, truncated: 17),
    the two MMAs' sum, up to eight scaled additions, two levels within the chunk, the total and the warps'
    levels (three with a total, four without): 32 of 2^-23 of the magnitudes, whatever K. An infinite
    activation gives the product's own infinities and NaNs in its token and none elsewhere."""
    W = weight_np(N, K, M + N + K)
    Xb = activation_bits_np(M, K, M + N + K + 1)
    img_ref = oracle.quantize(fmt, W)
    w = oracle.dequant_f32(fmt, img_ref, N, K).astype(np.float64)
    x = (Xb.astype(np.uint32) << 16).view(np.float32).astype(np.float64)
    img, X = emb.quantize(fmt, torch.from_numpy(W).cuda()), to_dev_bf16(Xb)
    Y = torch.full((M, N), float("nan"), device="cuda")
    emb.emb_qmatmul(fmt, img, X, Y, M, N, K)
    again = torch.full_like(Y, float("nan"))
    emb.emb_qmatmul(fmt, img, X, again, M, N, K)
    assert torch.equal(Y.view(torch.int32), again.view(torch.int32))
    err, bound = np.abs(Y.cpu().numpy() - x @ w.T), 32 * 2.0 ** -23 * (np.abs(x) @ np.abs(w).T) + 1e-12
    assert (err <= bound).all(), f"worst {float((err / bound).max()):.2f} of the bound"
    X[M - 1, 7] = float("inf")
    emb.emb_qmatmul(fmt, img, X, again, M, N, K)
    assert torch.equal(again[: M - 1].view(torch.int32), Y[: M - 1].view(torch.int32))
    with np.errstate(invalid="ignore"):
        want = np.where(w[:, 7] == 0, np.nan, np.sign(w[:, 7]) * np.inf)
    assert np.array_equal(again[M - 1].cpu().numpy(), want.astype(np.float32), equal_nan=True)
    assert emb.emb_device_status() == emb.EMB_OK


@pytest.mark.parametrize("fmt,N,K", [(emb.EMB_Q4_0, 4090, 11008), (emb.EMB_Q6_0, 4096, 11008), (emb.EMB_Q4_0, 4864, 14336),
                                     (emb.EMB_Q4_0, 1100, 16448)])
def test_long_row_gemv_error_at_one_token(cuda_device, fmt, N, K):
    kernel, args, _ = route(fmt, 1, N, K)
    assert kernel == "gemv_tc_kernel" and args[3] == 1  # compensated totals
    test_long_row_gemv_error_does_not_grow_with_k(cuda_device, fmt, 1, N, K)


@pytest.mark.parametrize("fmt,M,N,K,splits", [(emb.EMB_Q4_0, 193, 2432, 8448, 4), (emb.EMB_Q4_0, 481, 2373, 6592, 4),
                                              (emb.EMB_Q6_0, 151, 4864, 8960, 4), (emb.EMB_Q8_0, 287, 893, 12256, 8)])
def test_k_splits_are_clusters_that_run_at_once(cuda_device, fmt, M, N, K, splits):
    """A cluster stays within a part of the chip, so fewer than SMs / splits run at once: 36 of four
    and 15 of eight on 152 SMs. Nineteen row tiles and two token tiles, or twice the row tiles, are no
    wave of four splits; seven row tiles and two token tiles are one of eight."""
    kernel, _, grid = route(fmt, M, N, K)
    assert kernel == "gemm_tc_kernel"
    if torch.cuda.get_device_properties(0).multi_processor_count == 152:
        assert (grid[2] == 8) == (splits == 8) and grid[0] * grid[1] <= {8: 15, 4: 36, 2: 76, 1: 152}[grid[2]]
    Y, Yref, B, _, _ = run_case(fmt, M, N, K, seed=M + N + K)
    check_close(Y, Yref, B, f"fmt={fmt} M={M} N={N} K={K}")


# lines of the tensor-core GEMV's rule: few row tiles at two to four tokens (on either side), a last round
# that is mostly empty at two, one exactly full wave of the register kernel at one token and one row
# tile more, short rows beyond one round and two rounds of tiles at up to eight tokens and more
@pytest.mark.parametrize("fmt,M,N,K,kernel", [
    (emb.EMB_Q8_0, 2, 912, 8192, "gemv_kernel"), (emb.EMB_Q8_0, 2, 913, 8192, "gemv_tc_kernel"),
    (emb.EMB_Q8_0, 3, 640, 6144, "gemv_kernel"), (emb.EMB_Q8_0, 4, 300, 6144, "gemv_tc_kernel"),
    (emb.EMB_Q4_0, 2, 160, 2048, "gemv_kernel"), (emb.EMB_Q4_0, 3, 129, 4096, "gemv_tc_kernel"),
    (emb.EMB_Q6_0, 4, 112, 4096, "gemv_kernel"), (emb.EMB_Q6_0, 3, 513, 576, "gemv_tc_kernel"),
    (emb.EMB_Q8_0, 2, 4999, 8704, "gemv_kernel"), (emb.EMB_Q4_0, 1, 1216, 5120, "gemv_kernel"),
    (emb.EMB_Q4_0, 1, 1217, 5120, "gemv_tc_kernel"), (emb.EMB_Q4_0, 1, 13000, 4160, "gemv_tc_kernel"),
    (emb.EMB_Q8_0, 8, 4865, 128, "gemm_tc_kernel"), (emb.EMB_Q4_0, 8, 4864, 128, "gemv_tc_kernel"),
    (emb.EMB_Q6_0, 9, 4865, 256, "gemm_tc_kernel"), (emb.EMB_Q8_0, 16, 9729, 512, "gemm_tc_kernel"),
    (emb.EMB_Q4_0, 6, 9729, 256, "gemm_tc_kernel"), (emb.EMB_Q4_0, 6, 9728, 256, "gemv_tc_kernel")])
def test_tensor_core_gemv_rule(cuda_device, fmt, M, N, K, kernel):
    assert route(fmt, M, N, K)[0] == kernel
    Y, Yref, B, _, _ = run_case(fmt, M, N, K, seed=M + N + K)
    check_close(Y, Yref, B, f"fmt={fmt} M={M} N={N} K={K}")


# gated layers, two rows per CTA of the register kernel, have lines of their own
@pytest.mark.parametrize("fmt,M,N,K,kernel", [
    (emb.EMB_Q6_0, 2, 512, 8192, "gemv_kernel"), (emb.EMB_Q6_0, 2, 514, 8192, "gemv_tc_kernel"),
    (emb.EMB_Q8_0, 4, 512, 4096, "gemv_kernel"), (emb.EMB_Q8_0, 3, 130, 1024, "gemv_tc_kernel"),
    (emb.EMB_Q4_0, 3, 160, 2080, "gemv_kernel"), (emb.EMB_Q4_0, 3, 162, 2080, "gemv_tc_kernel")])
def test_tensor_core_gemv_rule_gated(cuda_device, fmt, M, N, K, kernel):
    assert route(fmt, M, N, K, emb.EMB_EPI_SWIGLU)[0] == kernel
    W, Xb = weight_np(N, K, M + N + K), activation_bits_np(M, K, M + N + K + 1)
    img, Y = emb.quantize(fmt, torch.from_numpy(W).cuda()), torch.empty(M, N // 2, dtype=torch.bfloat16, device="cuda")
    emb.emb_qlayer_seq([(fmt, img, N, K, to_dev_bf16(Xb), Y, emb.EMB_EPI_SWIGLU)], M)
    ref, bound = oracle.epilogue_reference(oracle.EPI_SWIGLU, *oracle.qmatmul(fmt, oracle.quantize(fmt, W), Xb, N, K))
    assert (np.abs(Y.float().cpu().numpy().astype(np.float64) - ref) <= bound).all()
