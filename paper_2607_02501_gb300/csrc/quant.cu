// Quantisation (offline packing) and test-support dequantisation kernels.
//
// Formats: the library's definitions of the paper's 8-, 6- and 4-bit weight
// configurations (Section 4, Table 3), written out in include/emb_qmm.h.
// Arithmetic is IEEE fp32 with explicit round-to-nearest intrinsics so that the
// packed bytes are reproducible bit for bit: max|w| (or the signed extreme),
// one correctly rounded division, one fp16 rounding of the scale, one correctly
// rounded division per weight and roundf (half away from zero).
#include <algorithm>

#include "common.cuh"

namespace emb {
namespace {

constexpr unsigned kFull = 0xffffffffu;

// The packing kernels read 4 bytes per weight and write 0.56 to 1.06, so HBM bounds them as
// long as enough loads are in flight and the arithmetic stays near a dozen instructions per
// weight. A warp owns 8 * LOADS = 32 consecutive blocks (4 KB of W, contiguous because rows
// are whole blocks): eight 16-byte loads per lane, all issued before the first use. Four lanes
// share a block, lane s of them holding weights 4s .. 4s+3 and 16+4s .. 16+4s+3: the block's
// extreme takes two shuffles, the per-block divisions are spread over eight weights a lane, and
// a Q4_0 lane holds both nibbles of its four bytes. Codes leave as 32-bit words (Q4_0: 128
// contiguous bytes per warp store), the 32 scales as one 16-bit store per lane.
// Measured (GB300, 0.84 of the copy bandwidth): Q4_0 22016 x 4096 72.0 us (5.7 TB/s) against
// 362.8 for one weight per lane behind a memset of the whole image; Q8_0 8000 x 4096 28.7 (was
// 122), Q6_0 8000 x 4128 32.8 (was 165). Eight lanes per block instead of four: 95.8.
// Matrices of up to 38912 blocks, which would leave SMs without a CTA, go 8 blocks to a warp (LOADS = 1):
// Q4_0 508 x 32 3.9 -> 2.2 (2.7 with the memset), 1216 x 1024 3.3 -> 2.7.
constexpr int kPackThreads = 256;

// roundf(w / d) clamped to [lo, hi] for the four weights of v, plus `bias`, one per byte.
// The quotient is first taken as w * (1 / d), within 2^-23 |w / d| < 3e-5 of the correctly
// rounded one wherever it is not clamped; the nearest integer (ties to even, by adding
// 1.5 * 2^23) is then the one of the true quotient unless that lies within kTieSlack of a
// half, where the division itself and roundf (half away from zero) decide.
constexpr float kTieSlack = 1e-4f;
__device__ __forceinline__ uint32_t pack4(const float4 v, float d, float r, float lo, float hi, uint32_t bias) {
    const float magic = 12582912.0f;  // 1.5 * 2^23
    const float w[4] = {v.x, v.y, v.z, v.w};
    uint32_t q[4];
    float off = 0.0f;  // largest distance from the nearest integer
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const float t = fminf(fmaxf(__fmul_rn(w[e], r), lo), hi);
        const float g = __fadd_rn(t, magic);
        off = fmaxf(off, fabsf(__fsub_rn(t, __fsub_rn(g, magic))));
        q[e] = __float_as_uint(g);
    }
    if (off > 0.5f - kTieSlack) {
#pragma unroll
        for (int e = 0; e < 4; ++e)
            q[e] = uint32_t(int(fminf(fmaxf(roundf(__fdiv_rn(w[e], d)), lo), hi)));
    }
    // the low byte of each (two's complement), then the bias without carries between bytes:
    // codes and biases add up to at most 63 for the biased formats, whose codes are >= -bias
    const uint32_t p = __byte_perm(__byte_perm(q[0], q[1], 0x0040), __byte_perm(q[2], q[3], 0x0040), 0x5410);
    return bias ? ((p ^ 0x80808080u) - (0x80808080u - bias)) : p;
}

// Bits of the largest magnitude among four weights (ordered as unsigned integers).
__device__ __forceinline__ uint32_t abs_max(const float4 v) {
    return max(max(__float_as_uint(fabsf(v.x)), __float_as_uint(fabsf(v.y))),
               max(__float_as_uint(fabsf(v.z)), __float_as_uint(fabsf(v.w))));
}
// The first of four weights whose magnitude has the bits `top` (the last one if none has).
__device__ __forceinline__ float first_of(const float4 v, uint32_t top) {
    return __float_as_uint(fabsf(v.x)) == top   ? v.x
           : __float_as_uint(fabsf(v.y)) == top ? v.y
           : __float_as_uint(fabsf(v.z)) == top ? v.z
                                                : v.w;
}

template <int FMT, int LOADS>
__global__ void __launch_bounds__(kPackThreads) pack_kernel(const float* __restrict__ W, int64_t N, int64_t K,
                                                            uint8_t* __restrict__ codes,
                                                            uint8_t* __restrict__ high,
                                                            __half* __restrict__ scales, const Layout L) {
    constexpr float kLo = FMT == EMB_Q8_0 ? -127.0f : FMT == EMB_Q4_0 ? -8.0f : -32.0f;
    constexpr float kHi = FMT == EMB_Q8_0 ? 127.0f : FMT == EMB_Q4_0 ? 7.0f : 31.0f;
    constexpr float kDiv = FMT == EMB_Q8_0 ? 127.0f : kLo;
    constexpr uint32_t kBias = FMT == EMB_Q8_0 ? 0u : FMT == EMB_Q4_0 ? 0x08080808u : 0x20202020u;
    constexpr int kBlocks = 8 * LOADS;  // per warp, LOADS pairs of loads per lane
    const int lane = threadIdx.x & 31, sub = lane & 3;
    const int64_t nb = K / kQBlock, total = N * nb;
    const int64_t thread = int64_t(blockIdx.x) * kPackThreads + threadIdx.x;
    const int64_t b0 = (thread >> 5) * kBlocks;  // first block of this warp
    // padding bytes of the image (part of the format): between the planes, after each scale row
    if (blockIdx.x == 0) {
        const int64_t gap0 = L.codes_bytes, gap0_end = FMT == EMB_Q6_0 ? L.high_off : L.scales_off;
        for (int64_t i = gap0 + threadIdx.x; i < gap0_end; i += kPackThreads) codes[i] = 0;
        if constexpr (FMT == EMB_Q6_0)
            for (int64_t i = L.high_off + N * K / 4 + threadIdx.x; i < L.scales_off; i += kPackThreads) codes[i] = 0;
    }
    const int pad = int(L.ldS - nb);
    if (pad)
        for (int64_t i = thread; i < N * pad; i += int64_t(gridDim.x) * kPackThreads)
            scales[(i / pad) * L.ldS + nb + i % pad] = __ushort_as_half(0);
    if (b0 >= total) return;

    float4 v[LOADS][2];
#pragma unroll
    for (int i = 0; i < LOADS; ++i) {
        const int64_t b = b0 + 8 * i + (lane >> 2);
        const float4* src = reinterpret_cast<const float4*>(W + b * kQBlock) + sub;
        v[i][0] = b < total ? __ldcs(src) : make_float4(0, 0, 0, 0);
        v[i][1] = b < total ? __ldcs(src + 4) : make_float4(0, 0, 0, 0);
    }
    __half mine = __ushort_as_half(0);  // the scale of block b0 + lane
#pragma unroll
    for (int i = 0; i < LOADS; ++i) {
        const float4 lo = v[i][0], hi = v[i][1];
        const uint32_t top_lo = abs_max(lo), top_hi = abs_max(hi);
        uint32_t top = max(top_lo, top_hi);
        top = max(top, __shfl_xor_sync(kFull, top, 1));
        top = max(top, __shfl_xor_sync(kFull, top, 2));
        float num = __uint_as_float(top);
        if constexpr (FMT != EMB_Q8_0) {
            // the signed weight of largest magnitude, lowest index on ties (every lane's first
            // four weights come before any lane's last four); +0 for a zero block
            const uint32_t in_lo = __ballot_sync(kFull, top_lo == top) >> (lane & 28) & 0xFu;
            const uint32_t in_hi = __ballot_sync(kFull, top_hi == top) >> (lane & 28) & 0xFu;
            const float first = first_of(in_lo ? lo : hi, top);
            const float extreme = __shfl_sync(kFull, first, (lane & 28) + __ffs(in_lo ? in_lo : in_hi) - 1);
            num = top == 0u ? 0.0f : extreme;
        }
        const __half dh = __float2half_rn(__fdiv_rn(num, kDiv));
        const float d = __half2float(dh);
        uint32_t q_lo = kBias, q_hi = kBias;
        if (d != 0.0f) {
            const float r = __frcp_rn(d);
            q_lo = pack4(lo, d, r, kLo, kHi, kBias);
            q_hi = pack4(hi, d, r, kLo, kHi, kBias);
        }
        const __half dl = __shfl_sync(kFull, dh, (lane & 7) * 4);
        if ((lane >> 3) == i) mine = dl;
        const int64_t b = b0 + 8 * i + (lane >> 2);
        if constexpr (FMT == EMB_Q8_0) {
            if (b < total) {
                uint32_t* dst = reinterpret_cast<uint32_t*>(codes + b * 32) + sub;
                __stcs(dst, q_lo);
                __stcs(dst + 4, q_hi);
            }
        } else {
            // low plane: byte j = low nibble of code j | low nibble of code j + 16 << 4
            if (b < total)
                __stcs(reinterpret_cast<uint32_t*>(codes + b * 16) + sub,
                       (q_lo & 0x0F0F0F0Fu) | (q_hi & 0x0F0F0F0Fu) << 4);
            if constexpr (FMT == EMB_Q6_0) {
                // high plane: byte j = high bits of codes j, j+8, j+16, j+24 at bit pairs 0..3, so
                // word p of a block comes from lanes p and p + 2
                const int at = 2 * (sub >> 1);
                uint32_t hw = (q_lo >> 4 & 0x03030303u) << at | (q_hi >> 4 & 0x03030303u) << (4 + at);
                hw |= __shfl_xor_sync(kFull, hw, 2);
                if (sub < 2 && b < total) __stcs(reinterpret_cast<uint32_t*>(high + b * 8) + sub, hw);
            }
        }
    }
    const int64_t b = b0 + lane;
    if (lane < kBlocks && b < total) {
        const int64_t n = pad ? b / nb : 0;
        scales[pad ? n * L.ldS + (b - n * nb) : b] = mine;
    }
}

__device__ __forceinline__ float deq_one(int fmt, const uint8_t* codes, const uint8_t* high,
                                         const __half* scales, int64_t K, int64_t ldS, int64_t n,
                                         int64_t k) {
    const float d = __half2float(scales[n * ldS + k / kQBlock]);
    int q;
    if (fmt == EMB_Q8_0) {
        q = int(reinterpret_cast<const int8_t*>(codes)[n * K + k]);
    } else {
        const int64_t b = k / kQBlock, i = k % kQBlock;
        const uint8_t byte = codes[n * (K / 2) + b * 16 + (i & 15)];
        q = int((i < 16) ? (byte & 0xF) : (byte >> 4));
        if (fmt == EMB_Q6_0) {
            const uint8_t hb = high[n * (K / 4) + b * 8 + (i & 7)];
            q = (q | (((hb >> (2 * (i >> 3))) & 3) << 4)) - 32;
        } else {
            q -= 8;
        }
    }
    return __fmul_rn(d, float(q));  // exact: 11-bit x at most 8-bit significands
}

__global__ void dequant_f32_kernel(int fmt, const uint8_t* __restrict__ codes,
                                   const uint8_t* __restrict__ high,
                                   const __half* __restrict__ scales, int64_t N, int64_t K,
                                   int64_t ldS, float* __restrict__ out) {
    const int64_t total = N * K;
    for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < total;
         i += int64_t(gridDim.x) * blockDim.x)
        out[i] = deq_one(fmt, codes, high, scales, K, ldS, i / K, i % K);
}

__global__ void dequant_bf16_kernel(int fmt, const uint8_t* __restrict__ codes,
                                    const uint8_t* __restrict__ high,
                                    const __half* __restrict__ scales, int64_t N, int64_t K,
                                    int64_t ldS, __nv_bfloat16* __restrict__ out) {
    const int64_t total = N * K;
    for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < total;
         i += int64_t(gridDim.x) * blockDim.x)
        out[i] = __float2bfloat16_rn(deq_one(fmt, codes, high, scales, K, ldS, i / K, i % K));
}

int grid_for(int64_t items, int per_block) {
    int64_t g = (items + per_block - 1) / per_block;
    if (g > 152 * 64) g = 152 * 64;
    return int(g < 1 ? 1 : g);
}

template <int LOADS>
cudaError_t launch_pack(int fmt, const float* W, int64_t N, int64_t K, uint8_t* base, const Layout& L, cudaStream_t s) {
    __half* scales = reinterpret_cast<__half*>(base + L.scales_off);
    const int64_t per_cta = int64_t(8 * LOADS) * (kPackThreads / 32);
    const int64_t ctas = (N * (K / kQBlock) + per_cta - 1) / per_cta;
    if (ctas > int64_t(0x7fffffff)) return cudaErrorInvalidConfiguration;
    const unsigned grid = unsigned(ctas);
    if (fmt == EMB_Q8_0)
        pack_kernel<EMB_Q8_0, LOADS><<<grid, kPackThreads, 0, s>>>(W, N, K, base, nullptr, scales, L);
    else if (fmt == EMB_Q4_0)
        pack_kernel<EMB_Q4_0, LOADS><<<grid, kPackThreads, 0, s>>>(W, N, K, base, nullptr, scales, L);
    else
        pack_kernel<EMB_Q6_0, LOADS><<<grid, kPackThreads, 0, s>>>(W, N, K, base, base + L.high_off, scales, L);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_quantize(int fmt, const float* W, int64_t N, int64_t K, void* img,
                            cudaStream_t s) {
    const Layout L = layout_of(fmt, N, K);
    uint8_t* base = static_cast<uint8_t*>(img);
    // fewer blocks per warp while those of 32 would leave SMs without a CTA (see the kernel)
    return N * (K / kQBlock) <= int64_t(256) * 152 ? launch_pack<1>(fmt, W, N, K, base, L, s)
                                                   : launch_pack<4>(fmt, W, N, K, base, L, s);
}

cudaError_t launch_dequant_f32(int fmt, const void* img, int64_t N, int64_t K, float* out,
                               cudaStream_t s) {
    const Layout L = layout_of(fmt, N, K);
    const uint8_t* base = static_cast<const uint8_t*>(img);
    dequant_f32_kernel<<<grid_for(N * K, 256), 256, 0, s>>>(
        fmt, base, base + L.high_off, reinterpret_cast<const __half*>(base + L.scales_off), N, K,
        L.ldS, out);
    return cudaGetLastError();
}

cudaError_t launch_dequant_bf16(int fmt, const void* img, int64_t N, int64_t K, uint16_t* out,
                                cudaStream_t s) {
    const Layout L = layout_of(fmt, N, K);
    const uint8_t* base = static_cast<const uint8_t*>(img);
    dequant_bf16_kernel<<<grid_for(N * K, 256), 256, 0, s>>>(
        fmt, base, base + L.high_off, reinterpret_cast<const __half*>(base + L.scales_off), N, K,
        L.ldS, reinterpret_cast<__nv_bfloat16*>(out));
    return cudaGetLastError();
}

}  // namespace emb
