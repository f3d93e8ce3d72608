// The non-matmul steps of one transformer layer of the shared backbone and the action
// expert (the paper's single backbone execution path, Section 3.2): RMSNorm of the fp32
// residual stream into the bf16 activations of the next linear, rotary position
// embedding of q and k in place, and grouped-head attention of a chunk of queries over a
// prefix key/value cache plus the chunk's own keys. Definitions: RMSNorm (Zhang and
// Sennrich, 2019), rotary embedding with rotate-half pairs (Su et al., 2021), scaled
// dot-product attention (Vaswani et al., 2017); all keys are visible to every query.
//
// Every kernel is launched with programmatic stream serialisation and reads its inputs
// only after griddepcontrol.wait, so it chains behind the layer launches of emb_qlayer_seq.
#include <algorithm>
#include <cmath>
#include <mutex>
#include <type_traits>

#include "ptx.cuh"

namespace emb {
namespace {

cudaError_t launch_pdl(const void* fn, dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                       void** args, unsigned cluster_z = 1) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    int na = 1;
    if (cluster_z > 1) {
        attr[1].id = cudaLaunchAttributeClusterDimension;
        attr[1].val.clusterDim.x = 1;
        attr[1].val.clusterDim.y = 1;
        attr[1].val.clusterDim.z = cluster_z;
        na = 2;
    }
    cfg.attrs = attr;
    cfg.numAttrs = na;
    return cudaLaunchKernelExC(&cfg, fn, args);
}

// ------------------------------------------------------------------ RMSNorm
// One CTA per token: the sum of squares in fp32 (per-thread partial sums of 4-element
// groups, then a shuffle tree and the warps' sums in order), mean = sum / D, one correctly
// rounded square root and reciprocal, then y = bf16(x * inv * gamma). Latency bounds it (0.3 MB at
// 50 x 1024), so a thread loads its elements of x and gamma once, up to KEEP groups of each in
// registers and gamma's loads on their way during the reduction, and one barrier is left: every
// thread adds the warps' sums for itself. A thread takes up to four groups before a CTA takes more
// threads than 256 (a thread per group, us: 50 x 4096 2.44 instead of 1.41, 150 x 4096 2.85 instead of
// 1.93), and many tokens take 256 throughout (512: 816 x 2048 4.1).
// Per launch, before (256 threads, x read twice, two barriers) and now, us: 50 x 1024 1.49 -> 1.13,
// 1 x 4096 2.00 -> 1.28, 50 x 4096 2.12 -> 1.41, 300 x 8192 4.64 -> 2.51, 816 x 2048 2.62 -> 2.46,
// 816 x 8192 5.59 -> 5.82, 1200 x 8192 9.48 -> 6.75.

// x and gamma are read with ordinary loads (not the read-only path): the previous launch may have
// written them while this grid was already resident (programmatic dependent launch); its writes are
// visible to ordinary loads after griddepcontrol.wait.
template <int NT, int KEEP>
__global__ void __launch_bounds__(NT) rmsnorm_kernel(const float* x, const float* gamma,
                                                     __nv_bfloat16* __restrict__ y, int D, float eps) {
    ptx::griddep_launch_dependents();
    ptx::griddep_wait();  // x is the residual stream the previous launch wrote
    const int64_t row = blockIdx.x;
    const float* xr = x + row * D;
    __nv_bfloat16* yr = y + row * D;
    const int i0 = threadIdx.x * 4;
    float4 v[KEEP], gm[KEEP];
#pragma unroll
    for (int k = 0; k < KEEP; ++k)
        v[k] = i0 + k * NT * 4 < D ? *reinterpret_cast<const float4*>(xr + i0 + k * NT * 4) : make_float4(0, 0, 0, 0);
#pragma unroll
    for (int k = 0; k < KEEP; ++k)
        if (i0 + k * NT * 4 < D) gm[k] = *reinterpret_cast<const float4*>(gamma + i0 + k * NT * 4);
    float ss = 0.0f;
    auto add = [&](const float4& q) {
        ss = fmaf(q.x, q.x, ss);
        ss = fmaf(q.y, q.y, ss);
        ss = fmaf(q.z, q.z, ss);
        ss = fmaf(q.w, q.w, ss);
    };
#pragma unroll
    for (int k = 0; k < KEEP; ++k) add(v[k]);
    for (int i = i0 + KEEP * NT * 4; i < D; i += NT * 4) add(*reinterpret_cast<const float4*>(xr + i));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
    __shared__ float warp_ss[NT / 32];
    if ((threadIdx.x & 31) == 0) warp_ss[threadIdx.x >> 5] = ss;
    __syncthreads();
    float t = 0.0f;
#pragma unroll
    for (int w = 0; w < NT / 32; ++w) t += warp_ss[w];
    const float inv = __fdiv_rn(1.0f, __fsqrt_rn(__fadd_rn(__fdiv_rn(t, float(D)), eps)));
    auto store = [&](int i, const float4& q, const float4& g) {
        const __nv_bfloat162 lo = __floats2bfloat162_rn(__fmul_rn(__fmul_rn(q.x, inv), g.x),
                                                        __fmul_rn(__fmul_rn(q.y, inv), g.y));
        const __nv_bfloat162 hi = __floats2bfloat162_rn(__fmul_rn(__fmul_rn(q.z, inv), g.z),
                                                        __fmul_rn(__fmul_rn(q.w, inv), g.w));
        uint2 u;
        u.x = *reinterpret_cast<const uint32_t*>(&lo);
        u.y = *reinterpret_cast<const uint32_t*>(&hi);
        *reinterpret_cast<uint2*>(yr + i) = u;
    };
#pragma unroll
    for (int k = 0; k < KEEP; ++k)
        if (i0 + k * NT * 4 < D) store(i0 + k * NT * 4, v[k], gm[k]);
    for (int i = i0 + KEEP * NT * 4; i < D; i += NT * 4)
        store(i, *reinterpret_cast<const float4*>(xr + i), *reinterpret_cast<const float4*>(gamma + i));
}

// ------------------------------------------------------------------ rotary embedding
// A thread rotates VEC consecutive pairs (elements i .. i + VEC - 1 and the same + d/2) of one head
// of one token, with one load and store of VEC bf16 for either half. The host
// passes each pair's inverse frequency base^(-2i/d), computed in fp64, as two floats
// (hi + lo). The angle p * (hi + lo) is formed as an unevaluated sum A + a with one exact
// FMA residual (p < 2^24 is exact in fp32), its sine and cosine as sincosf(A) corrected by a: error
// ~1e-7 at every position, against ~|angle| * 2^-24 for a plain fp32 angle. To first order while the
// largest angle stays below 4096 (|a| < 2^-12 + 2^-13, so a^2 / 2 < 7e-8); beyond it (LARGE) a grows
// to a radian and more and takes its own sine and cosine. The frequencies go through shared memory (filled before
// the dependency wait): read from the parameter bank, where a warp's 32 different entries take 32
// turns, and with one pair, a 64-bit division and 2-byte accesses per thread, 816 tokens x 9 heads of
// 256 took 16.8 us; now 4.3 (15 MB moved), 50 tokens x 9 heads of 128 2.4 -> 1.4 us.
constexpr int kRopeMaxPairs = 256;

struct RopeParams {
    __nv_bfloat16* x;   // [M][n_heads][head_dim]
    __nv_bfloat16* x2;  // [M][n_heads2][head_dim] at the same positions, or nothing (n_heads2 = 0)
    int64_t units, pos0;  // units: VEC pairs of one head of one token
    int n_heads, n_heads2, head_dim;
    float inv_hi[kRopeMaxPairs], inv_lo[kRopeMaxPairs];
};

template <int VEC>
struct alignas(2 * VEC) BfVec {
    __nv_bfloat16 v[VEC];
};

template <int VEC, bool LARGE>
__global__ void __launch_bounds__(256) rope_kernel(const __grid_constant__ RopeParams p) {
    __shared__ float inv_hi[kRopeMaxPairs], inv_lo[kRopeMaxPairs];
    const int half = p.head_dim / 2;
    ptx::griddep_launch_dependents();
    for (int i = threadIdx.x; i < half; i += 256) {
        inv_hi[i] = p.inv_hi[i];
        inv_lo[i] = p.inv_lo[i];
    }
    __syncthreads();
    ptx::griddep_wait();  // x was written by the previous launch
    const uint32_t per_head = uint32_t(half / VEC), heads = uint32_t(p.n_heads + p.n_heads2);
    const int64_t per_token = int64_t(heads) * per_head;
    for (int64_t u = int64_t(blockIdx.x) * 256 + threadIdx.x; u < p.units; u += int64_t(gridDim.x) * 256) {
        int64_t m;
        uint32_t r;  // unit of the token: head, then the pairs within it
        if (p.units <= int64_t(0xffffffffu)) {
            m = uint32_t(u) / uint32_t(per_token);
            r = uint32_t(u) - uint32_t(m) * uint32_t(per_token);
        } else {
            m = u / per_token;
            r = uint32_t(u - m * per_token);
        }
        const uint32_t h = r / per_head;
        const int i = int(r - h * per_head) * VEC;
        const bool second = h >= uint32_t(p.n_heads);  // the heads of x come first, then those of x2
        __nv_bfloat16* xp = second ? p.x2 + (m * p.n_heads2 + (h - uint32_t(p.n_heads))) * int64_t(p.head_dim) + i
                                   : p.x + (m * p.n_heads + h) * int64_t(p.head_dim) + i;
        const BfVec<VEC> va = *reinterpret_cast<const BfVec<VEC>*>(xp);
        const BfVec<VEC> vb = *reinterpret_cast<const BfVec<VEC>*>(xp + half);
        BfVec<VEC> oa, ob;
        const float pos = float(p.pos0 + m);
#pragma unroll
        for (int e = 0; e < VEC; ++e) {
            const float hi = inv_hi[i + e];
            const float A = __fmul_rn(pos, hi);
            const float a = __fadd_rn(fmaf(pos, hi, -A), __fmul_rn(pos, inv_lo[i + e]));
            float sA, cA;
            sincosf(A, &sA, &cA);
            float c, s;
            if constexpr (LARGE) {
                // sine and cosine of a by their series (error below 1e-10 up to 1/16), then the addition formulas
                const float a2 = __fmul_rn(a, a);
                float sa = __fmul_rn(a, fmaf(a2, fmaf(a2, 1.0f / 120.0f, -1.0f / 6.0f), 1.0f));
                float ca = fmaf(a2, fmaf(a2, 1.0f / 24.0f, -0.5f), 1.0f);
                if (fabsf(a) > 0.0625f) sincosf(a, &sa, &ca);
                c = fmaf(cA, ca, -__fmul_rn(sA, sa));
                s = fmaf(sA, ca, __fmul_rn(cA, sa));
            } else {
                c = fmaf(-a, sA, cA);
                s = fmaf(a, cA, sA);
            }
            const float xa = __bfloat162float(va.v[e]), xb = __bfloat162float(vb.v[e]);
            oa.v[e] = __float2bfloat16_rn(__fsub_rn(__fmul_rn(xa, c), __fmul_rn(xb, s)));
            ob.v[e] = __float2bfloat16_rn(__fadd_rn(__fmul_rn(xb, c), __fmul_rn(xa, s)));
        }
        *reinterpret_cast<BfVec<VEC>*>(xp) = oa;
        *reinterpret_cast<BfVec<VEC>*>(xp + half) = ob;
    }
}

template <bool LARGE>
const void* rope_fn(int vec) {
    return vec == 8   ? reinterpret_cast<const void*>(rope_kernel<8, LARGE>)
           : vec == 4 ? reinterpret_cast<const void*>(rope_kernel<4, LARGE>)
           : vec == 2 ? reinterpret_cast<const void*>(rope_kernel<2, LARGE>)
                      : reinterpret_cast<const void*>(rope_kernel<1, LARGE>);
}

// ------------------------------------------------------------------ attention
// Tensor-core attention (mma.sync m16n8k16, bf16 operands, fp32 accumulation). The rows of
// one key/value head g are its (query m, head) pairs, row r = m * G + (h - g * G) with G the
// heads per key/value head, so every query head of a group shares the key and value tiles.
// CTA = (row block, key/value head, key split) of four warps, which walk the split's keys in
// tiles of 64 (double-buffered in shared memory by cp.async, rows padded by 16 bytes so
// fragment loads are conflict-free). WK = 1: a row block is 64 rows, 16 per warp, and every warp
// takes all 64 keys. WK = 4, for few rows (a decode step's one query per head would leave
// three warps of four without a row): a row block is 16 rows, every warp takes 16 of a tile's
// keys, and the warps' partial results are combined in shared memory.
// Per tile: S = Q K^T (Q fragments held in registers for the whole kernel), an online softmax
// in base 2 on the accumulator fragments (row max and sums over the four lanes that share a row),
// then O += P V with P split into bf16 hi + lo parts (two MMAs, weight error 2^-16) and V
// fragments from ldmatrix.trans. The key splits of one row block form a cluster along z; their
// (max, sum, output) partials are combined through distributed shared memory in split order
// (deterministic).
// What bounds it: latency. mma.sync does 1016 bf16 multiply-adds per cycle and SM here, which is
// 7 us for M = 816, 8 heads, 816 keys (26.4 us measured, 84.2 before); the rest is each warp's
// chain of loads, scores, exponentials and products with one or two warps per scheduler, and the
// clusters' exchange. Consecutive MMAs go to different accumulators, weights are 2^x (one
// multiply into base 2 per score), and unchanged row maxima skip the rescaling of the output.
constexpr int kAttnWarps = 4;
constexpr int kAttnThreads = 32 * kAttnWarps;
template <int WK>
constexpr int kAttnRows = 16 * kAttnWarps / WK;  // rows of a CTA
constexpr int kKeyTile = 64;
constexpr int kMaxSplits = 16;      // cluster size along the keys (16: non-portable, opted in)
constexpr int kMinSplitKeys = 32;   // keys per split, at least

template <int D>
struct AttnSmem {
    static constexpr int kPitch = D + 8;                 // bf16 per padded key row
    __nv_bfloat16 k[2][kKeyTile][kPitch];
    __nv_bfloat16 v[2][kKeyTile][kPitch];
    float part_o[16 * kAttnWarps][D];  // one 16-row partial result per warp
    float part_m[16 * kAttnWarps], part_l[16 * kAttnWarps];
    float cta_m[16], cta_l[16];        // WK > 1: the CTA's rows after its warps are combined
};

struct AttnParams {
    const __nv_bfloat16* Q;
    const __nv_bfloat16* K0;
    const __nv_bfloat16* V0;
    const __nv_bfloat16* K1;
    const __nv_bfloat16* V1;
    __nv_bfloat16* O;
    int64_t n0, n1;
    int M, H, Hk;
    float scale_log2;  // scale * log2(e): scores are kept in base 2
};

__device__ __forceinline__ void mma_16816(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, "
        "{%8, %9}, {%0, %1, %2, %3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// 2^x (results below the normal range become zero; -inf gives 0).
__device__ __forceinline__ float exp2_fast(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ void ldsm_x4(uint32_t saddr, uint32_t& r0, uint32_t& r1, uint32_t& r2,
                                        uint32_t& r3) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
                 : "r"(saddr));
}
__device__ __forceinline__ void ldsm_x4_trans(uint32_t saddr, uint32_t& r0, uint32_t& r1, uint32_t& r2,
                                              uint32_t& r3) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
                 : "r"(saddr));
}

// 16-byte global -> shared copy; src_bytes 0 writes zeros (the source is not read).
__device__ __forceinline__ void cp_async16(uint32_t saddr, const void* g, int src_bytes) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(saddr), "l"(g), "r"(src_bytes)
                 : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait1() { asm volatile("cp.async.wait_group 1;" ::: "memory"); }

__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
    const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t*>(&v);
}
__device__ __forceinline__ float2 unpack_bf16x2(uint32_t w) {
    return make_float2(__uint_as_float(w << 16), __uint_as_float(w & 0xFFFF0000u));
}

template <int D, int WK>
__global__ void __launch_bounds__(kAttnThreads) attention_kernel(const __grid_constant__ AttnParams p) {
    constexpr int KS = D / 16;  // k-steps of the score MMAs (head dims)
    constexpr int NT = D / 8;   // n-tiles of the output (head dims)
    constexpr int NJ = kKeyTile / 8 / WK;   // 8-key n-tiles of a warp's share of a tile
    constexpr int kRows = kAttnRows<WK>;
    using SM = AttnSmem<D>;
    extern __shared__ __align__(128) uint8_t smem_raw[];
    SM& sm = *reinterpret_cast<SM*>(smem_raw);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int quad = lane >> 2, qc = lane & 3;
    const int g = blockIdx.y, G = p.H / p.Hk;
    const int64_t rows_total = int64_t(p.M) * G;
    const int64_t row0 = int64_t(blockIdx.x) * kRows;
    const int splits = gridDim.z, z = blockIdx.z;
    const int64_t n = p.n0 + p.n1;
    const int64_t k_lo = z * n / splits, k_hi = (z + 1) * n / splits;
    const int64_t kv_stride = int64_t(p.Hk) * D;
    const int wrow = WK == 1 ? warp * 16 : 0;  // the warp's rows of the CTA, and keys of a tile
    const int wkey = WK == 1 ? 0 : warp * 16;

    ptx::griddep_launch_dependents();
    ptx::griddep_wait();  // Q and the chunk's keys and values come from the previous launches

    // tile loader: 64 keys x D of keys and of values, 16-byte chunks, zero past the split
    constexpr int kChunksPerRow = D / 8, kPass = kAttnThreads / kChunksPerRow;
    const int lc = threadIdx.x % kChunksPerRow, lj = threadIdx.x / kChunksPerRow;
    const int64_t col = int64_t(g) * D + lc * 8;
    auto issue_tile = [&](int64_t t0, int stage) {
#pragma unroll
        for (int i = 0; i < kKeyTile / kPass; ++i) {
            const int j = lj + i * kPass;
            const bool ok = t0 + j < k_hi;
            const int64_t kk = ok ? t0 + j : k_lo;  // any valid row when nothing is read
            const bool cached = kk < p.n0;
            const int64_t off = (cached ? kk : kk - p.n0) * kv_stride + col;
            cp_async16(ptx::smem_u32(&sm.k[stage][j][lc * 8]), (cached ? p.K0 : p.K1) + off, ok ? 16 : 0);
            cp_async16(ptx::smem_u32(&sm.v[stage][j][lc * 8]), (cached ? p.V0 : p.V1) + off, ok ? 16 : 0);
        }
    };
    const int ntiles = int((k_hi - k_lo + kKeyTile - 1) / kKeyTile);
    if (ntiles > 0) issue_tile(k_lo, 0);
    cp_async_commit();

    // global row -> (query, head) -> its Q / O row; -1 past the last row
    auto q_row = [&](int64_t r) -> int64_t {
        return r < rows_total ? (r / G) * int64_t(p.H) * D + (int64_t(g) * G + r % G) * D : -1;
    };
    const int64_t offA = q_row(row0 + wrow + quad), offB = q_row(row0 + wrow + quad + 8);

    // Q fragments for the whole kernel (A operand, row-major 16 x D); ordinary loads, since
    // the previous launch wrote Q while this grid was already resident
    uint32_t qf[KS][4];
    auto ldq = [&](int64_t off) { return *reinterpret_cast<const uint32_t*>(p.Q + off); };
#pragma unroll
    for (int ks = 0; ks < KS; ++ks) {
        const int c = ks * 16 + 2 * qc;
        qf[ks][0] = offA >= 0 ? ldq(offA + c) : 0u;
        qf[ks][1] = offB >= 0 ? ldq(offB + c) : 0u;
        qf[ks][2] = offA >= 0 ? ldq(offA + c + 8) : 0u;
        qf[ks][3] = offB >= 0 ? ldq(offB + c + 8) : 0u;
    }

    float o[NT][4];
#pragma unroll
    for (int j = 0; j < NT; ++j) o[j][0] = o[j][1] = o[j][2] = o[j][3] = 0.0f;
    float mA = -INFINITY, mB = -INFINITY, lA = 0.0f, lB = 0.0f;

    for (int it = 0; it < ntiles; ++it) {
        const int stage = it & 1;
        const int64_t t0 = k_lo + int64_t(it) * kKeyTile;
        if (it + 1 < ntiles) issue_tile(t0 + kKeyTile, stage ^ 1);
        cp_async_commit();
        cp_async_wait1();  // this thread's copies of tile `it` have landed
        __syncthreads();   // and every thread's

        // S = Q K^T for the warp's keys, 8 per n-tile; one ldmatrix gives the B fragments of two
        // k-steps (lanes 8i .. 8i + 7 address the eight keys at dims 8i). The n-tiles are the inner
        // loop: consecutive MMAs then do not wait for one another.
        float sc[NJ][4];
#pragma unroll
        for (int j = 0; j < NJ; ++j) sc[j][0] = sc[j][1] = sc[j][2] = sc[j][3] = 0.0f;
        const uint32_t kbase = ptx::smem_u32(&sm.k[stage][wkey + (lane & 7)][(lane >> 3) * 8]);
#pragma unroll
        for (int ks = 0; ks < KS; ks += 2) {
            uint32_t b[NJ][4];
#pragma unroll
            for (int j = 0; j < NJ; ++j)
                ldsm_x4(kbase + j * 8 * SM::kPitch * 2 + ks * 32, b[j][0], b[j][1], b[j][2], b[j][3]);
#pragma unroll
            for (int j = 0; j < NJ; ++j) mma_16816(sc[j], qf[ks], b[j][0], b[j][1]);
#pragma unroll
            for (int j = 0; j < NJ; ++j) mma_16816(sc[j], qf[ks + 1], b[j][2], b[j][3]);
        }
        // scores in base 2, keys past the split masked (last tile only), row maxima (rows A =
        // quad, B = quad + 8)
        const int left = int(min(k_hi - t0, int64_t(kKeyTile)));
        float tA = -INFINITY, tB = -INFINITY;
#pragma unroll
        for (int j = 0; j < NJ; ++j) {
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                sc[j][e] = __fmul_rn(sc[j][e], p.scale_log2);
                sc[j][2 + e] = __fmul_rn(sc[j][2 + e], p.scale_log2);
            }
        }
        if (left < kKeyTile) {
#pragma unroll
            for (int j = 0; j < NJ; ++j)
#pragma unroll
                for (int e = 0; e < 2; ++e)
                    if (wkey + j * 8 + 2 * qc + e >= left) sc[j][e] = sc[j][2 + e] = -INFINITY;
        }
#pragma unroll
        for (int j = 0; j < NJ; ++j) {
            tA = fmaxf(tA, fmaxf(sc[j][0], sc[j][1]));
            tB = fmaxf(tB, fmaxf(sc[j][2], sc[j][3]));
        }
#pragma unroll
        for (int x = 1; x <= 2; x <<= 1) {
            tA = fmaxf(tA, __shfl_xor_sync(0xffffffffu, tA, x));
            tB = fmaxf(tB, __shfl_xor_sync(0xffffffffu, tB, x));
        }
        const float nA = fmaxf(mA, tA), nB = fmaxf(mB, tB);
        // (a row without a finite score so far subtracts 0: its weights are 2^-inf = 0)
        const float sA0 = nA == -INFINITY ? 0.0f : nA, sB0 = nB == -INFINITY ? 0.0f : nB;
        const float cA = exp2_fast(mA - sA0), cB = exp2_fast(mB - sB0);
        float sA = 0.0f, sB = 0.0f;
#pragma unroll
        for (int j = 0; j < NJ; ++j) {
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                sc[j][e] = exp2_fast(sc[j][e] - sA0);
                sc[j][2 + e] = exp2_fast(sc[j][2 + e] - sB0);
                sA += sc[j][e];
                sB += sc[j][2 + e];
            }
        }
        lA = lA * cA + sA;  // lane-partial sums; the four lanes of a row are added at the end
        lB = lB * cB + sB;
        if (__any_sync(0xffffffffu, nA != mA || nB != mB)) {  // else every factor is 1
#pragma unroll
            for (int j = 0; j < NT; ++j) {
                o[j][0] *= cA;
                o[j][1] *= cA;
                o[j][2] *= cB;
                o[j][3] *= cB;
            }
        }
        mA = nA;
        mB = nB;
        // O += P V: k-steps of 16 keys; P as hi + lo bf16 A fragments
#pragma unroll
        for (int kk = 0; kk < NJ / 2; ++kk) {
            uint32_t ah[4], al[4];
            const float* s0 = sc[2 * kk];
            const float* s1 = sc[2 * kk + 1];
            const float src[4][2] = {{s0[0], s0[1]}, {s0[2], s0[3]}, {s1[0], s1[1]}, {s1[2], s1[3]}};
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                ah[r] = pack_bf16x2(src[r][0], src[r][1]);
                const float2 h = unpack_bf16x2(ah[r]);
                al[r] = pack_bf16x2(__fsub_rn(src[r][0], h.x), __fsub_rn(src[r][1], h.y));
            }
            // ldmatrix.trans: lanes 0-7 keys 16kk..+7, 8-15 keys +8..+15 (dims 8jj..),
            // lanes 16-31 the same keys at dims 8jj + 8
            const int key = wkey + kk * 16 + (lane & 7) + ((lane >> 3) & 1) * 8;
            const uint32_t vrow = ptx::smem_u32(&sm.v[stage][key][(lane >> 4) * 8]);
#pragma unroll
            for (int jj = 0; jj < NT; jj += 4) {
                uint32_t b[2][4];
                ldsm_x4_trans(vrow + jj * 16, b[0][0], b[0][1], b[0][2], b[0][3]);
                ldsm_x4_trans(vrow + jj * 16 + 32, b[1][0], b[1][1], b[1][2], b[1][3]);
#pragma unroll
                for (int i = 0; i < 4; ++i) mma_16816(o[jj + i], ah, b[i >> 1][2 * (i & 1)], b[i >> 1][2 * (i & 1) + 1]);
#pragma unroll
                for (int i = 0; i < 4; ++i) mma_16816(o[jj + i], al, b[i >> 1][2 * (i & 1)], b[i >> 1][2 * (i & 1) + 1]);
            }
        }
        __syncthreads();  // every warp is done with this stage before it is refilled
    }
#pragma unroll
    for (int x = 1; x <= 2; x <<= 1) {
        lA += __shfl_xor_sync(0xffffffffu, lA, x);
        lB += __shfl_xor_sync(0xffffffffu, lB, x);
    }

    auto store4 = [&](int64_t at, float4 v, float L) {  // four normalised outputs
        const float inv = __fdiv_rn(1.0f, L);
        const __nv_bfloat162 lo = __floats2bfloat162_rn(__fmul_rn(v.x, inv), __fmul_rn(v.y, inv));
        const __nv_bfloat162 hi = __floats2bfloat162_rn(__fmul_rn(v.z, inv), __fmul_rn(v.w, inv));
        uint2 u;
        u.x = *reinterpret_cast<const uint32_t*>(&lo);
        u.y = *reinterpret_cast<const uint32_t*>(&hi);
        *reinterpret_cast<uint2*>(p.O + at) = u;
    };
    if (WK == 1 && splits == 1) {
        const float iA = __fdiv_rn(1.0f, lA), iB = __fdiv_rn(1.0f, lB);
#pragma unroll
        for (int j = 0; j < NT; ++j) {
            const int c = j * 8 + 2 * qc;
            if (offA >= 0)
                *reinterpret_cast<__nv_bfloat162*>(p.O + offA + c) =
                    __floats2bfloat162_rn(__fmul_rn(o[j][0], iA), __fmul_rn(o[j][1], iA));
            if (offB >= 0)
                *reinterpret_cast<__nv_bfloat162*>(p.O + offB + c) =
                    __floats2bfloat162_rn(__fmul_rn(o[j][2], iB), __fmul_rn(o[j][3], iB));
        }
        return;
    }
    // each warp's partial result into shared memory
    const int lrA = warp * 16 + quad, lrB = lrA + 8;
#pragma unroll
    for (int j = 0; j < NT; ++j) {
        const int c = j * 8 + 2 * qc;
        *reinterpret_cast<float2*>(&sm.part_o[lrA][c]) = make_float2(o[j][0], o[j][1]);
        *reinterpret_cast<float2*>(&sm.part_o[lrB][c]) = make_float2(o[j][2], o[j][3]);
    }
    if (qc == 0) {
        sm.part_m[lrA] = mA;
        sm.part_l[lrA] = lA;
        sm.part_m[lrB] = mB;
        sm.part_l[lrB] = lB;
    }
    // max, sum and output of the partials that share a row, added in order
    auto merge = [](const float* qm, const float* ql, const float4* qo, auto count, float& mx, float& L, float4& O) {
        constexpr int kCount = decltype(count)::value;
        mx = -INFINITY;
#pragma unroll
        for (int q = 0; q < kCount; ++q)
            mx = fmaxf(mx, qm[q]);
        const float m0 = mx == -INFINITY ? 0.0f : mx;
        L = 0.0f;
        O = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll
        for (int q = 0; q < kCount; ++q) {
            // a partial without a finite score has weight 0: its sums are 0 without keys (or with
            // scores of -inf alone), and NaN with a score of NaN, which has to show
            const float w = exp2_fast(qm[q] - m0);
            L = fmaf(ql[q], w, L);
            O.x = fmaf(qo[q].x, w, O.x);
            O.y = fmaf(qo[q].y, w, O.y);
            O.z = fmaf(qo[q].z, w, O.z);
            O.w = fmaf(qo[q].w, w, O.w);
        }
    };
    if constexpr (WK > 1) {
        // the four warps' partials of the CTA's 16 rows: one thread per 4 dims
        __syncthreads();
        for (int e = threadIdx.x; e < 16 * (D / 4); e += kAttnThreads) {
            const int r = e / (D / 4), c = (e % (D / 4)) * 4;
            float qm[WK], ql[WK], mx, L;
            float4 qo[WK], O;
#pragma unroll
            for (int w = 0; w < WK; ++w) {
                qm[w] = sm.part_m[16 * w + r];
                ql[w] = sm.part_l[16 * w + r];
                qo[w] = *reinterpret_cast<const float4*>(&sm.part_o[16 * w + r][c]);
            }
            merge(qm, ql, qo, std::integral_constant<int, WK>{}, mx, L, O);
            if (splits == 1) {
                const int64_t off = q_row(row0 + r);
                if (off >= 0) store4(off + c, O, L);
            } else {
                *reinterpret_cast<float4*>(&sm.part_o[r][c]) = O;  // read by this thread only so far
                if (c == 0) {
                    sm.cta_m[r] = mx;
                    sm.cta_l[r] = L;
                }
            }
        }
        if (splits == 1) return;
    }
    ptx::cluster_sync();
    // CTA z combines rows z, z + splits, ... of the row block, one thread per 4 dims; a thread
    // has the loads of 16 / splits elements in flight at once
    const int elems = (kRows + splits - 1) / splits * (D / 4);
    auto combine = [&](auto count) {
        constexpr int kSp = decltype(count)::value, kAtOnce = kMaxSplits / kSp;
        for (int e0 = threadIdx.x; e0 < elems; e0 += kAttnThreads * kAtOnce) {
            float qm[kAtOnce][kSp], ql[kAtOnce][kSp];
            float4 qo[kAtOnce][kSp];
            int64_t off[kAtOnce];
#pragma unroll
            for (int u = 0; u < kAtOnce; ++u) {
                const int e = e0 + u * kAttnThreads;
                const int lr = z + e / (D / 4) * splits, c = (e % (D / 4)) * 4;
                off[u] = e < elems && lr < kRows ? q_row(row0 + lr) : -1;
                if (off[u] < 0) continue;
                off[u] += c;
                const uint32_t am = ptx::smem_u32(WK > 1 ? &sm.cta_m[lr & 15] : &sm.part_m[lr]);
                const uint32_t al_ = ptx::smem_u32(WK > 1 ? &sm.cta_l[lr & 15] : &sm.part_l[lr]);
                const uint32_t ao = ptx::smem_u32(&sm.part_o[lr][c]);
#pragma unroll
                for (int q = 0; q < kSp; ++q) {
                    qm[u][q] = ptx::ld_dsmem_f32(ptx::map_dsmem(am, q));
                    ql[u][q] = ptx::ld_dsmem_f32(ptx::map_dsmem(al_, q));
                    qo[u][q] = ptx::ld_dsmem_f32x4(ptx::map_dsmem(ao, q));
                }
            }
#pragma unroll
            for (int u = 0; u < kAtOnce; ++u) {
                if (off[u] < 0) continue;
                float mx, L;
                float4 O;
                merge(qm[u], ql[u], qo[u], count, mx, L, O);
                store4(off[u], O, L);
            }
        }
    };
    if (splits == 2) combine(std::integral_constant<int, 2>{});
    else if (splits == 4) combine(std::integral_constant<int, 4>{});
    else if (splits == 8) combine(std::integral_constant<int, 8>{});
    else combine(std::integral_constant<int, 16>{});
    ptx::cluster_sync();  // remote shared memory must outlive its readers
}

// Which kernel (WK) and how many key splits (one cluster, a power of two) a call takes: the
// least time by a model in microseconds fitted on GB300. A CTA costs 2.5, per tile of 64 keys 1.8
// (D = 128) or 1.2 (D = 64) with 16 rows per warp and 1.0 or 0.5 with the keys shared out to the
// warps; CTAs that share an SM slow one another by a quarter each, clusters beyond those that run at
// once queue; a cluster adds 4.0 or 1.3 for its exchange and 0.8 more at 16 CTAs. With the keys
// shared out, the warps' merge costs 0.8 where no cluster's does, and 0.5 or 2.0 more beside one or two
// other CTAs on the SM (without these two terms 34 queries of 32 heads and 7 keys took 5.3 us instead of 3.8, 152
// queries of 32 heads on 4 and 16 keys 5.9 instead of 4.3, 50 queries of 16 heads on 8 of 64, 919 keys 10.3
// instead of 7.9; over 420 calls the plan now loses 1.5 % against the best one, geometric mean).
// Measured (us per launch, graph-replayed; before: 64 rows per CTA and as many splits as keys
// allow): M = 816, 8 heads on one key/value head of 128, 816 keys 84.2 -> 26.4 (2 splits); 280
// queries and keys, 32 heads 43.2 -> 16.9 (1); one query, 32
// heads, 281 keys 10.9 -> 5.5 (WK = 4, 8 splits); 400 queries, 16 heads on 4 of 64, 900 keys
// 41.5 -> 13.7 (4); one query, 8 heads on one, 4001 keys 14.5 -> 7.7 (WK = 4, 16).
struct AttnPlan {
    bool shared_keys;  // WK = 4
    int splits;
};

// The opt-in shared-memory size and cluster size are per-device function attributes. Clusters of 2^i CTAs
// of the kernel that run at once are asked once per device: fewer than the CTAs that do, since a cluster
// stays within a part of the chip (76 clusters of four in two rounds: 38 queries of 32 heads on 4, 3282 keys
// 41.7 us, in 20 of eight 25.8).
constexpr int kSplitKinds = 5;  // 1, 2, 4, 8, 16
struct AttnResident {
    int n[kSplitKinds];
};
template <int D, int WK>
cudaError_t prepare_attention(AttnResident& at_once) {
    static std::mutex mu;
    static AttnResident known[64] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    std::lock_guard<std::mutex> lock(mu);
    if (dev >= 0 && dev < 64 && known[dev].n[0]) {
        at_once = known[dev];
        return cudaSuccess;
    }
    auto* kernel = attention_kernel<D, WK>;
    const int smem = int(sizeof(AttnSmem<D>));
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    for (int i = 0; i < kSplitKinds && e == cudaSuccess; ++i) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(1, 1, 1u << i);
        cfg.blockDim = dim3(kAttnThreads);
        cfg.dynamicSmemBytes = size_t(smem);
        cudaLaunchAttribute attr;
        attr.id = cudaLaunchAttributeClusterDimension;
        attr.val.clusterDim.x = 1;
        attr.val.clusterDim.y = 1;
        attr.val.clusterDim.z = 1u << i;
        cfg.attrs = &attr;
        cfg.numAttrs = 1;
        e = cudaOccupancyMaxActiveClusters(&at_once.n[i], kernel, &cfg);
        at_once.n[i] = std::max(1, at_once.n[i]);
    }
    if (e == cudaSuccess && dev >= 0 && dev < 64) known[dev] = at_once;
    return e;
}

template <int D>
cudaError_t plan_attention(int64_t rows, int64_t Hk, int64_t n, AttnPlan& best) {
    const int count = device_sm_count();
    const double sms = count > 0 ? count : 152.0;
    const double per_sm = D == 64 ? 3.0 : 2.0;
    best = AttnPlan{false, 1};
    double best_t = 1e30;
    for (int few = 0; few < 2; ++few) {
        AttnResident at_once;
        const cudaError_t e = few ? prepare_attention<D, 4>(at_once) : prepare_attention<D, 1>(at_once);
        if (e != cudaSuccess) return e;
        const double blocks = double((rows + (few ? 15 : 63)) / (few ? 16 : 64)) * double(Hk);
        const double tile = few ? (D == 64 ? 0.5 : 1.0) : (D == 64 ? 1.2 : 1.8);
        for (int i = 0; i < kSplitKinds; ++i) {
            const int sp = 1 << i;
            if (sp > 1 && n < sp * int64_t(kMinSplitKeys)) break;
            const double ctas = blocks * sp;
            const double tiles = double((((n + sp - 1) / sp) + kKeyTile - 1) / kKeyTile);
            const double share = 1.0 + 0.25 * (std::min(std::ceil(ctas / sms), per_sm) - 1.0);
            const double x = blocks / double(at_once.n[i]);
            const double rounds = x <= 1.0 ? 1.0 : 0.5 * (x + std::ceil(x));
            const double beside = std::min(std::ceil(ctas / sms), per_sm) - 1.0;  // other CTAs on an SM
            const double t = rounds * (tiles * tile * share + 2.5 + (sp > 1 ? (few ? 1.3 : 4.0) : 0.0)) +
                             (sp == kMaxSplits ? 0.8 : 0.0) + (few ? (sp == 1 ? 0.8 : 0.0) + 0.5 * beside * beside : 0.0);
            if (t < best_t * 0.99) {
                best_t = t;
                best = AttnPlan{few != 0, sp};
            }
        }
    }
    return cudaSuccess;
}

template <int D, int WK>
cudaError_t launch_attention_wk(const AttnParams& p, int splits, cudaStream_t s) {
    AttnParams pc = p;
    void* args[] = {&pc};
    const int64_t row_blocks = (int64_t(p.M) * (p.H / p.Hk) + kAttnRows<WK> - 1) / kAttnRows<WK>;
    return launch_pdl(reinterpret_cast<const void*>(attention_kernel<D, WK>),
                      dim3(unsigned(row_blocks), unsigned(p.Hk), unsigned(splits)), dim3(kAttnThreads),
                      sizeof(AttnSmem<D>), s, args, unsigned(splits));
}

template <int D>
cudaError_t launch_attention_d(const AttnParams& p, cudaStream_t s) {
    AttnPlan pl;
    const cudaError_t e = plan_attention<D>(int64_t(p.M) * (p.H / p.Hk), p.Hk, p.n0 + p.n1, pl);
    if (e != cudaSuccess) return e;
    return pl.shared_keys ? launch_attention_wk<D, 4>(p, pl.splits, s) : launch_attention_wk<D, 1>(p, pl.splits, s);
}

}  // namespace

cudaError_t launch_rmsnorm(const float* x, const float* gamma, uint16_t* y, int64_t M, int64_t D,
                           float eps, cudaStream_t s) {
    const float* xa = x;
    const float* ga = gamma;
    __nv_bfloat16* ya = reinterpret_cast<__nv_bfloat16*>(y);
    int Di = int(D);
    void* args[] = {&xa, &ga, &ya, &Di, &eps};
    const int groups = Di / 4;
    const int count = device_sm_count();
    const int64_t sms = count > 0 ? count : 152;
    const bool many = M > 2 * sms;
    // longer rows than four groups per thread hold: 512 threads for few tokens, 1024 for up to one CTA per
    // SM of the longest; for many, 256 that keep one group where those that keep four, five CTAs per SM at
    // once, would leave their last wave more than a third empty (816 x 10240 8.0 instead of 6.7)
    const int64_t at_once = 5 * sms, waves = (M + at_once - 1) / at_once;
    const bool last_empty = waves > 1 && 3 * M < 2 * at_once * waves;
    const int nt = groups <= 128 ? 128 : groups <= 1024 || many ? 256 : groups > 2048 && M <= sms ? 1024 : 512;
    const void* fn = nt == 128    ? reinterpret_cast<const void*>(rmsnorm_kernel<128, 1>)
                     : nt == 512  ? reinterpret_cast<const void*>(rmsnorm_kernel<512, 4>)
                     : nt == 1024 ? reinterpret_cast<const void*>(rmsnorm_kernel<1024, 4>)
                     : groups <= 256 || (groups > 1024 && last_empty) ? reinterpret_cast<const void*>(rmsnorm_kernel<256, 1>)
                     : groups <= 512                                  ? reinterpret_cast<const void*>(rmsnorm_kernel<256, 2>)
                                                                      : reinterpret_cast<const void*>(rmsnorm_kernel<256, 4>);
    return launch_pdl(fn, dim3(unsigned(M)), dim3(unsigned(nt)), 0, s, args);
}

cudaError_t launch_rope(uint16_t* x, int64_t n_heads, uint16_t* x2, int64_t n_heads2, int64_t M,
                        int64_t head_dim, int64_t pos0, double base, cudaStream_t s) {
    RopeParams p;
    p.x = reinterpret_cast<__nv_bfloat16*>(x);
    p.x2 = reinterpret_cast<__nv_bfloat16*>(x2);
    p.pos0 = pos0;
    p.n_heads = int(n_heads);
    p.n_heads2 = int(n_heads2);
    p.head_dim = int(head_dim);
    // base^(-2i/d) as the product of two powers, i = 16 j + k: at most 32 calls of pow instead of one
    // per pair, within two roundings of fp64
    double coarse[kRopeMaxPairs / 16], fine[16];
    const int half_d = int(head_dim / 2);
    for (int j = 0; 16 * j < half_d; ++j) coarse[j] = std::pow(base, -32.0 * double(j) / double(head_dim));
    for (int k = 0; k < 16 && k < half_d; ++k) fine[k] = std::pow(base, -2.0 * double(k) / double(head_dim));
    for (int i = 0; i < half_d; ++i) {
        const double v = coarse[i >> 4] * fine[i & 15];
        p.inv_hi[i] = float(v);
        p.inv_lo[i] = float(v - double(p.inv_hi[i]));
    }
    // Pairs per thread: the widest access that divides a head's half (both halves then start on
    // its boundary), fewer while that leaves the SMs short of threads.
    const int64_t half = head_dim / 2, pairs = M * (n_heads + n_heads2) * half;
    int vec = half % 8 == 0 ? 8 : half % 4 == 0 ? 4 : half % 2 == 0 ? 2 : 1;
    while (vec > 1 && pairs / vec < int64_t(152) * 256) vec /= 2;
    p.units = pairs / vec;
    const int64_t blocks = std::min<int64_t>((p.units + 255) / 256, 152 * 8);
    // (the frequencies rise or fall with i, as the base is below or above one)
    const bool large = double(pos0 + M) * std::max(p.inv_hi[0], p.inv_hi[half_d - 1]) >= 4096.0;
    void* args[] = {&p};
    return launch_pdl(large ? rope_fn<true>(vec) : rope_fn<false>(vec), dim3(unsigned(blocks)), dim3(256), 0, s, args);
}

cudaError_t launch_attention(const uint16_t* Q, const uint16_t* K0, const uint16_t* V0, int64_t n0,
                             const uint16_t* K1, const uint16_t* V1, int64_t n1, uint16_t* O,
                             int64_t M, int64_t H, int64_t Hk, int64_t D, float scale, cudaStream_t s) {
    AttnParams p;
    p.Q = reinterpret_cast<const __nv_bfloat16*>(Q);
    p.K0 = reinterpret_cast<const __nv_bfloat16*>(K0);
    p.V0 = reinterpret_cast<const __nv_bfloat16*>(V0);
    p.K1 = reinterpret_cast<const __nv_bfloat16*>(K1);
    p.V1 = reinterpret_cast<const __nv_bfloat16*>(V1);
    p.O = reinterpret_cast<__nv_bfloat16*>(O);
    p.n0 = n0;
    p.n1 = n1;
    p.M = int(M);
    p.H = int(H);
    p.Hk = int(Hk);
    p.scale_log2 = float(double(scale) * 1.4426950408889634);
    return D == 64 ? launch_attention_d<64>(p, s) : launch_attention_d<128>(p, s);
}

}  // namespace emb
