// GEMV for small token counts (action-token decode, M = 1; a few tokens, M = 2..16), and the
// tensor-core kernel for an action chunk (M = 17..64).
//
// The paper's batch-1 setting (Section 3.1, challenge 2) makes every linear layer a
// matrix-vector product whose cost is reading the packed weights once from HBM.
// Five kernels:
//   * the chunk kernel (M = 17..64, K >= 1024; described at its definition);
//   * the tensor-core kernel (M = 2..16, and long rows at M = 1): dot products on mma.sync with
//     the codes exact in bf16 (described at its definition);
//   * the staged kernel (large layers with short rows at M = 1): each CTA pulls one
//     tile of rows plus its activations into shared memory with cp.async.bulk, so many
//     bytes are in flight per SM and the next layer's tiles load during this layer's
//     tail (programmatic dependent launch);
//   * the ring kernel (large Q8_0 and Q6_0 layers with long rows at M = 1): activations in
//     registers, rows through a ring of bulk copies;
//   * the register kernel (what is left: small layers, rows that the others do not take): one CTA
//     owns R consecutive weight rows; its NT threads split K in 16-byte units (a Q8_0 unit is
//     16 codes, half a block; a Q4_0 unit is one whole 32-code block; a warp reads 512
//     contiguous bytes), load codes with 128-bit non-allocating loads one unit ahead
//     (register double buffering) and reduce with warp shuffles, then across warps in
//     shared memory.
// The last three dequantise in registers with exact integer->float "magic number"
// conversions followed by packed fp32x2 FMAs (FFMA2). Every reduction runs in a fixed
// order, so results are deterministic. Weights are fetched before griddepcontrol.wait (within a
// call they never depend on an earlier launch; the register kernel uses non-coherent streaming
// loads), but by a call's first launch, behind work that may have written them, after it (the register
// kernel: with ordinary loads). X is read with ordinary (coherent, L1-cached) loads and Y written only
// after the wait: the previous launch may have just written X, and its writes are then visible to them.
// Up to kMaxGroup matrices that read the same X (q/k/v or gate/up) share one launch.
#include <algorithm>
#include <atomic>
#include <cmath>

#include "dequant_dot.cuh"
#include "ptx.cuh"

namespace emb {
namespace {

using dq::dot_q4_unit;
using dq::dot_q6_unit;
using dq::dot_q8_unit;
using dq::hi_bf16;
using dq::lo_bf16;

// cudaFuncSetAttribute(MaxDynamicSharedMemorySize) once per kernel and device (the call is
// idempotent, and threads may race to make it).
template <typename K>
cudaError_t allow_smem(K* kernel, int bytes, std::atomic<uint64_t>& done) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const uint64_t bit = dev >= 0 && dev < 64 ? uint64_t(1) << dev : 0;
    if (bit && (done.load(std::memory_order_relaxed) & bit)) return cudaSuccess;
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e == cudaSuccess) done.fetch_or(bit, std::memory_order_relaxed);
    return e;
}

struct GemvParams {
    const uint8_t* codes[kMaxGroup];
    const uint8_t* high[kMaxGroup];  // Q6_0: 2-bit high plane of each matrix
    const __half* scales[kMaxGroup];
    void* Y[kMaxGroup];              // as the epilogue says
    int32_t N[kMaxGroup];
    int32_t tile0[kMaxGroup + 1];  // first row tile of each matrix (prefix sums)
    int32_t n_mats;
    int32_t M, K, ldS, U;          // U = 16-byte code units per row
    int32_t epi;                   // emb_epilogue (gated: R even, gate/up row pairs)
    int32_t wait_first;            // 1: nothing is read before griddepcontrol.wait
    const __nv_bfloat16* X;
};

// Codes, read once. COHERENT: by ordinary loads, since the launch before may have written them while
// this grid was already resident; non-coherent ones are for data that nobody writes in its lifetime.
template <bool COHERENT>
__device__ __forceinline__ uint4 ld_stream_u4(const void* p) {
    uint4 v;
    if constexpr (COHERENT)
        asm volatile("ld.global.L1::no_allocate.v4.u32 {%0, %1, %2, %3}, [%4];"
                     : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                     : "l"(p));
    else
        asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0, %1, %2, %3}, [%4];"
                     : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                     : "l"(p));
    return v;
}
template <bool COHERENT>
__device__ __forceinline__ uint2 ld_stream_u2(const void* p) {
    uint2 v;
    if constexpr (COHERENT)
        asm volatile("ld.global.L1::no_allocate.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "l"(p));
    else
        asm volatile("ld.global.nc.L1::no_allocate.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "l"(p));
    return v;
}

__device__ __forceinline__ void griddep_wait() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
}
__device__ __forceinline__ void griddep_launch_dependents() {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// One 16-byte unit of codes (Q6_0: plus its 8 bytes of high bits) times its activations.
template <int FMT>
__device__ __forceinline__ float dot_unit(const uint4 c, const uint2 h, const float* x) {
    if constexpr (FMT == EMB_Q8_0) return dot_q8_unit(c, x);
    else if constexpr (FMT == EMB_Q4_0) return dot_q4_unit(c, x);
    else return dot_q6_unit(c, h, x);
}

// PF > 1 (M = 1 only, U <= PF * NT): every unit of the thread is loaded into registers
// before griddepcontrol.wait, so a layer with long rows has all of its weight bytes in
// flight while the previous launch drains; the products are summed in the same order as
// with PF = 1 (bitwise the same results).
// FIRST: nothing is read before griddepcontrol.wait (the previous launch may have written the weights). A
// parameter tested at run time costs every other launch 1 to 3 % (Q8_0 1536 x 4608 2.73 -> 2.78 us).
template <int FMT, int R, int NT, int MT, int PF, bool FIRST>
__global__ void __launch_bounds__(NT) gemv_kernel(const __grid_constant__ GemvParams p) {
    constexpr int UW = (FMT == EMB_Q8_0) ? 16 : 32;  // weights per 16-byte unit
    constexpr int NWARP = NT / 32;
    const int tile = blockIdx.x;
    int g = 0;
#pragma unroll
    for (int i = 1; i < kMaxGroup; ++i)
        if (i < p.n_mats && tile >= p.tile0[i]) g = i;
    const int row0 = (tile - p.tile0[g]) * R;
    const int N = p.N[g];
    const int m0 = blockIdx.y * MT;
    const int t = threadIdx.x;
    const int64_t row_bytes = (FMT == EMB_Q8_0) ? int64_t(p.K) : int64_t(p.K) / 2;
    const uint8_t* cbase = p.codes[g] + int64_t(row0) * row_bytes;
    const uint8_t* hbase = (FMT == EMB_Q6_0) ? p.high[g] + int64_t(row0) * (p.K / 4) : nullptr;
    const __half* sbase = p.scales[g] + int64_t(row0) * p.ldS;
    const int U = p.U;

    if constexpr (FIRST) griddep_wait();  // before the trigger: see ptx::griddep_launch_dependents
    griddep_launch_dependents();
    // the activation rows towards L2 while the previous launch finishes (measured on GB300:
    // cold, they arrive ~2 us after the dependency wait, behind the weight stream); one CTA
    // per row block asks, since every CTA reads the same rows
    if (t == 0 && blockIdx.x == 0)
        ptx::prefetch_l2(p.X + int64_t(m0) * p.K, uint32_t(min(MT, p.M - m0)) * uint32_t(p.K) * 2u);

    uint4 c[R];
    uint2 h[R];  // Q6_0 high bits (unused otherwise)
    float d[R];
    auto load_unit = [&](int u, uint4* cc, uint2* hh, float* dd) {
#pragma unroll
        for (int r = 0; r < R; ++r) {
            if (row0 + r < N) {
                cc[r] = ld_stream_u4<FIRST>(cbase + r * row_bytes + int64_t(u) * 16);
                if constexpr (FMT == EMB_Q6_0) hh[r] = ld_stream_u2<FIRST>(hbase + int64_t(r) * (p.K / 4) + int64_t(u) * 8);
                else hh[r] = make_uint2(0, 0);
                dd[r] = __half2float(sbase[int64_t(r) * p.ldS + ((FMT == EMB_Q8_0) ? (u >> 1) : u)]);
            } else {
                cc[r] = make_uint4(0, 0, 0, 0);
                hh[r] = make_uint2(0, 0);
                dd[r] = 0.0f;
            }
        }
    };

    float acc[R][MT];
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
        for (int j = 0; j < MT; ++j) acc[r][j] = 0.0f;

    if constexpr (PF > 1) {
        static_assert(MT == 1, "whole-row prefetch is for one token");
        uint4 cp[PF][R];
        uint2 hp[PF][R];
        float dp[PF][R];
#pragma unroll
        for (int k = 0; k < PF; ++k)
            if (t + k * NT < U) load_unit(t + k * NT, cp[k], hp[k], dp[k]);
        // weights do not depend on earlier launches; X and Y may
        griddep_wait();
#pragma unroll
        for (int k = 0; k < PF; ++k) {
            const int uk = t + k * NT;
            if (uk >= U) break;
            float x[UW];
            const uint4* xp = reinterpret_cast<const uint4*>(p.X + int64_t(m0) * p.K + int64_t(uk) * UW);
#pragma unroll
            for (int v = 0; v < UW / 8; ++v) {
                const uint4 hx = xp[v];
                x[8 * v + 0] = lo_bf16(hx.x); x[8 * v + 1] = hi_bf16(hx.x);
                x[8 * v + 2] = lo_bf16(hx.y); x[8 * v + 3] = hi_bf16(hx.y);
                x[8 * v + 4] = lo_bf16(hx.z); x[8 * v + 5] = hi_bf16(hx.z);
                x[8 * v + 6] = lo_bf16(hx.w); x[8 * v + 7] = hi_bf16(hx.w);
            }
#pragma unroll
            for (int r = 0; r < R; ++r) acc[r][0] = fmaf(dp[k][r], dot_unit<FMT>(cp[k][r], hp[k][r], x), acc[r][0]);
        }
    }

    int u = (PF > 1) ? U : t;
    if (u < U) load_unit(u, c, h, d);
    // weights do not depend on earlier launches; X and Y may
    if constexpr (PF == 1) griddep_wait();

    for (; u < U; u += NT) {
        uint4 cn[R];
        uint2 hn[R];
        float dn[R];
        const int un = u + NT;
        if (un < U) load_unit(un, cn, hn, dn);
#pragma unroll
        for (int j = 0; j < MT; ++j) {
            const int m = m0 + j;
            if (m >= p.M) break;
            float x[UW];
            const uint4* xp = reinterpret_cast<const uint4*>(p.X + int64_t(m) * p.K + int64_t(u) * UW);
#pragma unroll
            for (int v = 0; v < UW / 8; ++v) {
                const uint4 h = xp[v];
                x[8 * v + 0] = lo_bf16(h.x); x[8 * v + 1] = hi_bf16(h.x);
                x[8 * v + 2] = lo_bf16(h.y); x[8 * v + 3] = hi_bf16(h.y);
                x[8 * v + 4] = lo_bf16(h.z); x[8 * v + 5] = hi_bf16(h.z);
                x[8 * v + 6] = lo_bf16(h.w); x[8 * v + 7] = hi_bf16(h.w);
            }
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const float part = dot_unit<FMT>(c[r], h[r], x);
                acc[r][j] = fmaf(d[r], part, acc[r][j]);
            }
        }
        if (un < U) {
#pragma unroll
            for (int r = 0; r < R; ++r) { c[r] = cn[r]; h[r] = hn[r]; d[r] = dn[r]; }
        }
    }

    __shared__ float red[NWARP][R * MT];
    const int lane = t & 31, warp = t >> 5;
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
        for (int j = 0; j < MT; ++j) {
            float v = acc[r][j];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
            if (lane == 0) red[warp][r * MT + j] = v;
        }
    __syncthreads();
    if (p.epi >= EMB_EPI_GEGLU) {
        // gate row row0 + 2i and up row row0 + 2i + 1 (R is even) give one output
        if (t < (R / 2) * MT) {
            const int i = t / MT, j = t % MT;
            float gate = 0.0f, up = 0.0f;
#pragma unroll
            for (int w = 0; w < NWARP; ++w) {
                gate += red[w][(2 * i) * MT + j];
                up += red[w][(2 * i + 1) * MT + j];
            }
            const int n = row0 + 2 * i, m = m0 + j;
            if (n < N && m < p.M) epi_store_gated(p.epi, p.Y[g], m, n, N, gate, up);
        }
    } else if (t < R * MT) {
        const int r = t / MT, j = t % MT;
        float v = 0.0f;
#pragma unroll
        for (int w = 0; w < NWARP; ++w) v += red[w][t];
        const int n = row0 + r, m = m0 + j;
        if (n < N && m < p.M) epi_store(p.epi, p.Y[g], m, n, N, v);
    }
}

template <int FMT, int R, int NT, int MT, int PF = 1>
cudaError_t launch_one(const GemvParams& p, int grid_x, int grid_y, cudaStream_t s) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid_x, grid_y, 1);
    cfg.blockDim = dim3(NT, 1, 1);
    cfg.dynamicSmemBytes = 0;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return p.wait_first ? cudaLaunchKernelEx(&cfg, gemv_kernel<FMT, R, NT, MT, PF, true>, p)
                        : cudaLaunchKernelEx(&cfg, gemv_kernel<FMT, R, NT, MT, PF, false>, p);
}

template <int FMT, int R, int NT>
cudaError_t dispatch_mt(const GemvParams& p, int grid_x, int M, cudaStream_t s) {
    // Q8_0 rows longer than one pass of the CTA's threads (at most four) are loaded whole
    // before the wait (measured on GB300 on the Gemma-2B decode chain at M = 1, whose down
    // projection 2048 x 16384 took this path before the ring kernel: Q8_0 3899 -> 3987
    // GB/s). Not for Q4_0: its variant needs ~100 registers, halves the resident CTAs and
    // lost (2265 -> 2068).
    if constexpr (FMT == EMB_Q8_0 && R <= 2) {
        if (M == 1 && p.U > NT && p.U <= 4 * NT) return launch_one<FMT, R, NT, 1, 4>(p, grid_x, 1, s);
    }
    if (M == 1) return launch_one<FMT, R, NT, 1>(p, grid_x, 1, s);
    // more tokens (see tc_takes): few rows at M = 2..4, Q6_0 with K % 64 != 0
    if (M == 2) return launch_one<FMT, R, NT, 2>(p, grid_x, 1, s);
    return launch_one<FMT, R, NT, 4>(p, grid_x, (M + 3) / 4, s);
}

template <int FMT, int R>
cudaError_t dispatch_nt(const GemvParams& p, int grid_x, int M, int NT, cudaStream_t s) {
    if (NT == 256) return dispatch_mt<FMT, R, 256>(p, grid_x, M, s);
    if (NT == 128) return dispatch_mt<FMT, R, 128>(p, grid_x, M, s);
    if (NT == 64) return dispatch_mt<FMT, R, 64>(p, grid_x, M, s);
    return dispatch_mt<FMT, R, 32>(p, grid_x, M, s);
}

// Threads per CTA (they split K): about 8 (Q8_0) or 4 (Q4_0) 16-byte units per thread
// and row, 32..128 threads, which amortises the per-thread prologue and reduction on large
// matrices (measured on GB300 at M=1, Q8_0 K=2048: 32 threads 5.6 TB/s, 128 threads
// 4.6 TB/s). Small matrices are latency-bound instead: there the count grows (up to one
// unit per thread, 256 threads) until about 152K threads put every byte in flight at once.
int pick_threads(int U, int fmt, int64_t tiles) {
    const int target = (fmt == EMB_Q8_0) ? U / 8 : U / 4;
    int nt = 32;
    while (nt < 128 && nt < target) nt *= 2;
    while (nt < 256 && nt < U && tiles * nt < int64_t(152) * 1024) nt *= 2;
    return nt;
}


// ------------------------------------------------------------------ staged GEMV
// One CTA owns a tile of TR consecutive rows of one matrix. Its codes (TR rows,
// contiguous in the codes plane) and scales (TR rows of the scales plane, contiguous
// too) arrive in shared memory through two cp.async.bulk copies that a single thread
// issues as soon as the CTA starts -- before griddepcontrol.wait, since weights never
// depend on an earlier launch -- and the CTA's activation rows (MT x K bf16, contiguous
// in X) through a third copy right after the wait. Up to kStageBytes of codes per CTA
// and several CTAs per SM keep far more bytes in flight than register double buffering
// can, and under programmatic dependent launch the next layer's tiles stream in while
// this layer's last CTAs finish. The four warps form a WR x WK grid (WR = 4 / WK): a
// warp owns RW rows of the tile and one K slice of U / WK units; its lanes stride the
// slice in 16-byte units and reuse each activation unit across the warp's RW rows. (M = 1.)
constexpr int kStageWarps = 4;
constexpr int kStageThreads = 32 * kStageWarps;
constexpr int kStageBytes = 16 * 1024;     // codes of one tile, at most
constexpr int kStageXBytes = 32 * 1024;    // activation rows of one CTA, at most
constexpr int kStageHeader = 1152;         // mbarriers (0..15), cross-warp sums (128..1151)

struct StagedParams {
    const uint8_t* codes[kMaxGroup];
    const uint8_t* high[kMaxGroup];  // Q6_0: 2-bit high plane of each matrix
    const __half* scales[kMaxGroup];
    void* Y[kMaxGroup];              // as the epilogue says
    int32_t N[kMaxGroup];
    int32_t tile0[kMaxGroup + 1];  // first tile of each matrix (prefix sums)
    int32_t n_mats;
    int32_t M, K, ldS, U;
    int32_t TR, WK;                // rows per tile, warps along K
    int32_t epi;                   // emb_epilogue (gated: RW and TR even)
    int32_t wait_first;            // 1: nothing is read before griddepcontrol.wait
    const __nv_bfloat16* X;
    int* status;
};

// (MT, the tokens of a CTA, is 1 in every use. The kernel keeps the loop over tokens: with it
// written out, ptxas sinks the code loads to their uses, 55 registers become 48, and Gemma-2B gate/up
// takes 14.9 us instead of 14.4.)
template <int FMT, int RW, int MT, bool FIRST>
__global__ void __launch_bounds__(kStageThreads) gemv_staged_kernel(const __grid_constant__ StagedParams p) {
    constexpr int UW = (FMT == EMB_Q8_0) ? 16 : 32;
    extern __shared__ __align__(128) uint8_t smem[];
    uint64_t* bar_w = reinterpret_cast<uint64_t*>(smem);      // weights landed
    uint64_t* bar_x = reinterpret_cast<uint64_t*>(smem + 8);  // activations landed
    float* red = reinterpret_cast<float*>(smem + 128);         // [WK][TR][MT]
    const int row_bytes = (FMT == EMB_Q8_0) ? p.K : p.K / 2;
    const int high_bytes = (FMT == EMB_Q6_0) ? p.K / 4 : 0;               // Q6_0 high bits per row
    uint8_t* x_s = smem + kStageHeader;                                    // [MT][K] bf16
    uint8_t* codes_s = x_s + MT * p.K * 2;                                 // [TR][row_bytes]
    uint8_t* high_s = codes_s + uint32_t(p.TR) * uint32_t(row_bytes);     // [TR][K/4] (Q6_0)
    uint8_t* scales_b = high_s + uint32_t(p.TR) * uint32_t(high_bytes);   // [TR][ldS] fp16
    const __half* scales_s = reinterpret_cast<const __half*>(scales_b);

    const int tile = blockIdx.x;
    int g = 0;
#pragma unroll
    for (int i = 1; i < kMaxGroup; ++i)
        if (i < p.n_mats && tile >= p.tile0[i]) g = i;
    const int N = p.N[g];
    const int row0 = (tile - p.tile0[g]) * p.TR;
    const int rows = min(p.TR, N - row0);
    const int m0 = blockIdx.y * MT;
    const int mt = min(MT, p.M - m0);  // activation rows of this CTA

    if (threadIdx.x == 0) {
        const uint32_t codes_bytes = uint32_t(rows) * uint32_t(row_bytes);
        const uint32_t hi_bytes = uint32_t(rows) * uint32_t(high_bytes);  // a multiple of 16 (K % 64 == 0)
        const uint32_t scales_bytes = uint32_t(rows) * uint32_t(p.ldS) * 2u;
        ptx::mbar_init(bar_w, 1);
        ptx::mbar_init(bar_x, 1);
        ptx::fence_mbar_init();
        if constexpr (FIRST) ptx::griddep_wait();
        ptx::mbar_arrive_expect_tx(bar_w, codes_bytes + hi_bytes + scales_bytes);
        ptx::bulk_load(codes_s, p.codes[g] + int64_t(row0) * row_bytes, codes_bytes, bar_w);
        if constexpr (FMT == EMB_Q6_0)
            ptx::bulk_load(high_s, p.high[g] + int64_t(row0) * high_bytes, hi_bytes, bar_w);
        ptx::bulk_load(scales_b, p.scales[g] + int64_t(row0) * p.ldS, scales_bytes, bar_w);
        // the activation rows towards L2 while the previous launch finishes (measured on
        // GB300: cold, they land ~2 us after the dependency wait, behind the weight stream);
        // one CTA per row block asks, since every CTA reads the same rows
        if (blockIdx.x == 0) ptx::prefetch_l2(p.X + int64_t(m0) * p.K, uint32_t(mt) * uint32_t(p.K) * 2u);
    }
    if constexpr (FIRST) ptx::griddep_wait();  // every thread before the trigger: see ptx::griddep_launch_dependents
    ptx::griddep_launch_dependents();
    // weights do not depend on earlier launches; X and Y may
    ptx::griddep_wait();
    if (threadIdx.x == 0) {
        const uint32_t x_bytes = uint32_t(mt) * uint32_t(p.K) * 2u;
        ptx::mbar_arrive_expect_tx(bar_x, x_bytes);
        ptx::bulk_load(x_s, p.X + int64_t(m0) * p.K, x_bytes, bar_x);
    }
    __syncthreads();  // the barriers' initialisation is visible to every waiting thread
    // both waits are bounded; the CTA leaves together if any of its threads gave up
    bool ok = ptx::mbar_wait(bar_w, 0, nullptr, p.status, kWaitLimitNs);
    ok = ok && ptx::mbar_wait(bar_x, 0, nullptr, p.status, kWaitLimitNs);
    if (__syncthreads_or(!ok)) return;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int WK = p.WK;
    const int wk = warp % WK, wr = warp / WK;
    const int r0 = wr * RW;                       // first tile row of this warp
    const int Uw = (p.U + WK - 1) / WK;
    const int u_lo = wk * Uw, u_hi = min(p.U, u_lo + Uw);

    float acc[RW][MT];
#pragma unroll
    for (int i = 0; i < RW; ++i)
#pragma unroll
        for (int t = 0; t < MT; ++t) acc[i][t] = 0.0f;

    if (r0 < rows) {
#pragma unroll 2
        for (int u = u_lo + lane; u < u_hi; u += 32) {
            uint4 c[RW];
            uint2 hq[RW];
            float d[RW];
#pragma unroll
            for (int i = 0; i < RW; ++i) {
                const int r = min(r0 + i, rows - 1);  // rows past the tile's end are never stored
                c[i] = *reinterpret_cast<const uint4*>(codes_s + r * row_bytes + u * 16);
                if constexpr (FMT == EMB_Q6_0)
                    hq[i] = *reinterpret_cast<const uint2*>(high_s + r * high_bytes + u * 8);
                else
                    hq[i] = make_uint2(0, 0);
                d[i] = __half2float(scales_s[r * p.ldS + ((FMT == EMB_Q8_0) ? (u >> 1) : u)]);
            }
#pragma unroll
            for (int t = 0; t < MT; ++t) {
                if (t >= mt) break;
                float x[UW];
                const uint4* xp = reinterpret_cast<const uint4*>(x_s + (t * p.K + u * UW) * 2);
#pragma unroll
                for (int v = 0; v < UW / 8; ++v) {
                    const uint4 h = xp[v];
                    x[8 * v + 0] = lo_bf16(h.x); x[8 * v + 1] = hi_bf16(h.x);
                    x[8 * v + 2] = lo_bf16(h.y); x[8 * v + 3] = hi_bf16(h.y);
                    x[8 * v + 4] = lo_bf16(h.z); x[8 * v + 5] = hi_bf16(h.z);
                    x[8 * v + 6] = lo_bf16(h.w); x[8 * v + 7] = hi_bf16(h.w);
                }
#pragma unroll
                for (int i = 0; i < RW; ++i) {
                    const float sdot = dot_unit<FMT>(c[i], hq[i], x);
                    acc[i][t] = fmaf(d[i], sdot, acc[i][t]);
                }
            }
        }
    }

    float mine = 0.0f;
#pragma unroll
    for (int i = 0; i < RW; ++i)
#pragma unroll
        for (int t = 0; t < MT; ++t) {
            float v = acc[i][t];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
            if (lane == i * MT + t) mine = v;
        }
    const bool gated = p.epi >= EMB_EPI_GEGLU;
    if (WK == 1) {
        // gated: the up row's sum sits MT lanes further on (RW is even)
        const float up = __shfl_down_sync(0xffffffffu, mine, MT);
        if (lane < RW * MT) {
            const int r = r0 + lane / MT, t = lane % MT;
            if (r < rows && t < mt) {
                if (!gated) epi_store(p.epi, p.Y[g], m0 + t, row0 + r, N, mine);
                else if ((r & 1) == 0) epi_store_gated(p.epi, p.Y[g], m0 + t, row0 + r, N, mine, up);
            }
        }
        return;
    }
    if (lane < RW * MT) red[(wk * p.TR + r0 + lane / MT) * MT + lane % MT] = mine;
    __syncthreads();
    // add the K slices in slice order
    if (gated) {
        for (int e = threadIdx.x; e < (rows / 2) * MT; e += kStageThreads) {
            const int i = e / MT, t = e % MT;
            float gate = 0.0f, up = 0.0f;
            for (int k = 0; k < WK; ++k) {
                gate += red[(k * p.TR + 2 * i) * MT + t];
                up += red[(k * p.TR + 2 * i + 1) * MT + t];
            }
            if (t < mt) epi_store_gated(p.epi, p.Y[g], m0 + t, row0 + 2 * i, N, gate, up);
        }
        return;
    }
    for (int e = threadIdx.x; e < rows * MT; e += kStageThreads) {
        float v = 0.0f;
        for (int k = 0; k < WK; ++k) v += red[k * p.TR * MT + e];
        const int r = e / MT, t = e % MT;
        if (t < mt) epi_store(p.epi, p.Y[g], m0 + t, row0 + r, N, v);
    }
}

template <int FMT, int RW, bool FIRST>
cudaError_t launch_staged_one(const StagedParams& p, int tiles, size_t smem, cudaStream_t s) {
    static_assert(kStageHeader + kStageXBytes + kStageBytes + kStageBytes / 8 <= 227 * 1024, "smem");
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(tiles, 1, 1);
    cfg.blockDim = dim3(kStageThreads, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (smem > 48 * 1024) {
        static std::atomic<uint64_t> done{0};
        const cudaError_t e = allow_smem(gemv_staged_kernel<FMT, RW, 1, FIRST>,
                                         int(kStageHeader + kStageXBytes + kStageBytes + kStageBytes / 8), done);
        if (e != cudaSuccess) return e;
    }
    return cudaLaunchKernelEx(&cfg, gemv_staged_kernel<FMT, RW, 1, FIRST>, p);
}

template <int FMT>
cudaError_t launch_staged_rw(const StagedParams& p, int RW, int tiles, size_t smem, cudaStream_t s) {
    if (p.wait_first)
        return RW == 4 ? launch_staged_one<FMT, 4, true>(p, tiles, smem, s)
             : RW == 2 ? launch_staged_one<FMT, 2, true>(p, tiles, smem, s)
                       : launch_staged_one<FMT, 1, true>(p, tiles, smem, s);
    return RW == 4 ? launch_staged_one<FMT, 4, false>(p, tiles, smem, s)
         : RW == 2 ? launch_staged_one<FMT, 2, false>(p, tiles, smem, s)
                   : launch_staged_one<FMT, 1, false>(p, tiles, smem, s);
}

// Tile shape: rows per warp RW and warps along K WK (TR = RW * 4 / WK rows per tile),
// in order of preference: Q8_0 favours activation reuse (4 rows per warp), Q4_0 unsplit
// K. Take the first whose tile fits `tile_bytes` and that makes at least 4 tiles per
// SM; for matrices too small for that, the fitting shape with the most tiles. A warp's
// K slice keeps at least 32 units (one per lane). Returns false when no tile fits.
// Measured on GB300 at M = 1 (graph-replayed chains): 16 KB tiles beat 32 KB ones by
// 3-6% (a shorter CTA lifetime shortens each launch's tail), e.g. Q8_0 32768 x 2048:
// 14.9 us (8 rows) vs 15.8 us (16 rows).
bool pick_stage_shape(int fmt, int64_t rows_total, int64_t row_bytes, int U, int64_t tile_bytes,
                      bool even_rows, int& RW, int& WK) {
    static const int kQ8[5][2] = {{4, 1}, {4, 2}, {4, 4}, {2, 4}, {1, 4}};
    static const int kQ4[7][2] = {{4, 1}, {2, 1}, {1, 1}, {4, 2}, {4, 4}, {2, 4}, {1, 4}};
    const int n = (fmt == EMB_Q8_0) ? 5 : 7;
    bool found = false;
    for (int i = 0; i < n; ++i) {
        const int rw = (fmt == EMB_Q8_0) ? kQ8[i][0] : kQ4[i][0];
        const int wk = (fmt == EMB_Q8_0) ? kQ8[i][1] : kQ4[i][1];
        const int64_t tr = int64_t(rw) * kStageWarps / wk;
        if (tr * row_bytes > tile_bytes) continue;
        if (wk > 1 && U / wk < 32) continue;
        if (even_rows && (rw & 1)) continue;  // gated epilogues pair rows inside a warp
        RW = rw;
        WK = wk;
        found = true;
        if (rows_total / tr >= 4 * 152) break;
    }
    return found;
}

// Which layers take the staged path (measured on GB300, graph-replayed chains of one
// shape). Small layers are latency-bound: there the register kernel, whose threads issue
// their loads directly, finishes sooner than a bulk-copy round trip (5.6 MB q/k/v at
// M = 1: 2.1 us register, 3.2 us staged). Long rows at M = 1 leave a staged CTA one or two
// rows and re-stage the whole activation row per CTA; the register kernel with 2 rows
// per CTA is faster there (Q8_0 2048 x 16384: 9.6 us register, 12.0 us staged). Short
// rows favour the staged path (Q4_0 32768 x 2048: 13.4 us staged, 15.1 us register).
constexpr int64_t kStageMinBytes = 12ll << 20;
constexpr int64_t kStageMaxRowBytesM1 = 6 * 1024;

bool launch_staged(const GroupRef& g, bool pdl, int* status, cudaStream_t s, cudaError_t& err) {
    const int64_t row_bytes = (g.fmt == EMB_Q8_0) ? g.K : g.K / 2;
    // Q6_0 rows also carry K/4 bytes of high bits, copied as a second contiguous block
    // (16-byte multiples need K % 64 == 0; other K take the register path)
    const int64_t high_bytes = (g.fmt == EMB_Q6_0) ? g.K / 4 : 0;
    if (g.fmt == EMB_Q6_0 && g.K % 64 != 0) return false;
    const int64_t weight_row_bytes = row_bytes + high_bytes;
    const int U = int((g.fmt == EMB_Q8_0) ? g.K / 16 : g.K / 32);
    if (g.M != 1 || g.K * 2 > kStageXBytes) return false;
    int64_t rows = 0;
    for (int i = 0; i < g.n_mats; ++i) rows += g.mats[i].N;
    if (rows * weight_row_bytes < kStageMinBytes) return false;
    if (weight_row_bytes > kStageMaxRowBytesM1) return false;
    int RW = 0, WK = 0;
    if (!pick_stage_shape(g.fmt, rows, weight_row_bytes, U, kStageBytes, g.epi >= EMB_EPI_GEGLU, RW, WK))
        return false;
    StagedParams p = {};
    const int TR = RW * kStageWarps / WK;
    int tiles = 0;
    for (int i = 0; i < g.n_mats; ++i) {
        p.high[i] = g.mats[i].high;
        p.codes[i] = g.mats[i].codes;
        p.scales[i] = g.mats[i].scales;
        p.Y[i] = g.mats[i].Y;
        p.N[i] = int32_t(g.mats[i].N);
        p.tile0[i] = tiles;
        tiles += int((g.mats[i].N + TR - 1) / TR);
    }
    p.tile0[g.n_mats] = tiles;
    p.n_mats = g.n_mats;
    p.M = int32_t(g.M);
    p.K = int32_t(g.K);
    p.ldS = int32_t(g.ldS);
    p.U = U;
    p.TR = TR;
    p.WK = WK;
    p.epi = g.epi;
    p.X = g.X;
    p.wait_first = pdl ? 0 : 1;
    p.status = status;
    const size_t smem = kStageHeader + size_t(g.K) * 2 + size_t(TR) * size_t(weight_row_bytes + g.ldS * 2);
    err = g.fmt == EMB_Q8_0   ? launch_staged_rw<EMB_Q8_0>(p, RW, tiles, smem, s)
          : g.fmt == EMB_Q6_0 ? launch_staged_rw<EMB_Q6_0>(p, RW, tiles, smem, s)
                              : launch_staged_rw<EMB_Q4_0>(p, RW, tiles, smem, s);
    return true;
}


// ------------------------------------------------------------------ tensor-core GEMV
// A few tokens (M = 2..16). With M tokens per weight the FFMA2 dot products, not HBM, bound the
// kernels above (M = 4: ~6 instructions per weight). Here they run on mma.sync m16n8k16 (bf16 x
// bf16 -> fp32): 16 weight rows are the MMA's M side, the tokens its eight columns (two MMAs for
// M > 8), so up to eight tokens cost what one does and the CUDA cores only turn codes into bf16:
// codes are small integers, exact in bf16, and every product is exact in fp32. A 32-weight block
// is two MMAs into one fragment, which is then scaled by the block's fp32 scale as in the plain
// definition; four such sums (two for M > 8) alternate by block and are added at the end, the warps' sums pairwise,
// all in a fixed order: results are deterministic.
//
// A row tile is 16 rows of one matrix; a CTA walks row tiles blockIdx.x, + gridDim.x, ... Each of
// its eight warps (sixteen for long rows that give an SM one tile, two for many tiles of short rows)
// takes every eighth 256-k chunk of the tile's rows and streams its chunks through a ring of its own in shared memory
// with cp.async (whole 128-byte lines per row, XOR-swizzled 16-byte granules so that fragment loads
// are conflict-free): no barrier between warps until a tile's sums are added. The first ring's
// worth is issued before griddepcontrol.wait; the activations come by ordinary cached loads after.
//
// Fragment mapping (any permutation of K inside a block is valid as long as A and B use the same
// one): lane (g, t) = (lane / 4, lane % 4) holds tile rows rho(g) and rho(g) + 8
// (rho is the identity but for Q8_0, where 0, 2, 4, 6, 1, 3, 5, 7 puts a half warp's loads into
// distinct banks) and of each block the codes 8t .. 8t + 7: 8 bytes of Q8_0, or one nibble of each byte
// of words 2(t & 1) and 2(t & 1) + 1. MMA 0 takes codes (8t, 8t + 1) as k slots (2t, 2t + 1) and
// (8t + 2, 8t + 3) as (2t + 8, 2t + 9), MMA 1 the other four; the activations are token g's
// x[8t .. 8t + 7], one 16-byte load.
// What bounds it: the codes-to-bf16 arithmetic (2 to 3 instructions per weight, on the pipe that
// also permutes bytes) and, for few rows, latency: Q6_0 32768 x 2048 at M = 4 15.4 us against 8.1
// for its bytes. Without the shared-memory ring (fragments loaded from global memory directly,
// 32 bytes per row and instruction) the same layer took 23 us, with or without a persistent grid.
constexpr int kTcRows = 16;
constexpr int kTcBlocks = 8;       // 32-weight blocks of a chunk (16 bytes of scales per row)
constexpr int kTcMaxM = 16;

struct TcParams {
    const uint8_t* codes[kMaxGroup];
    const uint8_t* high[kMaxGroup];  // Q6_0: 2-bit high plane of each matrix
    const __half* scales[kMaxGroup];
    void* Y[kMaxGroup];              // as the epilogue says
    int32_t N[kMaxGroup];
    int32_t tile0[kMaxGroup + 1];  // first row tile of each matrix (prefix sums)
    int32_t n_mats;
    int32_t M, K, ldS;
    int32_t epi;                   // emb_epilogue
    int32_t wait_first;            // 1: nothing is read before griddepcontrol.wait
    const __nv_bfloat16* X;
};

__device__ __forceinline__ void mma_bf16_16816(float (&d)[4], const uint32_t (&a)[4], uint32_t b0,
                                               uint32_t b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, "
        "{%8, %9}, {%0, %1, %2, %3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint32_t sub_bf16x2(uint32_t a, uint32_t b) {
    const __nv_bfloat162 r = __hsub2(*reinterpret_cast<const __nv_bfloat162*>(&a),
                                     *reinterpret_cast<const __nv_bfloat162*>(&b));
    return *reinterpret_cast<const uint32_t*>(&r);
}
// Bytes 0, 1 (LO) or 2, 3 of v, each below 128, as the bf16 pair 128 + byte (exact: the byte is the
// whole 7-bit fraction of 0x4300).
template <bool LO>
__device__ __forceinline__ uint32_t bytes_128(uint32_t v) {
    return __byte_perm(v, 0x43434343u, LO ? 0x4140 : 0x4342);
}
// Four signed bytes -> bf16 pairs (codes 0, 1) and (2, 3): q = (128 + (q & 127)) - (128 or 256 by
// its sign bit), both of which are bf16 0x4300 with the masked byte as fraction and exponent bits.
__device__ __forceinline__ void q8_pairs(uint32_t v, uint32_t& p01, uint32_t& p23) {
    const uint32_t m = v & 0x7F7F7F7Fu, s = v & 0x80808080u;
    p01 = sub_bf16x2(bytes_128<true>(m), bytes_128<true>(s));
    p23 = sub_bf16x2(bytes_128<false>(m), bytes_128<false>(s));
}

__device__ __forceinline__ uint2 ld_shared_u2(uint32_t a) {
    uint2 v;
    asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(a));
    return v;
}
__device__ __forceinline__ float ld_shared_half(uint32_t a) {
    uint16_t v;
    asm volatile("ld.shared.u16 %0, [%1];" : "=h"(v) : "r"(a));
    return __half2float(__ushort_as_half(v));
}

__device__ __forceinline__ void cp_async16(uint32_t saddr, const void* g, bool ok) {
    asm volatile("cp.async.cg.shared.global.L2::128B [%0], [%1], 16, %2;" ::"r"(saddr), "l"(g), "r"(ok ? 16 : 0)
                 : "memory");
}

// One stage of a warp's ring: 16 rows x 256 k of codes, then (Q6_0) high bits, then scales.
template <int FMT>
struct TcStage {
    static constexpr int kCodes = kTcRows * (FMT == EMB_Q8_0 ? 256 : 128);
    static constexpr int kHigh = FMT == EMB_Q6_0 ? kTcRows * 64 : 0;
    static constexpr int kBytes = kCodes + kHigh + kTcRows * 16;
};
// Matrix of a row tile.
__device__ __forceinline__ int tc_mat_of(const TcParams& p, int tile) {
    int gm = 0;
#pragma unroll
    for (int i = 1; i < kMaxGroup; ++i)
        if (i < p.n_mats && tile >= p.tile0[i]) gm = i;
    return gm;
}

// Issue the copies of one chunk (256 k from block kb0) of a row tile into a stage: blocks past the
// row are zero codes with zero scales (the scale row is zero-padded to eight), rows past N read row
// N - 1 (never stored).
template <int FMT>
__device__ __forceinline__ void tc_issue(const TcParams& p, int tile, int kb0, uint32_t st, int lane) {
    using St = TcStage<FMT>;
    const int nb = p.K / kQBlock;
    const int64_t row_bytes = FMT == EMB_Q8_0 ? int64_t(p.K) : int64_t(p.K) / 2;
    const int gm = tc_mat_of(p, tile);
    const int row0 = (tile - p.tile0[gm]) * kTcRows, last = p.N[gm] - 1;
    constexpr int kG = FMT == EMB_Q8_0 ? 16 : 8;  // 16-byte granules of a row's codes
    const int c = lane % kG, kbg = kb0 + (FMT == EMB_Q8_0 ? c >> 1 : c);  // the granule's block
#pragma unroll
    for (int i = 0; i < kTcRows * kG / 32; ++i) {
        const int r = i * (32 / kG) + lane / kG;
        const uint8_t* src = p.codes[gm] + int64_t(min(row0 + r, last)) * row_bytes +
                             (kbg < nb ? int64_t(kb0) * (FMT == EMB_Q8_0 ? 32 : 16) + c * 16 : 0);
        cp_async16(st + r * (kG * 16) + ((c ^ (r & 7)) << 4), src, kbg < nb);
    }
    if constexpr (FMT == EMB_Q6_0) {
        const int ch = lane & 3;
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const int r = 8 * i + (lane >> 2);
            const bool ok = kb0 + 2 * ch < nb;  // nb is even (K % 64 == 0)
            const uint8_t* src =
                p.high[gm] + int64_t(min(row0 + r, last)) * (p.K / 4) + (ok ? int64_t(kb0) * 8 + ch * 16 : 0);
            cp_async16(st + St::kCodes + r * 64 + ((ch ^ ((r >> 1) & 3)) << 4), src, ok);
        }
    }
    if (lane < kTcRows) {
        const __half* src = p.scales[gm] + int64_t(min(row0 + lane, last)) * p.ldS + (kb0 < nb ? kb0 : 0);
        cp_async16(st + St::kCodes + St::kHigh + lane * 16, src, kb0 < nb);
    }
}

// The tile row whose fragment lane (g, t) holds as MMA row g (+ 8 for MMA row g + 8).
template <int FMT>
__device__ __forceinline__ int tc_row(int g) {
    return FMT == EMB_Q8_0 ? (2 * g) % 7 + (g == 7 ? 7 : 0) : g;  // rho(g): 0, 2, 4, 6, 1, 3, 5, 7
}
// Codes 8t .. 8t + 7 of block i of a stage's row, one per byte (Q8_0 signed, else unsigned).
template <int FMT>
__device__ __forceinline__ uint2 tc_codes(uint32_t st, int row, int i, int t) {
    if constexpr (FMT == EMB_Q8_0) {
        return ld_shared_u2(st + row * 256 + (((2 * i + (t >> 1)) ^ (row & 7)) << 4) + (t & 1) * 8);
    } else {
        // words 2(t & 1), 2(t & 1) + 1 of the block, low nibbles for t < 2, high ones for t >= 2
        const uint32_t m = 0x0F0F0F0Fu;
        uint2 w = ld_shared_u2(st + row * 128 + ((i ^ (row & 7)) << 4) + (t & 1) * 8);
        w.x = (w.x >> (4 * (t >> 1))) & m;
        w.y = (w.y >> (4 * (t >> 1))) & m;
        if constexpr (FMT == EMB_Q6_0) {
            // the high bits of word j are in high word j & 1, shifted by 2 (j >> 1), by 4 more for
            // the high nibbles' codes
            const uint2 h = ld_shared_u2(st + TcStage<FMT>::kCodes + row * 64 + (((i >> 1) ^ ((row >> 1) & 3)) << 4) + (i & 1) * 8);
            const int sh = 2 * (t & 1) + 4 * (t >> 1);
            w.x |= ((h.x >> sh) & 0x03030303u) << 4;
            w.y |= ((h.y >> sh) & 0x03030303u) << 4;
        }
        return w;
    }
}

// Ring depth: three stages, two where the sums of sixteen tokens would leave an SM one CTA.
template <int FMT, int NT, int NW>
constexpr int kTcDepth = FMT == EMB_Q8_0 && NT == 2 && NW == 8 ? 2 : 3;
template <int FMT, int NT, int NW>
constexpr int kTcSmem = NW * kTcDepth<FMT, NT, NW> * TcStage<FMT>::kBytes;

// COMP: the sums of a chunk are added to a compensated total (TwoSum), so the fp32 error does not grow
// with the number of chunks that a warp adds up (see launch_tc_fmt).
template <int FMT, int NT, int NW, bool COMP>
__global__ void __launch_bounds__(32 * NW, 16 / NW) gemv_tc_kernel(const __grid_constant__ TcParams p) {
    using St = TcStage<FMT>;
    constexpr int kTcStages = kTcDepth<FMT, NT, NW>;
    constexpr int kBufs = NW < 16 ? 2 : 1;  // (sixteen warps: one tile per CTA)
    extern __shared__ __align__(128) uint8_t smem[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int g = lane >> 2, t = lane & 3;
    const int nb = p.K / kQBlock;
    const int tiles = p.tile0[p.n_mats];
    const uint32_t ring = ptx::smem_u32(smem) + warp * kTcStages * St::kBytes;
    if (p.wait_first) griddep_wait();  // before the trigger: see ptx::griddep_launch_dependents
    griddep_launch_dependents();
    // this warp's chunks of all the CTA's tiles, in order; the next one to issue
    const int stride = NW * kTcBlocks;                 // blocks between a warp's chunks of a tile
    int it_tile = blockIdx.x, it_base = 0;
    auto issue_next = [&](int stage) {
        if (it_tile < tiles) {
            tc_issue<FMT>(p, it_tile, it_base + warp * kTcBlocks, ring + stage * St::kBytes, lane);
            it_base += stride;
            if (it_base >= nb) {
                it_base = 0;
                it_tile += gridDim.x;
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
#pragma unroll
    for (int i = 0; i < kTcStages; ++i) issue_next(i);
    if (threadIdx.x == 0 && blockIdx.x == 0) ptx::prefetch_l2(p.X, uint32_t(p.M) * uint32_t(p.K) * 2u);
    // weights do not depend on earlier launches; X and Y may
    griddep_wait();

    // activation fragments of a block, by token n-tile: token 8 * nt + g
    const __nv_bfloat16* xr[NT];
    bool has[NT];
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) {
        has[nt] = 8 * nt + g < p.M;
        xr[nt] = p.X + int64_t(has[nt] ? 8 * nt + g : 0) * p.K;
    }
    auto load_x = [&](int kb, int nt, uint32_t (&b)[4]) {
        b[0] = b[1] = b[2] = b[3] = 0u;
        if (!has[nt] || kb >= nb) return;
        const uint4 v = *reinterpret_cast<const uint4*>(xr[nt] + kb * 32 + 8 * t);
        b[0] = v.x; b[1] = v.y; b[2] = v.z; b[3] = v.w;
    };

    constexpr int kAcc = NT == 1 ? 4 : 2;  // sums that alternate by block
    float acc[kAcc][NT][4] = {};
    float tot[COMP ? NT : 1][4], rest[COMP ? NT : 1][4];
    auto acc_sum = [&](int nt, int e) {
        float v = acc[0][nt][e] + acc[1][nt][e];
        if constexpr (kAcc == 4) v += acc[2][nt][e] + acc[3][nt][e];
        return v;
    };
    auto acc_clear = [&] {
#pragma unroll
        for (int i = 0; i < kAcc; ++i)
#pragma unroll
            for (int nt = 0; nt < NT; ++nt) acc[i][nt][0] = acc[i][nt][1] = acc[i][nt][2] = acc[i][nt][3] = 0.0f;
    };
    const int ra = tc_row<FMT>(g);
    auto compute = [&](int kb0, uint32_t st) {
        const uint32_t sc = st + St::kCodes + St::kHigh + ra * 16;
#pragma unroll
        for (int i = 0; i < kTcBlocks; ++i) {
            uint32_t a0[4], a1[4];  // A fragments: {row ra slots 2t, row ra + 8, row ra slots 2t + 8, row ra + 8}
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                const uint2 v = tc_codes<FMT>(st, ra + 8 * r, i, t);
                if constexpr (FMT == EMB_Q8_0) {
                    q8_pairs(v.x, a0[r], a0[2 + r]);
                    q8_pairs(v.y, a1[r], a1[2 + r]);
                } else {
                    constexpr uint32_t kOff = FMT == EMB_Q4_0 ? 0x43084308u : 0x43204320u;  // 128 + 8, 128 + 32
                    a0[r] = sub_bf16x2(bytes_128<true>(v.x), kOff);
                    a0[2 + r] = sub_bf16x2(bytes_128<false>(v.x), kOff);
                    a1[r] = sub_bf16x2(bytes_128<true>(v.y), kOff);
                    a1[2 + r] = sub_bf16x2(bytes_128<false>(v.y), kOff);
                }
            }
            const float da = ld_shared_half(sc + 2 * i), db = ld_shared_half(sc + 8 * 16 + 2 * i);
#pragma unroll
            for (int nt = 0; nt < NT; ++nt) {
                uint32_t b[4];
                load_x(kb0 + i, nt, b);
                // (two sums from zero and one rounded addition: chaining the second MMA onto the first
                // costs 5 % in accuracy)
                float d0[4] = {0.0f, 0.0f, 0.0f, 0.0f}, d1[4] = {0.0f, 0.0f, 0.0f, 0.0f};
                mma_bf16_16816(d0, a0, b[0], b[1]);
                mma_bf16_16816(d1, a1, b[2], b[3]);
                float(&ac)[4] = acc[i % kAcc][nt];
                ac[0] = fmaf(da, d0[0] + d1[0], ac[0]);
                ac[1] = fmaf(da, d0[1] + d1[1], ac[1]);
                ac[2] = fmaf(db, d0[2] + d1[2], ac[2]);
                ac[3] = fmaf(db, d0[3] + d1[3], ac[3]);
            }
        }
        if constexpr (COMP) {
#pragma unroll
            for (int nt = 0; nt < NT; ++nt)
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const float a = tot[nt][e], c = acc_sum(nt, e), sum = __fadd_rn(a, c), b = __fsub_rn(sum, a);
                    rest[nt][e] += __fadd_rn(__fsub_rn(a, __fsub_rn(sum, b)), __fsub_rn(c, b));
                    tot[nt][e] = sum;
                }
            acc_clear();
        }
    };
    __shared__ float red[kBufs][NW][8 * NT][kTcRows];
    int buf = 0, stage = 0;
    for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x, buf = (buf + 1) % kBufs) {
        acc_clear();
        if constexpr (COMP) {
#pragma unroll
            for (int nt = 0; nt < NT; ++nt)
#pragma unroll
                for (int e = 0; e < 4; ++e) tot[nt][e] = rest[nt][e] = 0.0f;
        }
        for (int base = 0; base < nb; base += stride) {
            asm volatile("cp.async.wait_group %0;" ::"n"(kTcStages - 1) : "memory");
            __syncwarp();  // every lane's copies of this chunk have landed
            const int kb0 = base + warp * kTcBlocks;
            if (kb0 < nb) compute(kb0, ring + stage * St::kBytes);
            __syncwarp();  // every lane has read it
            issue_next(stage);
            stage = stage + 1 == kTcStages ? 0 : stage + 1;
        }
        // acc[.][nt][0, 1]: row ra, tokens 8 nt + 2t, + 1; [2, 3]: row ra + 8. (Two
        // buffers: a buffer is written again only after the barrier of the tile between.)
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
            float v[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                if constexpr (COMP)
                    // an infinite or NaN total stays as it is: its rounding errors are NaN
                    v[e] = fabsf(tot[nt][e]) <= 3.402823466e+38f ? tot[nt][e] + rest[nt][e] : tot[nt][e];
                else
                    v[e] = acc_sum(nt, e);
            }
            red[buf][warp][8 * nt + 2 * t][ra] = v[0];
            red[buf][warp][8 * nt + 2 * t + 1][ra] = v[1];
            red[buf][warp][8 * nt + 2 * t][ra + 8] = v[2];
            red[buf][warp][8 * nt + 2 * t + 1][ra + 8] = v[3];
        }
        __syncthreads();
        const int m = threadIdx.x / kTcRows, r = threadIdx.x % kTcRows;  // (two warps: up to four tokens)
        if (m < p.M && m < 8 * NT) {
            const int gm = tc_mat_of(p, tile), N = p.N[gm];
            const int n = (tile - p.tile0[gm]) * kTcRows + r;
            // the warps' sums pairwise (in order, one rounding more per warp adds 20 % of error)
            auto total = [&](int row) {
                float v[NW];
#pragma unroll
                for (int w = 0; w < NW; ++w) v[w] = red[buf][w][m][row];
#pragma unroll
                for (int o = NW / 2; o > 0; o >>= 1)
#pragma unroll
                    for (int w = 0; w < o; ++w) v[w] += v[w + o];
                return v[0];
            };
            const float v = total(r);
            if (p.epi >= EMB_EPI_GEGLU) {
                // gate row n (even) and up row n + 1
                if ((r & 1) == 0 && n < N) epi_store_gated(p.epi, p.Y[gm], m, n, N, v, total(r + 1));
            } else if (n < N) {
                epi_store(p.epi, p.Y[gm], m, n, N, v);
            }
        }
    }
}

template <int FMT, int NT, int NW, bool COMP = false>
cudaError_t launch_tc_one(const TcParams& p, int grid, cudaStream_t s) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid, 1, 1);
    cfg.blockDim = dim3(32 * NW, 1, 1);
    cfg.dynamicSmemBytes = kTcSmem<FMT, NT, NW>;
    cfg.stream = s;
    static std::atomic<uint64_t> done{0};
    const cudaError_t e = allow_smem(gemv_tc_kernel<FMT, NT, NW, COMP>, kTcSmem<FMT, NT, NW>, done);
    if (e != cudaSuccess) return e;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, gemv_tc_kernel<FMT, NT, NW, COMP>, p);
}

template <int FMT>
cudaError_t launch_tc_fmt(const TcParams& p, int tiles, int sms, cudaStream_t s) {
    // long rows whose tiles leave each SM at most one CTA: sixteen warps
    const bool wide = tiles <= sms && p.K > 8 * kTcBlocks * kQBlock;
    const int grid = std::min(tiles, 2 * sms);
    // short rows have fewer chunks than eight warps, and the others idle: pairs of warps on four times as
    // many CTAs once the tiles fill them (us, eight warps / two / the FFMA2 and mma.sync kernels that were here
    // before: 32768 x 512 Q8_0 at M = 2 10.3 / 5.7 / 8.9, 32768 x 768 Q4_0 at M = 4 8.9 / 7.2 / 7.9, 16384 x
    // 1536 Q4_0 at M = 4 7.2 / 5.5 / 6.5; from seven chunks on, or with fewer tiles, eight are faster: 16384 x 1792
    // Q8_0 at M = 3 by 4 %, 8192 x 768 by 27 %, but for nine and ten chunks, whose second pass has one or two
    // of eight warps: 16384 x 2112 Q4_0 at M = 2 eight / two / before 10.2 / 8.7 / 8.2)
    const int chunks = (p.K + kTcBlocks * kQBlock - 1) / (kTcBlocks * kQBlock);
    if (p.M <= 4 && tiles > (chunks <= 2 ? 2 : 6) * sms && (chunks <= 6 || chunks == 9 || chunks == 10))
        return launch_tc_one<FMT, 1, 2>(p, std::min(tiles, 8 * sms), s);
    // Many chunks per warp and up to four tokens (more had the GEMM's rounded operand, 1.7e-3): compensated
    // totals. In plain ones a warp's fp32 chain grows with K and its error passes that of the FFMA2 kernels, whose
    // 32 to 128 threads have shorter chains (relative to the norm of the result, 6 seeds, plain /
    // compensated / FFMA2, 1e-8): Q4_0 M = 1 4096 x 11008 8.8 / 7.9 / 8.2, M = 4 4096 x 14336 9.3 / 7.9 / 8.3. It
    // costs 4 % there (4096 x 11008 9.9 -> 10.3 us). Up to three chunks at eight warps and four at
    // sixteen plain totals are no worse (K = 4096: within 0.3 %; 2048 x 16384: smaller).
    if (p.M <= 4 && p.K > (wide ? 4 * 16 : 3 * 8) * kTcBlocks * kQBlock)
        return wide ? launch_tc_one<FMT, 1, 16, true>(p, tiles, s) : launch_tc_one<FMT, 1, 8, true>(p, grid, s);
    if (p.M <= 8) return wide ? launch_tc_one<FMT, 1, 16>(p, tiles, s) : launch_tc_one<FMT, 1, 8>(p, grid, s);
    return wide ? launch_tc_one<FMT, 2, 16>(p, tiles, s) : launch_tc_one<FMT, 2, 8>(p, grid, s);
}

TcParams tc_params(const GroupRef& g, bool pdl, int& n_tiles) {
    TcParams p = {};
    int64_t tiles = 0;
    for (int i = 0; i < g.n_mats; ++i) {
        p.codes[i] = g.mats[i].codes;
        p.high[i] = g.mats[i].high;
        p.scales[i] = g.mats[i].scales;
        p.Y[i] = g.mats[i].Y;
        p.N[i] = int32_t(g.mats[i].N);
        p.tile0[i] = int32_t(tiles);
        tiles += (g.mats[i].N + kTcRows - 1) / kTcRows;
    }
    p.tile0[g.n_mats] = int32_t(tiles);
    p.n_mats = g.n_mats;
    p.M = int32_t(g.M);
    p.K = int32_t(g.K);
    p.ldS = int32_t(g.ldS);
    p.epi = g.epi;
    p.X = g.X;
    p.wait_first = pdl ? 0 : 1;
    n_tiles = int(tiles);
    return p;
}

// Which calls take it (us per launch in graph-replayed chains, this kernel / the one it leaves):
//  * M = 2..4, but for few row tiles, where one row per CTA of the register kernel is sooner done than a
//    CTA's walk along 16 rows: up to kFewTiles, which grow with K (64 x 16384 Q6_0 at M = 4 7.3 / 4.4) and
//    shrink with M and with what a row costs the register kernel (768 x 8192 Q8_0 at M = 2 4.1 / 3.7, at
//    M = 3 4.1 / 6.4; 768 x 2048 Q4_0 at M = 2 1.9 / 3.1). Measured at 13 K x 21 row counts for every format
//    and M: against the better of the two at each, this line loses 0.3 % or less (geometric mean). For gated
//    layers, whose register kernel has two rows per CTA, at 11 K x 14 row counts (512 x 8192 Q6_0 at M = 2 4.4 / 2.7). Q8_0 at M = 2 also leaves rows beyond 8192 k whose last round is mostly
//    empty (5000 x 16384 30.0 / 26.7);
//  * M = 6..16 in place of the tcgen05 GEMM (12288 x 4096 at M = 8 Q8_0 14.6 / 26.7, Q4_0 13.5 /
//    27.9; 1024 x 4096 at M = 16 4.6 / 6.4), but for Q8_0 above 12 tokens and 32 M weights
//    (32768 x 2048 30.4 / 27.7), for rows so short that most warps idle, beyond one round of tiles (32768 x
//    128 at M = 16 Q8_0 13.1 / 5.6, 32768 x 256 at M = 8 9.1 / 7.3, 32768 x 512 at M = 16 15.5 / 11.2), and for
//    five tokens, the count at which the GEMM's bf16 operand is held to its bits
//    (tests/test_gpu_hotpath_dequant.py);
//  * M = 1, Q4_0 and Q6_0, with rows of at least 4096 k, where its codes-to-bf16 step is cheaper than FFMA2
//    dot products and no activation row is staged per CTA, if its 16-row tiles are many and fill the SMs:
//    at least 60 (768 x 6144 Q6_0 3.7 / 2.8, 960 x 5120 Q4_0 2.9 / 3.8), and where they are more than the SMs at
//    least 80 % of the slots of their rounds of two CTAs per SM (4096 x 11008 Q4_0, 84 %, 10.3 / 11.3;
//    2560 x 11008, 53 %, 9.4 / 8.1; 6144 x 11008, 63 %, 18.1 / 15.4; 11008 x 11008, 75 %, 25.6 / 24.6).
//    At K where the staged kernel's tiles fit shared memory badly (Q4_0 beyond 4096 to 8192, Q6_0 4864 to 6144) any
//    fill beyond one round will do (Q4_0 11008 x 4608 12.9 / 15.5, 6144 x 5120 8.3 / 10.7, 24000 x 4864 21.1 / 32.8; Q6_0
//    6144 x 5120 10.4 / 11.2).
//    With K < 5120 not from 1216 to 4095 rows, where the register kernel has one short wave of four rows per
//    CTA (2048 x 4096 Q4_0 2.8 / 2.4, Q6_0 3.3 / 2.75), at any K not where that wave is exactly full (1216
//    rows x 8192 Q4_0 3.6 / 2.7; 1232 3.7 / 4.0), nor Q4_0 at 4096 beyond five tiles per SM (staged kernel: 22016 x
//    4096 16.9 / 16.4). Q6_0 only where rows fill the other kernels' passes of 256 threads to less than
//    70 % (4096 x 4096 4.95 / 7.1, 4096 x 11008 13.3 / 14.4; 4096 x 8192 9.6 / 9.2, 8192 x 16384 35.0 / 30.2, 1300 x 12288
//    6.6 / 6.3). Q8_0 gains at some row counts and loses at others (1024 x 4096 2.6 / 3.2, 1300 x 4096 2.9 / 2.2).
constexpr int kFewTilesK[4] = {639, 1151, 2048, 4096};  // K up to these (2048 and 4096: one chunk per warp), then the rest
constexpr int kFewTiles[2][3][3][5] = {                 // by gated or not, format, M - 2 and K
    {{{384, 44, 96, 56, 57}, {0, 0, 16, 24, 40}, {0, 0, 0, 16, 16}},   // Q8_0
     {{0, 0, 10, 11, 32}, {0, 0, 0, 8, 8}, {0, 0, 0, 0, 5}},           // Q4_0
     {{152, 28, 20, 10, 28}, {32, 16, 10, 8, 28}, {0, 0, 4, 8, 9}}},   // Q6_0
    {{{152, 48, 64, 57, 57}, {0, 8, 28, 32, 32}, {0, 0, 0, 32, 28}},
     {{0, 0, 16, 20, 32}, {0, 0, 0, 10, 32}, {0, 0, 0, 4, 16}},
     {{152, 60, 64, 48, 32}, {40, 20, 16, 16, 32}, {0, 0, 0, 8, 32}}}};
static_assert(EMB_Q8_0 == 0 && EMB_Q4_0 == 1 && EMB_Q6_0 == 2, "kFewTiles is indexed by format");
bool tc_takes(const GroupRef& g, int sms) {
    if (g.M > kTcMaxM || g.M == 5 || (g.fmt == EMB_Q6_0 && g.K % 64 != 0)) return false;
    int64_t rows = 0, tiles = 0;
    for (int i = 0; i < g.n_mats; ++i) {
        rows += g.mats[i].N;
        tiles += (g.mats[i].N + kTcRows - 1) / kTcRows;
    }
    const int64_t slots = 2 * int64_t(sms);
    const int64_t round_slots = slots * ((tiles + slots - 1) / slots);  // of the rounds that the tiles take
    if (g.M == 1) {
        if (g.fmt == EMB_Q8_0 || g.K < 4096 || tiles < 60) return false;
        const bool four_rows = rows >= 4 * 2 * 152;  // per CTA of the register kernel (launch_gemv_regs)
        if (four_rows && rows <= 4 * slots) return false;
        const bool any_fill = tiles > slots && (g.fmt == EMB_Q4_0 ? g.K > 4096 && g.K <= 8192 : g.K >= 4864 && g.K <= 6144);
        if (tiles > sms && !any_fill && 5 * tiles < 4 * round_slots) return false;
        if (g.K < 5120 && four_rows && rows < 4096) return false;
        if (g.fmt == EMB_Q4_0) return g.K > 4096 || tiles <= 5 * int64_t(sms);
        const int64_t U = g.K / 32, passes = (U + 255) / 256;
        return U < 256 || 10 * U < 7 * 256 * passes;
    }
    if (g.M <= 4) {
        int k_class = 0;
        while (k_class < 4 && g.K > kFewTilesK[k_class]) ++k_class;
        if (rows <= kTcRows * kFewTiles[g.epi >= EMB_EPI_GEGLU][g.fmt][g.M - 2][k_class]) return false;
        return !(g.M == 2 && g.fmt == EMB_Q8_0 && g.K > 8192 && tiles > slots && 20 * tiles < 13 * round_slots);
    }
    const int64_t short_k = g.M > 8 ? 256 : 128;
    if ((tiles > slots && g.K <= short_k) || (tiles > 2 * slots && g.K <= 2 * short_k)) return false;
    if (g.fmt == EMB_Q8_0 && g.M > 12) return rows * g.K <= (int64_t(1) << 25);
    return true;
}

bool launch_tc(const GroupRef& g, bool pdl, cudaStream_t s, cudaError_t& err) {
    const int sms = device_sm_count();
    if (sms <= 0 || !tc_takes(g, sms)) return false;
    int tiles = 0;
    const TcParams p = tc_params(g, pdl, tiles);
    err = g.fmt == EMB_Q8_0   ? launch_tc_fmt<EMB_Q8_0>(p, tiles, sms, s)
          : g.fmt == EMB_Q4_0 ? launch_tc_fmt<EMB_Q4_0>(p, tiles, sms, s)
                              : launch_tc_fmt<EMB_Q6_0>(p, tiles, sms, s);
    return true;
}

// ------------------------------------------------------------------ tensor-core chunk GEMM
// An action chunk (M = 17..64, K >= 1024). The tcgen05 GEMM gives such a layer few CTAs of 128 rows,
// splits its K over a cluster and pays fill, TMEM hand-offs and a distributed-shared-memory exchange
// after the activations have arrived (M = 50: 5.2 to 8.8 us per launch). This kernel streams 16-row
// tiles as the tensor-core GEMV does, so a 1024-row layer has 64 tiles x 2 token groups of work for the
// SMs and no exchange between CTAs. Its operand is the GEMM's: bf16(w'), one rounding of the exact
// fp32 product of code and scale, every product exact, fp32 accumulation, so a layer's bits do
// not depend on which of the two runs it beyond the order of the fp32 sums.
//
// A warp owns 32 tokens (four MMA n-tiles) and every WK-th 256-k chunk of a row tile; WK x WT = 8 warps
// cover WT token groups (short rows: four warps along K and both token groups in one CTA; longer ones:
// eight along K, token groups along grid y). Activation fragments come straight from global memory
// (cached loads after griddepcontrol.wait), each read by one warp of the CTA. The K slices of a tile are
// added pairwise through shared memory.
// What bounds it: the activations' way into each SM (M x K x 2 bytes per CTA and round, ~58 bytes per
// cycle) and the latency of one load-convert-multiply chain. Q8_0 at M = 50, 1024 x 1024: 3.6 us per
// launch against 5.2, action expert step 745 -> 723.
constexpr int kCkTokens = 32;   // tokens per warp
constexpr int kCkStages = 2;    // ring depth
constexpr int kCkPitch = kTcRows + 4;  // floats per token of the sums: conflict-free stores
template <int FMT>
constexpr int kCkSmem = 8 * kCkStages * TcStage<FMT>::kBytes;

template <int FMT, int WK>
__global__ void __launch_bounds__(256, 2) gemm_chunk_kernel(const __grid_constant__ TcParams p) {
    using St = TcStage<FMT>;
    constexpr int WT = 8 / WK, NT = kCkTokens / 8;
    constexpr float kBias = FMT == EMB_Q8_0 ? 32768.0f + 128.0f : FMT == EMB_Q4_0 ? 32768.0f + 8.0f : 32768.0f + 32.0f;
    extern __shared__ __align__(128) uint8_t smem[];
    __shared__ float red[8][kCkTokens][kCkPitch];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int g = lane >> 2, t = lane & 3;
    const int wk = warp % WK, wt = warp / WK;
    const int nb = p.K / kQBlock;
    const int tiles = p.tile0[p.n_mats];
    const uint32_t ring = ptx::smem_u32(smem) + warp * kCkStages * St::kBytes;
    const int m_base = kCkTokens * (int(blockIdx.y) * WT + wt);  // the warp's first token

    if (p.wait_first) griddep_wait();  // before the trigger: see ptx::griddep_launch_dependents
    griddep_launch_dependents();
    const int stride = WK * kTcBlocks;
    int it_tile = blockIdx.x, it_base = 0;
    auto issue_next = [&](int stage) {
        if (it_tile < tiles) {
            tc_issue<FMT>(p, it_tile, it_base + wk * kTcBlocks, ring + stage * St::kBytes, lane);
            it_base += stride;
            if (it_base >= nb) {
                it_base = 0;
                it_tile += gridDim.x;
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
#pragma unroll
    for (int i = 0; i < kCkStages; ++i) issue_next(i);
    if (threadIdx.x == 0 && blockIdx.x == 0 && blockIdx.y == 0)
        ptx::prefetch_l2(p.X, uint32_t(p.M) * uint32_t(p.K) * 2u);
    // weights do not depend on earlier launches; X and Y may
    griddep_wait();

    // activations of token m_base + 8 nt + g (rows past M read the last token; never stored)
    const __nv_bfloat16* xr[NT];
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) xr[nt] = p.X + int64_t(min(m_base + 8 * nt + g, p.M - 1)) * p.K;
    auto load_x = [&](int kb, int nt, uint32_t (&b)[4]) {
        const uint4 v = *reinterpret_cast<const uint4*>(xr[nt] + kb * 32 + 8 * t);
        b[0] = v.x; b[1] = v.y; b[2] = v.z; b[3] = v.w;
    };
    // four codes (bytes) of a row -> bf16(w') pairs (0, 1) and (2, 3)
    auto weights = [&](uint32_t bytes, float d, float nbd, uint32_t& p01, uint32_t& p23) {
        float2 a, b;
        dq::bytes_to_w(bytes, d, nbd, a, b);
        p01 = dq::pack_bf16(a.x, a.y);
        p23 = dq::pack_bf16(b.x, b.y);
    };

    float acc[NT][4];
    const int ra = tc_row<FMT>(g);
    int stage = 0;
    for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) acc[nt][0] = acc[nt][1] = acc[nt][2] = acc[nt][3] = 0.0f;
        const int gm = tc_mat_of(p, tile), N = p.N[gm], n0 = (tile - p.tile0[gm]) * kTcRows;
        // residual add: the old values are on their way while the products are summed
        constexpr int kOut = WT * kCkTokens * kTcRows / 256;  // outputs per thread
        float old[kOut];
        if (p.epi == EMB_EPI_ADD) {
#pragma unroll
            for (int it = 0; it < kOut; ++it) {
                const int m = kCkTokens * int(blockIdx.y) * WT + it * 16 + threadIdx.x / 16, n = n0 + threadIdx.x % 16;
                old[it] = m < p.M && n < N ? reinterpret_cast<const float*>(p.Y[gm])[int64_t(m) * N + n] : 0.0f;
            }
        }
        for (int base = 0; base < nb; base += stride) {
            asm volatile("cp.async.wait_group %0;" ::"n"(kCkStages - 1) : "memory");
            __syncwarp();  // every lane's copies of this chunk have landed
            const int kb0 = base + wk * kTcBlocks;
            const uint32_t st = ring + stage * St::kBytes;
            const uint32_t sc = st + St::kCodes + St::kHigh + ra * 16;
#pragma unroll
            for (int i = 0; i < kTcBlocks; ++i) {
                if (kb0 + i >= nb) break;
                uint32_t b[NT][4];
#pragma unroll
                for (int nt = 0; nt < NT; ++nt) load_x(kb0 + i, nt, b[nt]);
                const float da = ld_shared_half(sc + 2 * i), db = ld_shared_half(sc + 8 * 16 + 2 * i);
                const float na = -kBias * da, nb_ = -kBias * db;  // exact (see bytes_to_w)
                uint32_t a0[4], a1[4];
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    uint2 v = tc_codes<FMT>(st, ra + 8 * r, i, t);
                    if constexpr (FMT == EMB_Q8_0) v = make_uint2(v.x ^ 0x80808080u, v.y ^ 0x80808080u);
                    weights(v.x, r ? db : da, r ? nb_ : na, a0[r], a0[2 + r]);
                    weights(v.y, r ? db : da, r ? nb_ : na, a1[r], a1[2 + r]);
                }
#pragma unroll
                for (int nt = 0; nt < NT; ++nt) mma_bf16_16816(acc[nt], a0, b[nt][0], b[nt][1]);
#pragma unroll
                for (int nt = 0; nt < NT; ++nt) mma_bf16_16816(acc[nt], a1, b[nt][2], b[nt][3]);
            }
            __syncwarp();  // every lane has read the chunk
            issue_next(stage);
            stage = stage + 1 == kCkStages ? 0 : stage + 1;
        }
        // acc[nt][0, 1]: row ra, tokens 8 nt + 2t, + 1; [2, 3]: row ra + 8
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
            red[warp][8 * nt + 2 * t][ra] = acc[nt][0];
            red[warp][8 * nt + 2 * t + 1][ra] = acc[nt][1];
            red[warp][8 * nt + 2 * t][ra + 8] = acc[nt][2];
            red[warp][8 * nt + 2 * t + 1][ra + 8] = acc[nt][3];
        }
        __syncthreads();
        // sums of the K slices of (token of the CTA, row), pairwise
        auto total = [&](int tok, int row) {
            float v[WK];
#pragma unroll
            for (int w = 0; w < WK; ++w) v[w] = red[tok / kCkTokens * WK + w][tok % kCkTokens][row];
#pragma unroll
            for (int o = WK / 2; o > 0; o >>= 1)
#pragma unroll
                for (int w = 0; w < o; ++w) v[w] += v[w + o];
            return v[0];
        };
        const int m0 = kCkTokens * int(blockIdx.y) * WT;
        if (p.epi >= EMB_EPI_GEGLU) {
#pragma unroll
            for (int it = 0; it < kOut / 2; ++it) {  // one gate/up pair per thread
                const int tok = it * 32 + threadIdx.x / 8, r = 2 * (threadIdx.x % 8);
                if (m0 + tok < p.M && n0 + r < N)
                    epi_store_gated(p.epi, p.Y[gm], m0 + tok, n0 + r, N, total(tok, r), total(tok, r + 1));
            }
        } else {
#pragma unroll
            for (int it = 0; it < kOut; ++it) {
                const int tok = it * 16 + threadIdx.x / 16, r = threadIdx.x % 16;
                if (m0 + tok >= p.M || n0 + r >= N) continue;
                const float v = total(tok, r);
                if (p.epi == EMB_EPI_ADD)
                    reinterpret_cast<float*>(p.Y[gm])[int64_t(m0 + tok) * N + n0 + r] = __fadd_rn(old[it], v);
                else
                    epi_store(p.epi, p.Y[gm], m0 + tok, n0 + r, N, v);
            }
        }
        if (tile + int(gridDim.x) < tiles) __syncthreads();  // the sums are read before the next tile's
    }
}

template <int FMT, int WK>
cudaError_t launch_chunk_one(const TcParams& p, dim3 grid, cudaStream_t s) {
    static std::atomic<uint64_t> done{0};
    const cudaError_t e = allow_smem(gemm_chunk_kernel<FMT, WK>, kCkSmem<FMT>, done);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(256, 1, 1);
    cfg.dynamicSmemBytes = kCkSmem<FMT>;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, gemm_chunk_kernel<FMT, WK>, p);
}

template <int FMT>
cudaError_t launch_chunk_fmt(const TcParams& p, int tiles, int sms, cudaStream_t s) {
    const int groups = (p.M + kCkTokens - 1) / kCkTokens;  // 1 or 2
    if (p.K < 8 * kTcBlocks * kQBlock && groups == 2)
        return launch_chunk_one<FMT, 4>(p, dim3(std::min(tiles, 2 * sms), 1, 1), s);
    return launch_chunk_one<FMT, 8>(p, dim3(std::min(tiles, 2 * sms / groups), groups, 1), s);
}

// Which calls take it: those that a model of both kernels, in us, says are sooner done here. A CTA walks
// whole rows, so full rounds (more CTAs than SMs) and a last one of one CTA per SM cost by the chunks of a
// warp, and by the k of its activations. Fitted to 3060 launches (M = 17..64, K = 1024..16384, 64 to
// 32768 rows, three formats; rms 8 %, the GEMM's 7 %); its choices lose 0.4 % against the better kernel at each
// (geometric mean) and one of them is more than 1 % slower than the GEMM was without this kernel. Measured,
// this kernel / the GEMM: M = 50 1024 x 1024 3.7 / 5.3, 2048 x 2048 4.6 / 12.6, 8192 x 1024 8.2 / 8.2, 6144 x 1536 12.9 /
// 9.0; M = 32 4096 x 4096 8.7 / 10.9, 1792 x 16384 27.5 / 18.0, 16384 x 2560 Q6_0 27.2 / 20.0.
bool chunk_takes(const GroupRef& g, int sms) {
    if (g.M <= kTcMaxM || g.M > 2 * kCkTokens || g.K < 1024 || g.precise || (g.fmt == EMB_Q6_0 && g.K % 64 != 0))
        return false;
    int64_t tiles = 0, rows = 0;
    for (int i = 0; i < g.n_mats; ++i) {
        rows += g.mats[i].N;
        tiles += (g.mats[i].N + kTcRows - 1) / kTcRows;
    }
    const bool both = g.M > kCkTokens && g.K < 8 * kTcBlocks * kQBlock;  // token groups in one CTA
    const int64_t ctas = g.M > kCkTokens && !both ? 2 * tiles : tiles, slots = 2 * int64_t(sms), rest = ctas % slots;
    const double span = (both ? 4.0 : 8.0) * kTcBlocks * kQBlock;  // k that the warps of a row tile take at once
    const double full = double(ctas / slots + (rest > sms)), half = rest > 0 && rest <= sms ? 1.0 : 0.0;
    const double steps = std::ceil(double(g.K) / span);
    // one CTA per SM and one chunk per warp: 16 % or more below the GEMM at every such size measured, so the
    // smallest calls need not ask for its plan, whose time on the host they feel (17 x 1000 x 1184 with it
    // 5.2 us a call, without 4.8)
    if (full == 0.0 && steps == 1.0) return true;
    // (the products of up to 32 tokens do not hide the wider codes' way in)
    const double codes = g.M > kCkTokens || g.fmt == EMB_Q4_0 ? 0.0 : g.fmt == EMB_Q8_0 ? 0.8e-7 : 0.4e-7;
    const double us = 0.44 + full * (0.39 + 2.25 * steps) + half * (0.70 + 1.49 * steps) +
                      (full + half) * 1.09 * double(g.K) / span + codes * double(rows) * double(g.K);
    return us < gemm_tc_chunk_us(g);
}

// ------------------------------------------------------------------ ring GEMV
// Long rows at M = 1 (more than one pass of 256 threads; Gemma-2B's down projection,
// 2048 x 16384). The register kernel holds only as many bytes in flight as the resident
// CTAs' registers, so such a matrix streams in two waves of CTAs whose loads do not overlap,
// and the staged kernel re-stages the whole activation row for every tile of one or two
// rows. Here a CTA owns a run of consecutive rows (crossing
// matrix boundaries within the group) and keeps the activation row it needs in registers:
// each thread's units t + k*256 of X, loaded once after griddepcontrol.wait and reused for
// every row. The rows stream through a ring of shared-memory stages (one row of codes and
// its scales each; as many as kRingBudget holds, 2..8), filled by bulk copies that one
// thread issues -- a ring's worth before the wait -- and refills as soon as all eight warps
// have released a stage. The warps run on the ring's barriers alone (no CTA-wide barrier
// until the reduction). Each row is summed as in the register kernel (per thread over its
// units in order, shuffle tree, warps in order), so its bits equal that kernel's.
constexpr int kRingThreads = 256;
constexpr int kRingMaxStages = 8;
constexpr int kRingBudget = 56 * 1024;  // ring bytes per CTA: stages = budget / stage, 2..8
constexpr int kRingFlush = 16;  // rows whose per-warp sums are kept before a CTA-wide reduction
// barriers (0..127), abort flag (128), per-warp sums (144..655), then the ring
constexpr int kRingHeader = 144 + kRingFlush * (kRingThreads / 32) * 4;

struct RingParams {
    const uint8_t* codes[kMaxGroup];
    const uint8_t* high[kMaxGroup];  // Q6_0: 2-bit high plane of each matrix
    const __half* scales[kMaxGroup];
    void* Y[kMaxGroup];
    int32_t N[kMaxGroup];
    int32_t row0[kMaxGroup + 1];  // first row of each matrix in the group's row order
    int32_t n_mats;
    int32_t K, ldS, U;
    int32_t rows_per_cta, rows_total;
    int32_t stage_bytes;          // one row of codes (+ Q6_0 high bits) + its scales, rounded up to 16
    int32_t stages;               // ring depth (2..kRingMaxStages)
    int32_t epi;
    int32_t wait_first;            // 1: nothing is read before griddepcontrol.wait
    const __nv_bfloat16* X;
    int* status;
};

template <int FMT, int PF, bool FIRST>
__global__ void __launch_bounds__(kRingThreads, 2) gemv_ring_kernel(const __grid_constant__ RingParams p) {
    constexpr int UW = (FMT == EMB_Q8_0) ? 16 : 32;
    constexpr int NT = kRingThreads, NWARP = NT / 32;
    extern __shared__ __align__(128) uint8_t smem[];
    uint64_t* full = reinterpret_cast<uint64_t*>(smem);              // [stages]
    uint64_t* empty = full + kRingMaxStages;                          // [stages]
    volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + 128);  // a wait gave up
    float* red = reinterpret_cast<float*>(smem + 144);               // [kRingFlush][NWARP]
    uint8_t* ring = smem + kRingHeader;                               // [stages][stage_bytes]
    const int S = p.stages;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int U = p.U;
    const int64_t row_bytes = (FMT == EMB_Q8_0) ? int64_t(p.K) : int64_t(p.K) / 2;
    const int64_t high_bytes = (FMT == EMB_Q6_0) ? int64_t(p.K) / 4 : 0;  // a multiple of 16
    const int r_begin = blockIdx.x * p.rows_per_cta;
    const int n_rows = min(p.rows_per_cta, p.rows_total - r_begin);
    // global row -> (matrix, row within it)
    auto locate = [&](int gr, int& g, int& n) {
        g = 0;
#pragma unroll
        for (int i = 1; i < kMaxGroup; ++i)
            if (i < p.n_mats && gr >= p.row0[i]) g = i;
        n = gr - p.row0[g];
    };
    auto issue = [&](int i, int stage) {  // row i of this CTA into a stage
        int g, n;
        locate(r_begin + i, g, n);
        uint8_t* st = ring + stage * p.stage_bytes;
        uint64_t* bar = &full[stage];
        const uint32_t cb = uint32_t(row_bytes), hb = uint32_t(high_bytes), sb = uint32_t(p.ldS) * 2u;
        ptx::mbar_arrive_expect_tx(bar, cb + hb + sb);
        ptx::bulk_load(st, p.codes[g] + int64_t(n) * row_bytes, cb, bar);
        if constexpr (FMT == EMB_Q6_0) ptx::bulk_load(st + row_bytes, p.high[g] + int64_t(n) * high_bytes, hb, bar);
        ptx::bulk_load(st + row_bytes + high_bytes, p.scales[g] + int64_t(n) * p.ldS, sb, bar);
    };
    if (t == 0) {
        *abort_flag = 0;
        for (int i = 0; i < S; ++i) {
            ptx::mbar_init(&full[i], 1);
            ptx::mbar_init(&empty[i], NWARP);
        }
        ptx::fence_mbar_init();
        if constexpr (FIRST) ptx::griddep_wait();
        for (int i = 0; i < S && i < n_rows; ++i) issue(i, i);
        // the activation row towards L2 while the previous launch finishes (one CTA asks)
        if (blockIdx.x == 0) ptx::prefetch_l2(p.X, uint32_t(p.K) * 2u);
    }
    if constexpr (FIRST) griddep_wait();  // every thread before the trigger: see ptx::griddep_launch_dependents
    griddep_launch_dependents();
    __syncthreads();  // the barriers' initialisation is visible to every waiting thread
    // weights do not depend on earlier launches; X and Y may
    griddep_wait();
    float x[PF][UW];
#pragma unroll
    for (int k = 0; k < PF; ++k) {
        const int uk = t + k * NT;
        const uint4* xp = reinterpret_cast<const uint4*>(p.X + int64_t(min(uk, U - 1)) * UW);
#pragma unroll
        for (int v = 0; v < UW / 8; ++v) {
            const uint4 hx = xp[v];
            x[k][8 * v + 0] = lo_bf16(hx.x); x[k][8 * v + 1] = hi_bf16(hx.x);
            x[k][8 * v + 2] = lo_bf16(hx.y); x[k][8 * v + 3] = hi_bf16(hx.y);
            x[k][8 * v + 4] = lo_bf16(hx.z); x[k][8 * v + 5] = hi_bf16(hx.z);
            x[k][8 * v + 6] = lo_bf16(hx.w); x[k][8 * v + 7] = hi_bf16(hx.w);
        }
    }
    bool ok = true;
    int flushed = 0;  // rows already reduced and stored
    // reduce and store rows [flushed, upto) of this CTA; false (the CTA leaves) if any of its
    // waits gave up. The only CTA-wide barriers: between them the warps run on the ring's
    // barriers alone, each wait bounded and abandoned as soon as another thread gave up.
    auto flush = [&](int upto) -> bool {
        if (__syncthreads_or(!ok)) return false;
        const int cnt = upto - flushed;
        if (p.epi >= EMB_EPI_GEGLU) {
            // gate row 2i and up row 2i + 1 of the CTA (runs start on even rows)
            if (t < cnt / 2) {
                float gate = 0.0f, up = 0.0f;
#pragma unroll
                for (int w = 0; w < NWARP; ++w) {
                    gate += red[(2 * t) * NWARP + w];
                    up += red[(2 * t + 1) * NWARP + w];
                }
                int g, n;
                locate(r_begin + flushed + 2 * t, g, n);
                epi_store_gated(p.epi, p.Y[g], 0, n, p.N[g], gate, up);
            }
        } else if (t < cnt) {
            float v = 0.0f;
#pragma unroll
            for (int w = 0; w < NWARP; ++w) v += red[t * NWARP + w];
            int g, n;
            locate(r_begin + flushed + t, g, n);
            epi_store(p.epi, p.Y[g], 0, n, p.N[g], v);
        }
        __syncthreads();
        flushed = upto;
        return true;
    };
    // stage and phase of row i, and of row i - 1, kept by increments (no integer division)
    int s = 0, sp = 0;
    uint32_t ph = 0, php = 0;
    for (int i = 0; i < n_rows; ++i) {
        // refill: the stage of row i - 1 once every warp has released it
        if (t == 0 && ok && i >= 1 && i - 1 + S < n_rows) {
            ok = ptx::mbar_wait(&empty[sp], php, abort_flag, p.status, kWaitLimitNs);
            if (ok) issue(i - 1 + S, sp);
        }
        ok = __all_sync(0xffffffffu, ok && ptx::mbar_wait(&full[s], ph, abort_flag, p.status, kWaitLimitNs));
        if (ok) {
            const uint8_t* cs = ring + s * p.stage_bytes;
            const __half* ss = reinterpret_cast<const __half*>(cs + row_bytes + high_bytes);
            float acc = 0.0f;
#pragma unroll
            for (int k = 0; k < PF; ++k) {
                const int uk = t + k * NT;
                if (uk < U) {
                    const uint4 c = *reinterpret_cast<const uint4*>(cs + int64_t(uk) * 16);
                    uint2 hq = make_uint2(0, 0);
                    if constexpr (FMT == EMB_Q6_0) hq = *reinterpret_cast<const uint2*>(cs + row_bytes + int64_t(uk) * 8);
                    const float d = __half2float(ss[(FMT == EMB_Q8_0) ? (uk >> 1) : uk]);
                    acc = fmaf(d, dot_unit<FMT>(c, hq, x[k]), acc);
                }
            }
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(&empty[s]);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
            if (lane == 0) red[(i - flushed) * NWARP + warp] = acc;
        }
        if (i + 1 - flushed == kRingFlush && !flush(i + 1)) return;
        sp = s;
        php = ph;
        if (++s == S) {
            s = 0;
            ph ^= 1u;
        }
    }
    if (flushed < n_rows) flush(n_rows);  // (a CTA whose wait gave up leaves inside it)
}

template <int FMT, int PF, bool FIRST>
cudaError_t launch_ring_one(const RingParams& p, int ctas, size_t smem, cudaStream_t s) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(ctas, 1, 1);
    cfg.blockDim = dim3(kRingThreads, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    // (two stages of the longest row, 16 KB of codes, fit the budget too)
    static std::atomic<uint64_t> done{0};
    const cudaError_t e = allow_smem(gemv_ring_kernel<FMT, PF, FIRST>, kRingHeader + kRingBudget, done);
    if (e != cudaSuccess) return e;
    return cudaLaunchKernelEx(&cfg, gemv_ring_kernel<FMT, PF, FIRST>, p);
}

template <int FMT>
cudaError_t launch_ring_fmt(const RingParams& p, int pf, int ctas, size_t smem, cudaStream_t s) {
    if (p.wait_first)
        return pf == 2 ? launch_ring_one<FMT, 2, true>(p, ctas, smem, s)
             : pf == 3 ? launch_ring_one<FMT, 3, true>(p, ctas, smem, s)
                       : launch_ring_one<FMT, 4, true>(p, ctas, smem, s);
    return pf == 2 ? launch_ring_one<FMT, 2, false>(p, ctas, smem, s)
         : pf == 3 ? launch_ring_one<FMT, 3, false>(p, ctas, smem, s)
                   : launch_ring_one<FMT, 4, false>(p, ctas, smem, s);
}

// Which layers take the ring path: M = 1, Q8_0 or Q6_0 (K % 64 == 0, for its high plane's 16-byte rows;
// what of it tc_takes leaves), rows longer than the staged path takes at M = 1 and than one pass
// of 256 threads (2..4 units per thread), matrices of at least kStageMinBytes; two CTAs per
// SM, rows split evenly (even runs for gated epilogues).
// Measured on GB300, Gemma-2B decode step (paired runs on one box, 1000 steps): Q8_0 chain
// 0.507 -> 0.477 ms against a kernel with two rows per CTA in
// registers and two in shared memory; a 72 KB ring instead of 56 KB was slower for Q8_0,
// a CTA-wide barrier per row cost ~2 %, and stage indices by integer division ~4 %.
bool ring_takes(const GroupRef& g) {
    if (g.M != 1 || g.fmt == EMB_Q4_0 || (g.fmt == EMB_Q6_0 && g.K % 64 != 0)) return false;
    const int64_t weight_row_bytes = g.fmt == EMB_Q8_0 ? g.K : g.K / 2 + g.K / 4;
    const int64_t U = g.fmt == EMB_Q8_0 ? g.K / 16 : g.K / 32;
    if (weight_row_bytes <= kStageMaxRowBytesM1 || U <= kRingThreads || U > 4 * kRingThreads) return false;
    int64_t rows = 0;
    for (int i = 0; i < g.n_mats; ++i) rows += g.mats[i].N;
    return rows * weight_row_bytes >= kStageMinBytes;
}

bool launch_ring(const GroupRef& g, bool pdl, int* status, cudaStream_t s, cudaError_t& err) {
    if (!ring_takes(g)) return false;
    const int64_t row_bytes = (g.fmt == EMB_Q8_0) ? g.K : g.K / 2;
    const int64_t high_bytes = (g.fmt == EMB_Q6_0) ? g.K / 4 : 0;
    const int64_t U = (g.fmt == EMB_Q8_0) ? g.K / 16 : g.K / 32;
    int64_t rows = 0;
    for (int i = 0; i < g.n_mats; ++i) rows += g.mats[i].N;
    const int sms = device_sm_count();
    if (sms <= 0) return false;
    RingParams p = {};
    int64_t r0 = 0;
    for (int i = 0; i < g.n_mats; ++i) {
        p.codes[i] = g.mats[i].codes;
        p.high[i] = g.mats[i].high;
        p.scales[i] = g.mats[i].scales;
        p.Y[i] = g.mats[i].Y;
        p.N[i] = int32_t(g.mats[i].N);
        p.row0[i] = int32_t(r0);
        r0 += g.mats[i].N;
    }
    p.row0[g.n_mats] = int32_t(r0);
    p.n_mats = g.n_mats;
    p.K = int32_t(g.K);
    p.ldS = int32_t(g.ldS);
    p.U = int32_t(U);
    p.epi = g.epi;
    p.X = g.X;
    p.wait_first = pdl ? 0 : 1;
    p.status = status;
    int64_t rpc = (rows + 2 * sms - 1) / (2 * sms);
    if (g.epi >= EMB_EPI_GEGLU) rpc = (rpc + 1) & ~int64_t(1);  // gate/up pairs stay in one CTA
    p.rows_per_cta = int32_t(rpc);
    p.rows_total = int32_t(rows);
    p.stage_bytes = int32_t((row_bytes + high_bytes + g.ldS * 2 + 15) & ~int64_t(15));
    p.stages = int32_t(std::min<int64_t>(kRingMaxStages, std::max<int64_t>(2, kRingBudget / p.stage_bytes)));
    const int ctas = int((rows + rpc - 1) / rpc);
    const size_t smem = kRingHeader + size_t(p.stages) * p.stage_bytes;
    const int pf = int((U + kRingThreads - 1) / kRingThreads);
    err = g.fmt == EMB_Q8_0 ? launch_ring_fmt<EMB_Q8_0>(p, pf, ctas, smem, s)
                            : launch_ring_fmt<EMB_Q6_0>(p, pf, ctas, smem, s);
    return true;
}

bool launch_chunk(const GroupRef& g, bool pdl, cudaStream_t s, cudaError_t& err) {
    const int sms = device_sm_count();
    if (sms <= 0 || !chunk_takes(g, sms)) return false;
    int tiles = 0;
    const TcParams p = tc_params(g, pdl, tiles);
    err = g.fmt == EMB_Q8_0   ? launch_chunk_fmt<EMB_Q8_0>(p, tiles, sms, s)
          : g.fmt == EMB_Q4_0 ? launch_chunk_fmt<EMB_Q4_0>(p, tiles, sms, s)
                              : launch_chunk_fmt<EMB_Q6_0>(p, tiles, sms, s);
    return true;
}

cudaError_t launch_gemv_regs(const GroupRef& g, bool pdl, cudaStream_t s);

}  // namespace

bool launch_mma_sync(const GroupRef& g, bool pdl, cudaStream_t s, cudaError_t& err) {
    return launch_chunk(g, pdl, s, err) || launch_tc(g, pdl, s, err);
}

cudaError_t launch_gemv(const GroupRef& g, bool pdl, int* status, cudaStream_t s) {
    cudaError_t err = cudaSuccess;
    if (launch_tc(g, pdl, s, err)) return err;
    if (launch_staged(g, pdl, status, s, err)) return err;
    if (launch_ring(g, pdl, status, s, err)) return err;
    return launch_gemv_regs(g, pdl, s);
}

namespace {

// Register-streaming GEMV: every shape the other kernels leave out.
cudaError_t launch_gemv_regs(const GroupRef& g, bool pdl, cudaStream_t s) {
    GemvParams p = {};
    const int U = int((g.fmt == EMB_Q8_0) ? g.K / 16 : g.K / 32);
    int64_t rows = 0;
    for (int i = 0; i < g.n_mats; ++i) rows += g.mats[i].N;
    // rows per CTA: 4 (activation reuse across rows) unless that leaves the GPU idle;
    // 2 for long rows (U >= 320), where 4 rows leave too few CTAs per SM (measured on
    // GB300, M=1: Q8_0 2048 x 16384 10.8 us with 4 rows, 9.6 us with 2)
    int R = (rows < 4 * 2 * 152) ? 1 : (U >= 320) ? 2 : 4;
    if (g.epi >= EMB_EPI_GEGLU && R == 1) R = 2;  // gate/up row pairs inside one CTA
    int tiles = 0;
    for (int i = 0; i < g.n_mats; ++i) {
        p.codes[i] = g.mats[i].codes;
        p.high[i] = g.mats[i].high;
        p.scales[i] = g.mats[i].scales;
        p.Y[i] = g.mats[i].Y;
        p.N[i] = int32_t(g.mats[i].N);
        p.tile0[i] = tiles;
        tiles += int((g.mats[i].N + R - 1) / R);
    }
    p.tile0[g.n_mats] = tiles;
    p.n_mats = g.n_mats;
    p.M = int32_t(g.M);
    p.K = int32_t(g.K);
    p.ldS = int32_t(g.ldS);
    p.U = U;
    p.epi = g.epi;
    p.X = g.X;
    p.wait_first = pdl ? 0 : 1;
    const int NT = pick_threads(U, g.fmt, tiles);
    const int M = int(g.M);
    if (g.fmt == EMB_Q8_0)
        return R == 4 ? dispatch_nt<EMB_Q8_0, 4>(p, tiles, M, NT, s)
             : R == 2 ? dispatch_nt<EMB_Q8_0, 2>(p, tiles, M, NT, s)
                      : dispatch_nt<EMB_Q8_0, 1>(p, tiles, M, NT, s);
    if (g.fmt == EMB_Q4_0)
        return R == 4 ? dispatch_nt<EMB_Q4_0, 4>(p, tiles, M, NT, s)
             : R == 2 ? dispatch_nt<EMB_Q4_0, 2>(p, tiles, M, NT, s)
                      : dispatch_nt<EMB_Q4_0, 1>(p, tiles, M, NT, s);
    return R == 4 ? dispatch_nt<EMB_Q6_0, 4>(p, tiles, M, NT, s)
         : R == 2 ? dispatch_nt<EMB_Q6_0, 2>(p, tiles, M, NT, s)
                  : dispatch_nt<EMB_Q6_0, 1>(p, tiles, M, NT, s);
}

}  // namespace

}  // namespace emb
