// Tensor-core GEMM for the larger token counts of one closed-loop step (M = 50 action
// chunk, M = 280..816 prefix prefill): packed Q8_0/Q4_0 weights are staged in shared
// memory by TMA, dequantised by eight warps into bf16 tiles held in tensor memory, and
// fed to tcgen05 MMAs (A operand from TMEM, B from shared memory) whose fp32
// accumulators also live in TMEM.
//
// "Swap AB": the MMA's M side is 128 weight rows (output features n), its N side is the
// CTA's T tokens, so one weight tile is dequantised once for up to 256 tokens and the
// accumulator D[n][m] sits in TMEM lanes = n. The epilogue reads TMEM lane n (one
// thread per output feature) and writes Y[m][n] with 128-byte coalesced stores.
//
// TMEM (512 columns, one CTA per SM): the accumulators of the CTA's one or two token tiles
// (T columns each, rounded up to 32), then a ring of up to eight bf16 A tiles (32 columns =
// 64 k per tile, two values per column, row n in lane n). Keeping A out of shared memory leaves
// its bandwidth to the X tiles (written by TMA, read by the MMA at 64 bytes per cycle).
//
// Roles (320 threads):
//   warp 0        : TMA producer. Raw stages (256 codes of 128 rows + their 8 scales) are
//                   fetched before griddepcontrol.wait (weights never depend on the previous
//                   launch); X tiles (64 k x T tokens) after it.
//   warp 1        : TMEM allocation; waits for each step's X and A tile and issues its MMAs
//                   (4 x K=16 per 64-k step and token tile).
//   warps 2..9    : dequantisation (two threads per weight row, tcgen05.st into the
//                   warp's lane quarter), then the epilogue.
// Both issuing warps run converged on warp-uniform operands and elect one lane per instruction
// (ptx::elect_one says why: behind `lane == 0` an MMA took 100 to 200 cycles to issue, more than
// its tensor time; with a separate waiter warp in front of it Gemma-2B gate/up at M = 816 took
// 123 us, now 104). What bounds a 64-k step now (T = 208, cycles): the loads of X and codes into
// the SM 613 (58 bytes per cycle with all SMs loading), the dequantising warps' chain of barrier,
// arithmetic and TMEM store ~600, the tensor pipe 416. Sixteen dequantising warps, a separate
// group of epilogue warps, or a third raw stage (one X stage fewer) are all slower: gate/up
// 115, 113 and 121 us against 109 then.
// Grid: x = token tile (fastest: CTAs sharing a weight tile run together), y = weight-row
// tile, z = K split. With z > 1 the splits of one output tile form a thread-block cluster
// and are summed in a fixed order through distributed shared memory (deterministic).
// Every wait is bounded (ptx::mbar_wait); on expiry the kernel records EMB_ETIMEOUT,
// lets every copy and MMA it issued land, frees TMEM and returns.
//
// Precision: each operand value is bf16(w') -- one rounding of the exact fp32 w' -- so
// the products are exact and accumulate in fp32. For K < 1024, and for layers flagged
// EMB_PRECISE_OPERAND, the SPLIT variant also stages lo = bf16(w' - bf16(w')) and issues
// a second MMA per step, which brings the operand error from 2^-8 to 2^-16 relative (the
// 1e-3 * sum|w x| bound then holds for every input, not only statistically).
#include <cuda.h>
#include <algorithm>
#include <cmath>
#include <cstring>
#include <mutex>

#include "dequant_dot.cuh"
#include "ptx.cuh"

namespace emb {
namespace {

constexpr int kBN = 128;                   // weight rows per CTA (MMA M)
constexpr int kKC = 64;                    // k per A/X stage: one 128-byte bf16 atom row
constexpr int kKR = 256;                   // k per raw stage
constexpr int kStepsPerRaw = kKR / kKC;    // 4
constexpr int kRawStages = 2;
constexpr int kDeqWarps = 8;               // dequantisation (then epilogue) warps
constexpr int kThreads = 32 * (2 + kDeqWarps);
constexpr int kACols = kKC / 2;            // TMEM columns of one bf16 A tile (two values per column)
constexpr uint32_t kTmemCols = 512;        // accumulator + A stages
constexpr int kPlane = kBN * 128;          // 16 KB: 128 rows x 128 bytes of codes
constexpr int kScaleTile = kBN * 16;       // 2 KB: 128 rows x 8 fp16 scales
constexpr int kMaxStages = 8;              // X ring depth, at most
constexpr int kMaxAStages = 8;             // A ring depth, at most

struct GemmParams {
    CUtensorMap x_map;                     // X [M][K] bf16, box {64, T}, 128B swizzle
    const __nv_bfloat16* X;                // the same X (for its L2 prefetch)
    CUtensorMap codes_map[kMaxGroup];      // codes [N][row bytes] u8, box {128, 128}, 128B swizzle
    CUtensorMap scales_map[kMaxGroup];     // scales [N][ldS] u16, box {8, 128}
    CUtensorMap high_map[kMaxGroup];       // Q6_0 high bits [N][K/4] u8, box {64, 128}, no swizzle
    void* Y[kMaxGroup];                    // as the epilogue says
    int32_t N[kMaxGroup];
    int32_t tile0[kMaxGroup + 1];
    int32_t n_mats;
    int32_t M, K;
    int32_t T;                             // tokens per token tile, multiple of 16, <= 256
    int32_t P;                             // token tiles per CTA (1, or 2 sharing each A tile)
    int32_t splits;                        // K splits (cluster size along z)
    int32_t epi;                           // emb_epilogue
    int32_t stages;                        // X ring depth
    int32_t a_stages;                      // A ring depth (TMEM)
    uint32_t tmem_cols;
    int32_t persist;                       // 1: CTAs loop over items (no K split)
    int32_t n_tt, n_items;                 // persistent: token tiles per weight tile, items
    int32_t streamk;                       // 1: the items' raw stages split evenly over the CTAs
    int32_t wait_first;                    // 1: nothing is read before griddepcontrol.wait
    int32_t slot_floats;                   // stream-K: floats of one partial tile (P * T * 128)
    float* ws_part;                        // stream-K: one partial-tile slot per CTA
    uint32_t* ws_flag;                     // stream-K: one ready flag per CTA (zero between launches)
    int* status;
};

template <int FMT>
struct RawTraits {
    static constexpr int planes = (FMT == EMB_Q8_0) ? 2 : 1;  // 128-byte code chunks per raw stage
    static constexpr int bytes = planes * kPlane;
    // Q6_0: the high bits of a raw stage, 64 bytes per row (256 codes x 2 bits)
    static constexpr int hbytes = (FMT == EMB_Q6_0) ? kBN * 64 : 0;
    // w' = d*(f - bias) where f = 2^15 + byte is built by __byte_perm
    static constexpr float bias = (FMT == EMB_Q8_0) ? 32768.0f + 128.0f
                                : (FMT == EMB_Q4_0) ? 32768.0f + 8.0f : 32768.0f + 32.0f;
};

__device__ __forceinline__ uint4 lds128(const uint8_t* p) {
    return *reinterpret_cast<const uint4*>(p);
}

using dq::bytes_to_w;
using dq::pack_bf16;

// 8 consecutive w' (two input words) -> one 16-byte chunk of bf16 (hi), and for the split
// variant the residual chunk lo = bf16(w' - hi).
template <bool SPLIT>
__device__ __forceinline__ void make_chunk(uint32_t u0, uint32_t u1, float d, float nbd,
                                           uint4& hi, uint4& lo) {
    float2 a, b, c, e;
    bytes_to_w(u0, d, nbd, a, b);
    bytes_to_w(u1, d, nbd, c, e);
    hi = make_uint4(pack_bf16(a.x, a.y), pack_bf16(b.x, b.y), pack_bf16(c.x, c.y),
                    pack_bf16(e.x, e.y));
    if constexpr (SPLIT) {
        auto res = [](float2 v, uint32_t h) {
            const float2 hv = make_float2(__uint_as_float(h << 16), __uint_as_float(h & 0xFFFF0000u));
            const float2 r = __fadd2_rn(v, make_float2(-hv.x, -hv.y));  // exact
            return pack_bf16(r.x, r.y);
        };
        lo = make_uint4(res(a, hi.x), res(b, hi.y), res(c, hi.z), res(e, hi.w));
    }
}

// TMEM columns: the accumulators of the CTA's P token tiles, each rounded up to 32 columns,
// then the ring of A tiles (hi and lo tile of a step side by side for the split operand).
__host__ __device__ constexpr int acc_cols(int T) { return (T + 31) & ~31; }
__host__ __device__ constexpr int a_stage_cols(bool split) { return (split ? 2 : 1) * kACols; }

template <int FMT, bool SPLIT, int P, bool SK>
__global__ void __launch_bounds__(kThreads, 1) gemm_tc_kernel(const __grid_constant__ GemmParams p) {
    using RT = RawTraits<FMT>;
    static_assert(P == 1 || (P == 2 && !SPLIT), "two token tiles only without the split operand");
    static_assert(!(SK && SPLIT), "stream-K only without the split operand");
    extern __shared__ uint8_t smem_dyn[];
    uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_dyn) + 1023) &
                                               ~uintptr_t(1023));
    const int S = p.stages, SA = p.a_stages, T = p.T;
    const int a_col0 = P * acc_cols(T);  // TMEM column of the A ring
    uint8_t* x_ring = base;                                     // S x P x T x 128 B
    uint8_t* r_ring = x_ring + S * P * T * 128;                 // 2 x RT::bytes
    uint8_t* s_ring = r_ring + kRawStages * RT::bytes;          // 2 x 2 KB
    uint8_t* h_ring = s_ring + kRawStages * kScaleTile;          // Q6_0: 2 x 8 KB of high bits
    uint64_t* bars = reinterpret_cast<uint64_t*>(h_ring + kRawStages * RT::hbytes);
    uint64_t* raw_full = bars;
    uint64_t* raw_empty = bars + kRawStages;
    uint64_t* x_full = bars + 2 * kRawStages;
    uint64_t* x_empty = x_full + S;
    uint64_t* a_full = x_empty + S;
    uint64_t* a_empty = a_full + SA;
    uint64_t* acc_full = a_empty + SA;
    uint64_t* acc_empty = acc_full + 1;  // the epilogue warps have read the accumulator
    uint64_t* sk_full = acc_empty + 1;   // stream-K head: a chunk of a tail is in the X ring
    uint64_t* sk_free = sk_full + 1;     // stream-K head: every epilogue warp has added it
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(sk_free + 1);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
    int* sk_cnt = const_cast<int*>(abort_flag) + 1;  // stream-K: epilogue warps done with the tail
    int* sk_seen = sk_cnt + 1;                     // stream-K: epilogue warps done with the head
    // split-K partial tile [T][128] fp32 (token-major): reuses the X ring once every MMA
    // has completed
    float* part = reinterpret_cast<float*>(x_ring);

    const int warp = ptx::warp_uniform(int(threadIdx.x >> 5)), lane = threadIdx.x & 31;
    const int M = p.M, K = p.K;
    const int splits = gridDim.z, split = blockIdx.z;
    const int nr_all = (K + kKR - 1) / kKR, nk_all = (K + kKC - 1) / kKC;
    // Work items (weight tile, token tile), each over a range of raw stages (256 k) of its
    // row. Three schedules:
    //  * one item per CTA: grid x = token tile, y = weight tile, z = K split (a cluster
    //    along z shares one item; split s takes raw stages [s*nr/splits, (s+1)*nr/splits));
    //  * p.persist: CTA c takes whole items c, c + gridDim.x, ... in the order of token
    //    tiles within weight tiles, so the CTAs at work on a weight tile at one time read it
    //    once from HBM and then from L2;
    //  * SK (stream-K): the raw stages of all items, item after item, are cut into gridDim.x
    //    equal ranges, one per CTA, so every SM gets the same work whatever the tile count.
    //    A range starts inside an item (a "tail": its sum is left in the CTA's workspace
    //    slot, flagged ready) and/or ends inside one (a "head" holding k = 0: its CTA adds
    //    the tails of the CTAs after it, in CTA order, i.e. in k order, and runs the
    //    epilogue). Results are deterministic for a given grid.
    // With more than one item, rings and barrier phases run on across items; the next
    // item's codes and activations stream in while the current one's epilogue drains the
    // accumulator.
    const bool persist = p.persist != 0;
    constexpr bool streamk = SK;  // a separate instance: the plain schedules carry none of its code
    const int64_t sk_units = int64_t(p.n_items) * nr_all;  // stream-K: raw stages of all items
    // this CTA's segments j = 0 .. n_seg-1: item it0 + j*it_stride over raw stages [r0, r1),
    // r0 = 0 but for the first, r1 = nr_all but for the last
    int it0 = 0, it_stride = 1, r0_first = 0, r1_last = nr_all, n_seg = 1;
    if (streamk) {
        const int64_t u_beg = int64_t(blockIdx.x) * sk_units / gridDim.x;
        const int64_t u_end = int64_t(blockIdx.x + 1) * sk_units / gridDim.x;
        const int64_t last = (u_end - 1) / nr_all;
        it0 = int(u_beg / nr_all);
        r0_first = int(u_beg - int64_t(it0) * nr_all);
        r1_last = int(u_end - last * nr_all);
        n_seg = u_end > u_beg ? int(last) - it0 + 1 : 0;
    } else if (persist) {
        it0 = int(blockIdx.x);
        it_stride = int(gridDim.x);
        n_seg = int(blockIdx.x) < p.n_items ? (p.n_items - int(blockIdx.x) + int(gridDim.x) - 1) / int(gridDim.x) : 0;
    } else {
        r0_first = split * nr_all / splits;
        r1_last = (split + 1) * nr_all / splits;
    }
    // stream-K: a head (last segment holding k = 0 of an item that goes on) adds the tails of
    // CTAs [blockIdx.x + 1, sk_q_end): those whose ranges start inside that item
    int sk_q_end = int(blockIdx.x) + 1;
    if (streamk && n_seg > 0 && r1_last < nr_all && (n_seg > 1 || r0_first == 0)) {
        const int64_t item_end = int64_t(it0 + n_seg) * nr_all;
        while (sk_q_end < int(gridDim.x) && int64_t(sk_q_end) * sk_units / gridDim.x < item_end) ++sk_q_end;
    }
    struct Seg {
        int it, r0, r1;  // item, raw stages [r0, r1) of its row
    };
    auto seg_at = [&](int j) {
        Seg s;
        s.it = it0 + j * it_stride;
        s.r0 = j == 0 ? r0_first : 0;
        s.r1 = j == n_seg - 1 ? r1_last : nr_all;
        return s;
    };
    auto seg_nk = [&](const Seg& s) { return min(s.r1 * kStepsPerRaw, nk_all) - s.r0 * kStepsPerRaw; };
    struct Item {
        int g, n0, m0, N;
    };
    auto item_at = [&](int it) {
        const int tt = (persist || streamk) ? it % p.n_tt : int(blockIdx.x);
        const int tile = (persist || streamk) ? it / p.n_tt : int(blockIdx.y);
        Item r;
        r.g = 0;
#pragma unroll
        for (int i = 1; i < kMaxGroup; ++i)
            if (i < p.n_mats && tile >= p.tile0[i]) r.g = i;
        r.n0 = (tile - p.tile0[r.g]) * kBN;
        r.m0 = tt * P * T;  // first token of the item's first token tile
        r.N = p.N[r.g];
        return r;
    };

    if (threadIdx.x == 0) {
        for (int i = 0; i < kRawStages; ++i) {
            ptx::mbar_init(&raw_full[i], 1);
            ptx::mbar_init(&raw_empty[i], kDeqWarps);
        }
        for (int i = 0; i < S; ++i) {
            ptx::mbar_init(&x_full[i], 1);
            ptx::mbar_init(&x_empty[i], 1);
        }
        for (int i = 0; i < SA; ++i) {
            ptx::mbar_init(&a_full[i], kDeqWarps);
            ptx::mbar_init(&a_empty[i], 1);
        }
        ptx::mbar_init(acc_full, 1);
        ptx::mbar_init(acc_empty, kDeqWarps);
        ptx::mbar_init(sk_full, 1);
        ptx::mbar_init(sk_free, kDeqWarps);
        *abort_flag = 0;
        *sk_cnt = 0;
        *sk_seen = 0;
        ptx::fence_mbar_init();
        ptx::prefetch_tmap(&p.x_map);
        for (int i = 0; i < p.n_mats; ++i) {
            ptx::prefetch_tmap(&p.codes_map[i]);
            ptx::prefetch_tmap(&p.scales_map[i]);
            if constexpr (FMT == EMB_Q6_0) ptx::prefetch_tmap(&p.high_map[i]);
        }
    }
    if (warp == 1) {
        // all 512 columns: one CTA per SM (see ptx::tmem_alloc for why this never waits)
        ptx::tmem_alloc(tmem_slot, p.tmem_cols);
        ptx::tmem_relinquish();
    }
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    const uint32_t tmem = ptx::warp_uniform(*tmem_slot);
    if (p.wait_first) ptx::griddep_wait();  // every thread before the trigger: see ptx::griddep_launch_dependents
    ptx::griddep_launch_dependents();
    int items_done = 0;  // this CTA's items started by its role (phase of acc_full / acc_empty)

    if (warp == 0) {
        // -------------------------------------------------------------------- producer
        // the whole warp runs the loop; one elected lane issues the copies (see ptx::elect_one)
        const unsigned full = 0xffffffffu;
        const uint64_t pol_w = ptx::policy_evict_first();
        const uint64_t pol_x = ptx::policy_evict_last();
        int raw_issued = 0, x_issued = 0;  // over all items of the CTA
        bool stop = false, waited = false;
        int rbase = 0;         // raw stages of the earlier segments
        int s = 0;             // X stage, and how often the ring has gone round
        uint32_t xround = 0;
        for (int j = 0; j < n_seg && !stop; ++j, ++items_done) {
            const Seg sg = seg_at(j);
            const Item I = item_at(sg.it);
            const int nr = sg.r1 - sg.r0, nk = seg_nk(sg), ks0 = sg.r0 * kStepsPerRaw;
            auto issue_raw = [&](int r) {  // raw stage r of this segment (global rbase + r)
                const int slot = (rbase + r) % kRawStages;
                const int rg = sg.r0 + r;  // raw stage index within the whole row
                if (ptx::elect_one()) {
                    ptx::mbar_arrive_expect_tx(&raw_full[slot], RT::bytes + RT::hbytes + kScaleTile);
#pragma unroll
                    for (int pl = 0; pl < RT::planes; ++pl)
                        ptx::tma_load_2d(r_ring + slot * RT::bytes + pl * kPlane, &p.codes_map[I.g],
                                         &raw_full[slot], (rg * RT::planes + pl) * 128, I.n0, pol_w);
                    if constexpr (FMT == EMB_Q6_0)  // x = 64 bytes per raw stage: 16-byte aligned
                        ptx::tma_load_2d(h_ring + slot * RT::hbytes, &p.high_map[I.g], &raw_full[slot],
                                         rg * 64, I.n0, pol_w);
                    ptx::tma_load_2d(s_ring + slot * kScaleTile, &p.scales_map[I.g], &raw_full[slot],
                                     rg * (kKR / kQBlock), I.n0, pol_w);
                }
                __syncwarp();
            };
            if (!waited) {
                // the first raw stages before griddepcontrol.wait: weights never depend on
                // the previous launch; X may be written by it, so only its rows' way towards
                // L2 starts now (a hint: the TMA loads after the wait read the written values)
                for (; raw_issued < nr && raw_issued < kRawStages; ++raw_issued) issue_raw(raw_issued);
                const int x_rows = min(M - I.m0, P * T);
                if (lane == 0 && x_rows > 0 && I.n0 == 0 && I.g == 0 && sg.r0 == 0)  // one CTA per token tile
                    ptx::prefetch_l2(reinterpret_cast<const uint8_t*>(p.X) + int64_t(I.m0) * K * 2,
                                     uint32_t(min(int64_t(x_rows) * K * 2, int64_t(1) << 20)));
                ptx::griddep_wait();
                waited = true;
            }
            for (int i = 0; i < nk; ++i) {
                if (i % kStepsPerRaw == 0) {
                    const int rg_all = rbase + i / kStepsPerRaw;
                    if (rg_all >= raw_issued) {
                        if (rg_all >= kRawStages &&
                            !__all_sync(full, ptx::mbar_wait(&raw_empty[rg_all % kRawStages], ((rg_all / kRawStages) - 1) & 1,
                                                             abort_flag, p.status, kWaitLimitNs))) {
                            stop = true;
                            break;
                        }
                        issue_raw(i / kStepsPerRaw);
                        ++raw_issued;
                    }
                }
                if (xround > 0 && !__all_sync(full, ptx::mbar_wait(&x_empty[s], (xround - 1) & 1, abort_flag, p.status,
                                                                   kWaitLimitNs))) {
                    stop = true;
                    break;
                }
                if (ptx::elect_one()) {
                    ptx::mbar_arrive_expect_tx(&x_full[s], uint32_t(P * T) * 128u);
#pragma unroll
                    for (int q = 0; q < P; ++q)  // a tile past M reads zeros (its outputs are not stored)
                        ptx::tma_load_2d(x_ring + (s * P + q) * T * 128, &p.x_map, &x_full[s],
                                         (ks0 + i) * kKC, I.m0 + q * T, pol_x);
                }
                __syncwarp();
                ++x_issued;
                if (++s == S) {
                    s = 0;
                    ++xround;
                }
            }
            rbase += nr;
        }
        // every issued copy must land before this CTA's shared memory can be released
        for (int r = raw_issued - 1; r >= 0 && r >= raw_issued - kRawStages; --r)
            ptx::mbar_wait(&raw_full[r % kRawStages], (r / kRawStages) & 1, nullptr, p.status,
                           kWaitLimitNs);
        for (int i = x_issued - 1; i >= 0 && i >= x_issued - S; --i)
            ptx::mbar_wait(&x_full[i % S], (i / S) & 1, nullptr, p.status, kWaitLimitNs);
    } else if (warp == 1) {
        // ---------------------------------------------------------------- MMA issuer
        // the whole warp waits for step i's X tile and A tile (and, at an item's first step, for
        // the previous item's epilogue to have read the accumulator); one elected lane issues
        const unsigned full = 0xffffffffu;
        const uint32_t idesc = ptx::idesc_bf16_f32(kBN, T);
        const uint32_t x0 = ptx::smem_u32(x_ring);
        bool stop = false;
        int commits = 0;  // accumulator commits (one per finished segment)
        int s = 0, a = 0;  // X and A ring stages of the step and their phases
        uint32_t ph = 0, pha = 0;
        for (int j = 0; j < n_seg && !stop; ++j, ++items_done) {
            const int nk = seg_nk(seg_at(j));
            for (int i = 0; i < nk; ++i) {
                bool ok = true;
                if (i == 0 && items_done > 0)
                    ok = ptx::mbar_wait(acc_empty, (items_done - 1) & 1, abort_flag, p.status, kWaitLimitNs);
                ok = ok && ptx::mbar_wait(&x_full[s], ph, abort_flag, p.status, kWaitLimitNs) &&
                     ptx::mbar_wait(&a_full[a], pha, abort_flag, p.status, kWaitLimitNs);
                if (!__all_sync(full, ok)) {
                    stop = true;
                    break;
                }
                ptx::tc_fence_after();
                const uint32_t a_tm = tmem + uint32_t(a_col0 + a * a_stage_cols(SPLIT));
#pragma unroll
                for (int q = 0; q < P; ++q) {
                    // token tile q: its own X tile and accumulator, the same A tile
                    const uint64_t bdesc = ptx::smem_desc_sw128(x0 + (s * P + q) * T * 128);
                    const uint32_t d_tm = tmem + uint32_t(q * acc_cols(T));
#pragma unroll
                    for (int k = 0; k < kKC / 16; ++k) {  // 32 bytes along K: two 16-byte units
                        ptx::mma_bf16_ta(d_tm, a_tm + 8 * k, bdesc + 2 * k, idesc, (i | k) != 0);
                        if constexpr (SPLIT) ptx::mma_bf16_ta(d_tm, a_tm + kACols + 8 * k, bdesc + 2 * k, idesc, 1u);
                    }
                }
                ptx::mma_commit(&a_empty[a]);
                ptx::mma_commit(&x_empty[s]);
                if (++s == S) {
                    s = 0;
                    ph ^= 1u;
                }
                if (++a == SA) {
                    a = 0;
                    pha ^= 1u;
                }
            }
            // the item's accumulator is complete once every MMA issued so far has finished
            // (after a wait gave up: the MMAs issued so far, so that they finish before TMEM is freed)
            ptx::mma_commit(acc_full);
            ++commits;
        }
        if (commits > 0)  // the last item's MMAs finish before TMEM is freed
            ptx::mbar_wait(acc_full, (commits - 1) & 1, nullptr, p.status, kWaitLimitNs);
    } else {
        // ---------------------------------------------------------------- dequant
        // two threads per weight row: thread (row t, half h) produces 32 of the 64 bf16 of
        // each 64-k step (32-block 2j+h of step j) and stores them into its TMEM lane t,
        // 16 columns; a warp reaches only its lane quarter (warp % 4), so t = 32*(warp%4) + lane
        const int t = 32 * (warp & 3) + lane, h = (warp - 2) >> 2;
        const uint32_t a_lane = tmem + (uint32_t(32 * (warp & 3)) << 16) + uint32_t(16 * h);
        const unsigned full = 0xffffffffu;
        bool ok = true;
        int rbase = 0, xbase = 0;  // raw stages and steps of the earlier segments
        for (int j = 0; j < n_seg && ok; ++j, ++items_done) {
            const Seg sg = seg_at(j);
            const Item I = item_at(sg.it);
            const int nr = sg.r1 - sg.r0, nk = seg_nk(sg);
            // Software pipeline: step i's TMEM stores are completed (tcgen05.wait::st) and
            // signalled only after step i+1 has been computed, so the store latency overlaps
            // the next step's arithmetic instead of stalling this warp every step.
            int pending = -1;  // A stage whose stores are in flight, not yet signalled
            auto signal_pending = [&]() {
                if (pending >= 0) {
                    ptx::tmem_st_wait();
                    ptx::tc_fence_before();  // the stores are ordered before the arrive
                    __syncwarp();
                    if (lane == 0) ptx::mbar_arrive(&a_full[pending]);
                    pending = -1;
                }
            };
            for (int r = 0; r < nr && ok; ++r) {
                const int rg_all = rbase + r;
                const int rs = rg_all % kRawStages;
                ok = __all_sync(full, ptx::mbar_wait(&raw_full[rs], (rg_all / kRawStages) & 1, abort_flag,
                                                     p.status, kWaitLimitNs));
                if (!ok) break;
                const uint8_t* rbase_p = r_ring + rs * RT::bytes + t * 128;
                const uint4 sv = lds128(s_ring + rs * kScaleTile + t * 16);
                const uint32_t sw[4] = {sv.x, sv.y, sv.z, sv.w};
                float d[4], nbd[4];  // scale of block 2j + h (word j, half h), j = 0..3
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const uint16_t hb = uint16_t((sw[j] >> (16 * h)) & 0xFFFFu);
                    d[j] = __half2float(__ushort_as_half(hb));
                    nbd[j] = -RT::bias * d[j];  // exact (see bytes_to_w)
                }
#pragma unroll
                for (int j = 0; j < kStepsPerRaw; ++j) {
                    const int i = r * kStepsPerRaw + j;
                    if (i >= nk) break;
                    const int xs = xbase + i;
                    const int s = xs % SA;
                    const uint32_t a_dst = a_lane + uint32_t(a_col0 + s * a_stage_cols(SPLIT));
                    const int sx = t & 7;  // raw codes: 16-byte chunk c of row t lives at c ^ (t & 7)
                    uint32_t va[16], vl[16];  // this thread's 16 columns of the hi (and lo) tile
                    if constexpr (FMT == EMB_Q8_0) {
                        // atom j: codes 64j..64j+63 of the raw stage = plane j/2, chunks 4(j%2)..+3;
                        // this half: chunks 4(j%2)+2h, +1 (block 2j+h) -> output chunks 4h..4h+3
#pragma unroll
                        for (int e = 0; e < 2; ++e) {
                            const int cc = 2 * h + e;
                            const int c = (j & 1) * 4 + cc;
                            const uint4 v = lds128(rbase_p + (j >> 1) * kPlane + ((c ^ sx) << 4));
                            uint4 h0, l0, h1, l1;
                            make_chunk<SPLIT>(v.x ^ 0x80808080u, v.y ^ 0x80808080u, d[j], nbd[j], h0, l0);
                            make_chunk<SPLIT>(v.z ^ 0x80808080u, v.w ^ 0x80808080u, d[j], nbd[j], h1, l1);
                            // output chunks 2cc, 2cc+1 (k = 16cc .. 16cc+15) -> columns 8e .. 8e+7
                            const int q = 8 * e;
                            va[q + 0] = h0.x; va[q + 1] = h0.y; va[q + 2] = h0.z; va[q + 3] = h0.w;
                            va[q + 4] = h1.x; va[q + 5] = h1.y; va[q + 6] = h1.z; va[q + 7] = h1.w;
                            if constexpr (SPLIT) {
                                vl[q + 0] = l0.x; vl[q + 1] = l0.y; vl[q + 2] = l0.z; vl[q + 3] = l0.w;
                                vl[q + 4] = l1.x; vl[q + 5] = l1.y; vl[q + 6] = l1.z; vl[q + 7] = l1.w;
                            }
                        }
                    } else {
                        // atom j: blocks 2j, 2j+1; this half: block 2j+h -> output chunks 4h..4h+3.
                        // A block's byte i holds code i (low nibble) and code i+16 (high nibble).
                        const int b = 2 * j + h;
                        const uint4 v = lds128(rbase_p + ((b ^ sx) << 4));
                        const uint32_t m = 0x0F0F0F0Fu;
                        // Q4_0: the nibbles are the codes. Q6_0: OR in the high bits so that every
                        // byte holds a whole code: high word (w & 1) >> 2(w >> 1) has the high bits
                        // of low word w's codes at bits 0-1 (codes 4w+i) and 4-5 (codes 16+4w+i).
                        uint32_t c0 = v.x & m, c1 = v.y & m, c2 = v.z & m, c3 = v.w & m;
                        uint32_t e0 = (v.x >> 4) & m, e1 = (v.y >> 4) & m, e2 = (v.z >> 4) & m, e3 = (v.w >> 4) & m;
                        if constexpr (FMT == EMB_Q6_0) {
                            const uint2 hv = *reinterpret_cast<const uint2*>(h_ring + rs * RT::hbytes + t * 64 + b * 8);
                            const uint32_t hw[4] = {hv.x, hv.y, hv.x >> 2, hv.y >> 2};
                            c0 |= (hw[0] & 0x03030303u) << 4; e0 |= hw[0] & 0x30303030u;
                            c1 |= (hw[1] & 0x03030303u) << 4; e1 |= hw[1] & 0x30303030u;
                            c2 |= (hw[2] & 0x03030303u) << 4; e2 |= hw[2] & 0x30303030u;
                            c3 |= (hw[3] & 0x03030303u) << 4; e3 |= hw[3] & 0x30303030u;
                        }
                        uint4 hh[4], ll[4];
                        make_chunk<SPLIT>(c0, c1, d[j], nbd[j], hh[0], ll[0]);  // codes 0..7
                        make_chunk<SPLIT>(c2, c3, d[j], nbd[j], hh[1], ll[1]);  // 8..15
                        make_chunk<SPLIT>(e0, e1, d[j], nbd[j], hh[2], ll[2]);  // 16..23
                        make_chunk<SPLIT>(e2, e3, d[j], nbd[j], hh[3], ll[3]);  // 24..31
#pragma unroll
                        for (int q = 0; q < 4; ++q) {  // output chunk 4h+q -> columns 4q .. 4q+3
                            va[4 * q + 0] = hh[q].x; va[4 * q + 1] = hh[q].y;
                            va[4 * q + 2] = hh[q].z; va[4 * q + 3] = hh[q].w;
                            if constexpr (SPLIT) {
                                vl[4 * q + 0] = ll[q].x; vl[4 * q + 1] = ll[q].y;
                                vl[4 * q + 2] = ll[q].z; vl[4 * q + 3] = ll[q].w;
                            }
                        }
                    }
                    signal_pending();
                    if (xs >= SA) {
                        ok = __all_sync(full, ptx::mbar_wait(&a_empty[s], ((xs / SA) - 1) & 1, abort_flag,
                                                             p.status, kWaitLimitNs));
                        if (!ok) break;
                        ptx::tc_fence_after();  // the MMAs that read this A stage have completed
                    }
                    ptx::tmem_st_16(a_dst, va);
                    if constexpr (SPLIT) ptx::tmem_st_16(a_dst + kACols, vl);
                    pending = s;
                }
                if (!ok) break;
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive(&raw_empty[rs]);
            }
            if (ok) signal_pending();
            ptx::tmem_st_wait();  // no store of this warp is left in flight, whatever happened

            // ---------------------------------------------------------------- epilogue
            ptx::griddep_wait();  // Y may be read or written by the previous launch
            ok = __all_sync(full, ok && ptx::mbar_wait(acc_full, items_done & 1, abort_flag, p.status,
                                                       kWaitLimitNs));
            // stream-K: a tail goes to this CTA's workspace slot; a head first adds the tails of
            // the CTAs after it (those whose ranges start inside this item), in CTA order
            const bool sk_tail = streamk && sg.r0 > 0;
            const bool sk_head = streamk && sg.r0 == 0 && sg.r1 < nr_all;
            if (ok) {
                ptx::tc_fence_after();
                // TMEM lane quarter = warp % 4; the warps of a quarter take the 16-column groups of
                // the item's P * T token columns in turn
                const int quarter = warp & 3, slot = (warp - 2) >> 2;
                constexpr int kStride = 16 * (kDeqWarps / 4);
                const int row = quarter * 32 + lane;
                const uint32_t tlane = tmem + (uint32_t(quarter * 32) << 16);
                auto tcol = [&](int c) { return uint32_t(P == 2 && c >= T ? c - T + acc_cols(T) : c); };
                const int n = I.n0 + row, N = I.N;
                const int mt = I.m0;  // token of column 0
                void* Y = p.Y[I.g];
                const int epi = p.epi;
                // Emit 16 accumulator columns c0 .. c0+15 of this warp's rows, plus (stream-K
                // head) the staged last tail
                const uint32_t staged = ptx::smem_u32(x_ring);  // staged tail: [cols][128] fp32
                bool add_staged = false;
                auto emit = [&](uint32_t (&v)[16], int c0) {
                    if (add_staged) {
#pragma unroll
                        for (int e = 0; e < 16; ++e)
                            v[e] = __float_as_uint(__fadd_rn(
                                __uint_as_float(v[e]), ptx::ld_shared_f32(staged + uint32_t(((c0 + e) * kBN + row) * 4))));
                    }
                    if (splits == 1) {
                        if (epi >= EMB_EPI_GEGLU) {
                            // gate rows sit in even lanes, their up rows in the next lane: of tokens e
                            // and e + 1 the even lane takes the first and the odd lane the second, each
                            // getting the other half of its pair by one exchange, so that every lane
                            // evaluates an activation. Rows past N hold zeros (their weights were read
                            // as zeros), so every lane shuffles.
                            const int odd = lane & 1;
#pragma unroll
                            for (int e = 0; e < 16; e += 2) {
                                const float a = __uint_as_float(v[e]), b = __uint_as_float(v[e + 1]);
                                const float r = __shfl_xor_sync(0xffffffffu, odd ? a : b, 1);
                                const int m = mt + c0 + e + odd;
                                if (n < N && m < M)
                                    epi_store_gated(epi, Y, m, n - odd, N, odd ? r : a, odd ? b : r);
                            }
                        } else if (epi == EMB_EPI_ADD && n < N) {
                            // every read ahead of the stores: a read after a store to the same buffer
                            // would otherwise wait for that store
                            float* y = reinterpret_cast<float*>(Y) + int64_t(mt + c0) * N + n;
                            float old[16];
#pragma unroll
                            for (int e = 0; e < 16; ++e) old[e] = (mt + c0 + e < M) ? y[int64_t(e) * N] : 0.0f;
#pragma unroll
                            for (int e = 0; e < 16; ++e)
                                if (mt + c0 + e < M) y[int64_t(e) * N] = __fadd_rn(old[e], __uint_as_float(v[e]));
                        } else if (n < N) {
#pragma unroll
                            for (int e = 0; e < 16; ++e) {
                                const int m = mt + c0 + e;
                                if (m < M) epi_store(epi, Y, m, n, N, __uint_as_float(v[e]));
                            }
                        }
                    } else {
                        // token-major partial tile part[m][row] (a warp writes 32 consecutive rows)
#pragma unroll
                        for (int e = 0; e < 16; ++e) part[(c0 + e) * kBN + row] = __uint_as_float(v[e]);
                    }
                };
                if (sk_head) {
                    // Workspace slots are token-major [P*T][128] fp32. Each tail is staged into the
                    // (now idle) X ring by bulk copies, in column chunks that fit it. Every tail but
                    // the last is added into the accumulator in TMEM; the last one, when it fits in
                    // one chunk, is added by the store pass below.
                    const int slot_cols = P * T;
                    const int chunk_cols = min(slot_cols, ((S * P * T) / 4) & ~15);  // X ring bytes / 512
                    int chunk_no = 0;
                    for (int q = int(blockIdx.x) + 1; q < sk_q_end && ok; ++q) {
                        for (int k0 = 0; k0 < slot_cols && ok; k0 += chunk_cols, ++chunk_no) {
                            const int k1 = min(slot_cols, k0 + chunk_cols);
                            if (warp == 2 && lane == 0) {
                                bool good = true;
                                if (k0 == 0) {
                                    good = ptx::flag_wait(p.ws_flag + q, abort_flag, p.status, kWaitLimitNs);
                                    ptx::fence_proxy_async_global();  // the tail's stores, seen by the copy
                                }
                                if (good && chunk_no > 0)  // every warp has read the previous chunk
                                    good = ptx::mbar_wait(sk_free, (chunk_no - 1) & 1, abort_flag, p.status,
                                                          kWaitLimitNs);
                                if (good) {
                                    const uint32_t bytes = uint32_t(k1 - k0) * uint32_t(kBN) * 4u;
                                    ptx::mbar_arrive_expect_tx(sk_full, bytes);
                                    ptx::bulk_load(x_ring, p.ws_part + int64_t(q) * p.slot_floats + int64_t(k0) * kBN,
                                                   bytes, sk_full);
                                }
                            }
                            ok = __all_sync(full, ptx::mbar_wait(sk_full, chunk_no & 1, abort_flag, p.status,
                                                                 kWaitLimitNs));
                            if (!ok) break;
                            if (q == sk_q_end - 1 && chunk_cols == slot_cols) {
                                add_staged = true;  // the store pass adds it
                                break;
                            }
                            for (int c0 = 16 * slot; c0 < P * T; c0 += kStride) {
                                if (c0 < k0 || c0 >= k1) continue;  // chunks are whole 16-column groups
                                uint32_t v[16];
                                ptx::tmem_ld_16(tlane + tcol(c0), v);
                                ptx::tmem_ld_wait();
#pragma unroll
                                for (int e = 0; e < 16; ++e)
                                    v[e] = __float_as_uint(__fadd_rn(
                                        __uint_as_float(v[e]), ptx::ld_shared_f32(staged + uint32_t(((c0 - k0 + e) * kBN + row) * 4))));
                                ptx::tmem_st_16(tlane + tcol(c0), v);
                            }
                            ptx::tmem_st_wait();
                            __syncwarp();
                            if (lane == 0) ptx::mbar_arrive(sk_free);
                        }
                    }
                }
                if (sk_tail) {
                    float* part_out = p.ws_part + int64_t(blockIdx.x) * p.slot_floats;
                    for (int c0 = 16 * slot; c0 < P * T; c0 += kStride) {
                        uint32_t v[16];
                        ptx::tmem_ld_16(tlane + tcol(c0), v);
                        ptx::tmem_ld_wait();
                        float* dst = part_out + int64_t(c0) * kBN + row;  // a warp writes 32 consecutive rows
#pragma unroll
                        for (int e = 0; e < 16; ++e) __stcg(dst + e * kBN, __uint_as_float(v[e]));
                    }
                    // the last of the eight warps to finish publishes the tail
                    __threadfence();
                    __syncwarp();
                    if (lane == 0 && atomicAdd(sk_cnt, 1) == kDeqWarps - 1) {
                        __threadfence();
                        ptx::st_release_gpu(p.ws_flag + blockIdx.x, 1u);
                    }
                } else if (ok) {
                    // one TMEM load per wait (two per wait measured slower on GB300: the kernel's
                    // register count rose by 16 and the main loop lost 10-17 %)
                    for (int c0 = 16 * slot; c0 < P * T; c0 += kStride) {
                        uint32_t v[16];
                        ptx::tmem_ld_16(tlane + tcol(c0), v);
                        ptx::tmem_ld_wait();
                        emit(v, c0);
                    }
                }
                if (sk_head && ok) {
                    // the last of the eight warps to finish clears the flags it consumed
                    __syncwarp();
                    if (lane == 0 && atomicAdd(sk_seen, 1) == kDeqWarps - 1)
                        for (int q = int(blockIdx.x) + 1; q < sk_q_end; ++q) ptx::st_relaxed_gpu(p.ws_flag + q, 0u);
                }
                // the accumulator may be overwritten by the next item's MMAs
                ptx::tc_fence_before();
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive(acc_empty);
            }
            rbase += nr;
            xbase += nk;
        }
    }
    // the split-K exchange below (never persistent: one item per CTA) sums that item's tile
    const Item I_one = item_at(0);
    const int n0 = I_one.n0, m0 = I_one.m0, N = I_one.N, g = I_one.g;

    __syncwarp();  // the producer / MMA warps reconverge before the block-wide barriers
    ptx::tc_fence_before();
    if (splits > 1) {
        // split-K: every CTA of the cluster holds its partial tile; CTA s sums rows
        // [s*128/splits, (s+1)*128/splits) over the cluster in a fixed order through
        // distributed shared memory and stores them (deterministic, no global scratch)
        ptx::cluster_sync();
        if (!*abort_flag) {
            ptx::griddep_wait();  // (the MMA warp has not waited yet)
            // one thread of any warp = 4 consecutive rows of one token: 16-byte remote loads and
            // 16-byte coalesced stores to Y[m][n..n+3]
            const int rows = kBN / splits, r0 = split * rows, q4 = rows / 4;
            const uint32_t pbase = ptx::smem_u32(part);
            void* Y = p.Y[g];
            const int epi = p.epi;
            const bool vec = (N % 4) == 0;
            for (int w = threadIdx.x; w < q4 * T; w += kThreads) {
                const int c = w / q4, row = r0 + 4 * (w - c * q4);
                const int m = m0 + c, n = n0 + row;
                const uint32_t off = pbase + uint32_t(c * kBN + row) * 4u;
                float4 acc = ptx::ld_dsmem_f32x4(ptx::map_dsmem(off, 0));
                for (int q = 1; q < splits; ++q) {
                    const float4 v = ptx::ld_dsmem_f32x4(ptx::map_dsmem(off, q));
                    acc.x += v.x; acc.y += v.y; acc.z += v.z; acc.w += v.w;
                }
                if (m < M) {
                    if (vec && n + 3 < N) {
                        epi_store4(epi, Y, m, n, N, acc);
                    } else if (epi >= EMB_EPI_GEGLU) {  // rows n, n + 2 are gate rows (n % 4 == 0)
                        if (n < N) epi_store_gated(epi, Y, m, n, N, acc.x, acc.y);
                        if (n + 2 < N) epi_store_gated(epi, Y, m, n + 2, N, acc.z, acc.w);
                    } else {
                        if (n < N) epi_store(epi, Y, m, n, N, acc.x);
                        if (n + 1 < N) epi_store(epi, Y, m, n + 1, N, acc.y);
                        if (n + 2 < N) epi_store(epi, Y, m, n + 2, N, acc.z);
                        if (n + 3 < N) epi_store(epi, Y, m, n + 3, N, acc.w);
                    }
                }
            }
        }
        ptx::cluster_sync();  // remote shared memory must outlive its readers
    } else {
        __syncthreads();
    }
    if (warp == 1) {
        __syncwarp();
        ptx::tc_fence_after();
        ptx::tmem_dealloc(tmem, p.tmem_cols);
    }
}

// ------------------------------------------------------------------ host side

using EncodeTiledFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*,
                                   const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                                   const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                   CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
    static EncodeTiledFn fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void* f = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault,
                                             &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(f);
    });
    return fn;
}

bool encode_2d(CUtensorMap* m, CUtensorMapDataType dt, const void* base, uint64_t inner,
               uint64_t outer, uint64_t row_stride_bytes, uint32_t box_inner, uint32_t box_outer,
               CUtensorMapSwizzle sw, CUtensorMapL2promotion l2) {
    EncodeTiledFn fn = encode_fn();
    if (!fn) return false;
    const cuuint64_t dims[2] = {inner, outer};
    const cuuint64_t strides[1] = {row_stride_bytes};
    const cuuint32_t box[2] = {box_inner, box_outer};
    const cuuint32_t estr[2] = {1, 1};
    return fn(m, dt, 2, const_cast<void*>(base), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, sw, l2, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) ==
           CUDA_SUCCESS;
}

constexpr int kSmemLimit = 227 * 1024;

// Every CTA allocates all 512 TMEM columns, so no two may share an SM (a second one
// would block in tcgen05.alloc, and inside a split-K cluster wait on the first forever):
// the dynamic shared memory is padded above half of the SM's.
constexpr int kOneCtaPerSm = 120 * 1024;

template <int FMT, bool SPLIT>
int smem_bytes(int T, int S, int P) {
    const int need = 1024 + S * P * T * 128 +
                     kRawStages * (RawTraits<FMT>::bytes + RawTraits<FMT>::hbytes + kScaleTile) +
                     (2 * kRawStages + 2 * S + 2 * kMaxAStages + 4) * 8 + 32;
    return need > kOneCtaPerSm ? need : kOneCtaPerSm;
}

// X ring depth: as many stages as shared memory holds, at most kMaxStages.
template <int FMT, bool SPLIT>
int pick_stages(int T) {
    int S = kMaxStages;
    while (S > 2 && smem_bytes<FMT, SPLIT>(T, S, 1) > kSmemLimit) --S;
    return S;
}

// A ring depth: the tiles that fit TMEM beside the accumulators, at most kMaxAStages.
int a_stages_of(bool split, int T, int P) {
    return std::min(kMaxAStages, (int(kTmemCols) - P * acc_cols(T)) / a_stage_cols(split));
}

// X ring depth with two token tiles per CTA (P = 2), each at most 224 tokens; 0 if fewer than
// two stages fit shared memory or two A tiles TMEM.
template <int FMT>
int pick_stages_pair(int T) {
    if (a_stages_of(false, T, 2) < 2) return 0;
    int S = kMaxStages;
    while (S > 2 && smem_bytes<FMT, false>(T, S, 2) > kSmemLimit) --S;
    if (smem_bytes<FMT, false>(T, S, 2) > kSmemLimit) return 0;
    return S;
}

template <int FMT, bool SPLIT, int P, bool SK = false>
cudaError_t launch_kernel(const GemmParams& p, int grid_x, int grid_y, cudaStream_t s) {
    // grid: x = token tile (fastest, so the CTAs sharing a weight tile run together and
    // read it from L2 after the first), y = weight-row tile, z = K split (one cluster)
    const int bytes = smem_bytes<FMT, SPLIT>(p.T, p.stages, p.P);
    // the opt-in shared-memory size is a per-device function attribute
    static std::mutex mu;
    static bool done[64] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    {
        std::lock_guard<std::mutex> lock(mu);
        if (dev < 0 || dev >= 64 || !done[dev]) {
            e = cudaFuncSetAttribute(gemm_tc_kernel<FMT, SPLIT, P, SK>,
                                     cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemLimit);
            if (e != cudaSuccess) return e;
            if (dev >= 0 && dev < 64) done[dev] = true;
        }
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid_x, grid_y, p.splits);
    cfg.blockDim = dim3(kThreads, 1, 1);
    cfg.dynamicSmemBytes = size_t(bytes);
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    int na = 1;
    if (p.splits > 1) {
        attr[na].id = cudaLaunchAttributeClusterDimension;
        attr[na].val.clusterDim.x = 1;
        attr[na].val.clusterDim.y = 1;
        attr[na].val.clusterDim.z = unsigned(p.splits);
        ++na;
    }
    cfg.attrs = attr;
    cfg.numAttrs = na;
    return cudaLaunchKernelEx(&cfg, gemm_tc_kernel<FMT, SPLIT, P, SK>, p);
}

// Clusters of 2^i GEMM CTAs (one CTA per SM) that run at once, n[0] = SMs: fewer than SMs / 2^i, since
// a cluster stays within a part of the chip (GB300, 152 SMs: 76, 36 and 15 of two, four and eight; a
// 37th cluster of four doubles a launch, 19.4 -> 35.1 us, a 16th of eight too, 13.3 -> 23.5).
struct Resident {
    int n[4];
};
Resident resident_clusters() {
    static std::mutex mu;
    static Resident known[64] = {};
    int dev = 0;
    const int sms = device_sm_count();
    Resident r = {{sms, sms / 2, sms / 4, sms / 8}};
    if (sms <= 0 || cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return r;
    std::lock_guard<std::mutex> lock(mu);
    if (known[dev].n[0]) return known[dev];
    auto* kernel = gemm_tc_kernel<EMB_Q8_0, false, 1, false>;
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemLimit) != cudaSuccess) return r;
    for (int i = 1; i < 4; ++i) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(1, 1, 1u << i);
        cfg.blockDim = dim3(kThreads, 1, 1);
        cfg.dynamicSmemBytes = kSmemLimit;
        cudaLaunchAttribute attr;
        attr.id = cudaLaunchAttributeClusterDimension;
        attr.val.clusterDim.x = 1;
        attr.val.clusterDim.y = 1;
        attr.val.clusterDim.z = 1u << i;
        cfg.attrs = &attr;
        cfg.numAttrs = 1;
        int n = 0;
        if (cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) != cudaSuccess || n < 1) return r;
        r.n[i] = n;
    }
    known[dev] = r;
    return r;
}

// K splits (1, 2, 4 or 8: one cluster of CTAs per output tile, 8 being the portable
// cluster size) of the two-operand form and of fewer than 65 tokens: the count minimising a simple
// time model -- waves of 148 CTAs, each costing a fixed ~3 us plus its share of the tile's MMA work
// at ~11.6 TFLOP/s per SM -- subject to every split owning at least one 256-k raw stage and the
// partial tile fitting in the CTA's X ring.
int pick_splits(int64_t tiles, int T, int64_t K, int stages, bool split_operand) {
    const int64_t nr = (K + kKR - 1) / kKR;
    const double work_us = 2.0 * kBN * T * double(K) / 11.6e12 * 1e6 * (split_operand ? 2 : 1);
    const int64_t ring = int64_t(stages) * int64_t(T) * 128;
    const int64_t part = int64_t(kBN) * T * 4;
    int best = 1;
    double best_t = 1e30;
    for (int sp = 1; sp <= 8; sp *= 2) {
        if (sp > nr || (sp > 1 && part > ring)) break;
        const int64_t ctas = tiles * sp;
        const double t = double((ctas + 147) / 148) * (3.0 + work_us / sp);
        if (t < best_t * 0.97) { best_t = t; best = sp; }
    }
    return best;
}

}  // namespace

// Q6_0's high plane ([N][K/4] bytes) needs a 16-byte row pitch for its tensor map.
bool gemm_tc_supported(const GroupRef& g) {
    return g.M >= 1 && g.M <= int64_t(65535) * 256 && g.K <= (int64_t(1) << 30) &&
           (g.fmt != EMB_Q6_0 || g.K % 64 == 0) && encode_fn() != nullptr;
}

namespace {

struct GemmPlan {
    int T = 0, S = 0, P = 1, splits = 1;
    int grid_x = 0, grid_y = 0, persist = 0, streamk = 0;
    int n_tt = 0, n_items = 0;
    size_t ws_bytes = 0;  // stream-K workspace: flags, then grid_x partial-tile slots
};

// Stream-K workspace of a plan: one 32-bit flag per CTA in the first kSkFlagBytes, then one
// partial tile (P * T tokens x 128 rows, fp32) per CTA, each slot 256-byte aligned.
constexpr int kSkFlagBytes = 4096;  // room for 1024 CTAs
size_t sk_slot_bytes(int P, int T) { return size_t(roundup(int64_t(P) * T * kBN * 4, 256)); }
size_t sk_ws_bytes(int G, int P, int T) { return kSkFlagBytes + size_t(G) * sk_slot_bytes(P, T); }

// Cycle model of the plans (GB300, fitted to both formats' measured launches). A 64-k step of a
// CTA with P token tiles of T takes the largest of: the dequantisation warps' chain per A tile,
// ~620; moving its X tiles and raw codes into the SM, (128 P T + 8.7 K) bytes at the ~58 bytes
// per cycle an SM gets with all of them loading; the MMAs (2 per token of the CTA, always less
// than the loads). An item adds its drain, epilogue and restart.
double step_cycles(int P, int T) { return std::max(620.0, 2.22 * P * T + 150.0); }
double item_cycles(int P, int T) { return 6300.0 + 22.6 * P * T; }
// One launch: waves of CTAs that each take an item's share of K. A K split adds its cluster's
// exchange, ~3000 + 13 per token of the tile (four splits against none at 1000 x 1088 and 1152 x 1152, tiles of
// 96, 128, 160 and 256 tokens).
double plan_cycles(int64_t items, int P, int T, int splits, int64_t K, const Resident& at_once) {
    const int64_t nr = (K + kKR - 1) / kKR, nk = (K + kKC - 1) / kKC;
    const double steps = double(std::min(nk, (nr + splits - 1) / splits * kStepsPerRaw));
    const double exchange = splits > 1 ? 3000.0 + 13.0 * T : 0.0;
    const int64_t clusters = std::max(1, at_once.n[splits == 8 ? 3 : splits / 2]);
    const int64_t waves = (items + clusters - 1) / clusters;
    return double(waves) * (steps * step_cycles(P, T) + item_cycles(P, T) + exchange);
}

// The launch shape of one group. With streamk_ok the plan may take the stream-K schedule,
// which needs plan.ws_bytes of zero-filled workspace.
GemmPlan plan_gemm(const GroupRef& g, bool streamk_ok) {
    GemmPlan pl;
    int tiles = 0;
    for (int i = 0; i < g.n_mats; ++i) tiles += int((g.mats[i].N + kBN - 1) / kBN);
    // one token tile per CTA: balanced tiles of at most 256, rounded up to the MMA's N granule
    int64_t t_tiles = (g.M + 255) / 256;
    int T = int(roundup((g.M + t_tiles - 1) / t_tiles, 16));
    const bool split = g.K < 1024 || g.precise;
    int S = g.fmt == EMB_Q8_0   ? (split ? pick_stages<EMB_Q8_0, true>(T) : pick_stages<EMB_Q8_0, false>(T))
            : g.fmt == EMB_Q4_0 ? (split ? pick_stages<EMB_Q4_0, true>(T) : pick_stages<EMB_Q4_0, false>(T))
                                : (split ? pick_stages<EMB_Q6_0, true>(T) : pick_stages<EMB_Q6_0, false>(T));
    const Resident at_once = resident_clusters();
    const int sms = at_once.n[0];
    int splits = 1;
    double one_tile = 0.0;  // cycles of the plan with one token tile per CTA
    if (split || sms <= 0 || g.M <= 64) {
        splits = pick_splits(t_tiles * tiles, T, g.K, S, split);
        one_tile = plan_cycles(t_tiles * tiles, 1, T, splits, g.K, at_once);
    } else {
        // Token tiles and K splits together: a launch that leaves SMs idle may take smaller token
        // tiles, or a K split with its exchange, whichever the model says is at least 3 % faster than
        // what has fewer tiles. Tiles stay at 96 tokens and more: the model has their steps bound by
        // the dequantisation, equally long, but 64 measured 9 % slower (they read the weights more
        // often). Against splitting first (us): ViT M = 768 o, eight tiles of 96 for four of 192 in
        // four splits, 8.3 / 10.8; 8192 x 1024 at M = 128, one tile for two splits, 8.1 / 10.3;
        // unchanged: fc1 four tiles of 192, q/k/v five of 160, fc2 four of 192 in four splits.
        const int64_t tt0 = t_tiles, nr = (g.K + kKR - 1) / kKR;
        one_tile = 1e30;
        for (int64_t tt = tt0; tt <= tt0 + 12; ++tt) {
            const int Tc = int(roundup((g.M + tt - 1) / tt, 16));
            if (tt > tt0 && Tc < 96) break;
            const int Sc = g.fmt == EMB_Q8_0   ? pick_stages<EMB_Q8_0, false>(Tc)
                           : g.fmt == EMB_Q4_0 ? pick_stages<EMB_Q4_0, false>(Tc)
                                               : pick_stages<EMB_Q6_0, false>(Tc);
            for (int sp = 1; sp <= 8 && sp <= nr; sp *= 2) {
                if (sp > 1 && Sc < 4) break;  // the 512 T-byte partial tile lies in the X ring
                const double c = plan_cycles(tt * tiles, 1, Tc, sp, g.K, at_once);
                if (c < 0.97 * one_tile) {
                    one_tile = c;
                    t_tiles = tt;
                    T = Tc;
                    S = Sc;
                    splits = sp;
                }
            }
        }
    }
    int P = 1, grid_x = int(t_tiles);
    // Two token tiles per CTA halve the dequantisation and the code loads per token (each A tile
    // feeds the MMAs of both), for half as many CTAs: taken where the cycle model gains 5 %.
    // Llama-7B q/k/v at M = 280 (one wave of 96 CTAs instead of two of 192), Gemma-2B gate/up at
    // M = 816 (four rounds of two tiles instead of seven of one: 111 -> 104 us); narrow layers
    // keep one tile per CTA and split K instead.
    if (!split && t_tiles >= 2) {
        const int64_t t2 = 2 * ((g.M + 447) / 448);  // even count of tiles of at most 224
        const int T2 = int(roundup((g.M + t2 - 1) / t2, 16));
        const int S2 = (g.fmt == EMB_Q8_0)   ? pick_stages_pair<EMB_Q8_0>(T2)
                       : (g.fmt == EMB_Q4_0) ? pick_stages_pair<EMB_Q4_0>(T2)
                                             : pick_stages_pair<EMB_Q6_0>(T2);
        if (S2 >= 2 && T2 <= 224 && sms > 0) {
            const double c2 = plan_cycles(t2 / 2 * tiles, 2, T2, 1, g.K, at_once);
            if (c2 < 0.95 * one_tile) {
                P = 2;
                T = T2;
                S = S2;
                splits = 1;
                grid_x = int(t2 / 2);
            }
        }
    }
    // More items (weight tile x token tile) than SMs with one tile per CTA and no K split:
    // persistent CTAs, one per SM, each looping over items (barriers, TMEM and the first
    // copies' latency paid once per CTA; the next item's copies overlap this one's epilogue).
    int grid_y = tiles, persist = 0;
    {
        const int64_t items = int64_t(grid_x) * tiles;
        if (splits == 1 && sms > 0 && items > sms && items < (int64_t(1) << 30)) {
            persist = 1;
            pl.n_tt = grid_x;
            pl.n_items = int32_t(items);
            grid_x = sms;
            grid_y = 1;
        }
    }
    pl.T = T;
    pl.S = S;
    pl.P = P;
    pl.splits = splits;
    pl.grid_x = grid_x;
    pl.grid_y = grid_y;
    pl.persist = persist;
    // Stream-K: when the waves of whole items leave SMs idle (a last wave that is mostly
    // empty), cut the raw stages of all items into one equal range per SM. Both plans are
    // costed with the cycle model; stream-K adds, per
    // token of the CTA, 59 cycles for writing, publishing, staging and adding a partial tile and
    // 11.5 for every further tail a head adds (per-CTA %globaltimer stamps at 288 tokens: 147 KB
    // written in ~3 us, staged and added in ~1.7 us, a slower store pass after it). It is taken
    // where that gains 8 %. Measured with and without it, us per launch: Llama-7B gate/up at
    // M = 280 49.8 / 63.8; 24000 x 4096 at M = 130 44.2 / 61.0; 5000 x 5056 at M = 300 30.0 / 35.2;
    // not taken: Llama-7B o 22.9 / 20.2, Gemma-2B gate/up at M = 816 (every CTA ends several
    // items) 108 / 104, ViT q/k/v 19.6 / 11.1.
    if (streamk_ok && !split && g.M >= 128 && sms > 0) {
        const int64_t nr_all = (g.K + kKR - 1) / kKR;
        const double cur = plan_cycles(pl.persist ? pl.n_items : int64_t(grid_x) * grid_y, P, T, splits, g.K, at_once);
        struct Cand { int P, T, S; int64_t n_tt; };
        Cand cands[2];
        int nc = 0;
        {
            const int64_t tt1 = (g.M + 255) / 256;
            const int T1 = int(roundup((g.M + tt1 - 1) / tt1, 16));
            const int S1 = g.fmt == EMB_Q8_0   ? pick_stages<EMB_Q8_0, false>(T1)
                           : g.fmt == EMB_Q4_0 ? pick_stages<EMB_Q4_0, false>(T1)
                                               : pick_stages<EMB_Q6_0, false>(T1);
            cands[nc++] = Cand{1, T1, S1, tt1};
            const int64_t t2 = 2 * ((g.M + 447) / 448);
            const int T2 = int(roundup((g.M + t2 - 1) / t2, 16));
            const int S2 = g.fmt == EMB_Q8_0   ? pick_stages_pair<EMB_Q8_0>(T2)
                           : g.fmt == EMB_Q4_0 ? pick_stages_pair<EMB_Q4_0>(T2)
                                               : pick_stages_pair<EMB_Q6_0>(T2);
            if (S2 >= 2 && T2 <= 224) cands[nc++] = Cand{2, T2, S2, t2 / 2};
        }
        double best = cur / 1.08;
        for (int c = 0; c < nc; ++c) {
            const Cand& cd = cands[c];
            const int64_t items = cd.n_tt * tiles;
            const int64_t U = items * nr_all;
            if (items >= (int64_t(1) << 30) || U >= (int64_t(1) << 31)) continue;
            const int64_t G = std::min<int64_t>(std::min(sms, kSkFlagBytes / 4), U);
            // a head adds the tails of the CTAs whose ranges start inside its item
            const int64_t per = std::max<int64_t>(1, U / G);
            const double tails = double(std::max<int64_t>(1, (nr_all + per - 1) / per));
            const double ends = std::max(1.0, double(per) / double(nr_all));  // items a CTA ends
            const double t = double((U + G - 1) / G) * kStepsPerRaw * step_cycles(cd.P, cd.T) +
                             ends * item_cycles(cd.P, cd.T) + cd.P * cd.T * (59.0 + 11.5 * (tails - 1.0));
            if (t < best) {
                best = t;
                pl.T = cd.T;
                pl.S = cd.S;
                pl.P = cd.P;
                pl.splits = 1;
                pl.persist = 1;
                pl.streamk = 1;
                pl.n_tt = int(cd.n_tt);
                pl.n_items = int(items);
                pl.grid_x = int(G);
                pl.grid_y = 1;
                pl.ws_bytes = sk_ws_bytes(int(G), cd.P, cd.T);
            }
        }
    }
    return pl;
}

cudaError_t launch_plan(const GroupRef& g, const GemmPlan& pl, bool pdl, int* status, cudaStream_t s) {
    GemmParams p;
    memset(&p, 0, sizeof(p));
    const int T = pl.T, S = pl.S, P = pl.P, splits = pl.splits, grid_x = pl.grid_x, grid_y = pl.grid_y;
    const bool split = g.K < 1024 || g.precise;
    p.persist = pl.persist;
    p.streamk = pl.streamk;
    p.n_tt = pl.n_tt;
    p.n_items = pl.n_items;
    if (pl.streamk) {
        p.slot_floats = int32_t(sk_slot_bytes(P, T) / 4);
        p.ws_flag = static_cast<uint32_t*>(g.ws);
        p.ws_part = reinterpret_cast<float*>(static_cast<uint8_t*>(g.ws) + kSkFlagBytes);
    }
    int tiles = 0;
    if (!encode_2d(&p.x_map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, g.X, uint64_t(g.K), uint64_t(g.M),
                   uint64_t(g.K) * 2, kKC, uint32_t(T), CU_TENSOR_MAP_SWIZZLE_128B,
                   CU_TENSOR_MAP_L2_PROMOTION_L2_128B))
        return cudaErrorInvalidValue;
    tiles = 0;
    for (int i = 0; i < g.n_mats; ++i) {
        const MatRef& mr = g.mats[i];
        const uint64_t row_bytes = g.fmt == EMB_Q8_0 ? uint64_t(g.K) : uint64_t(g.K) / 2;
        if (!encode_2d(&p.codes_map[i], CU_TENSOR_MAP_DATA_TYPE_UINT8, mr.codes, row_bytes,
                       uint64_t(mr.N), row_bytes, 128, kBN, CU_TENSOR_MAP_SWIZZLE_128B,
                       CU_TENSOR_MAP_L2_PROMOTION_L2_256B))
            return cudaErrorInvalidValue;
        if (!encode_2d(&p.scales_map[i], CU_TENSOR_MAP_DATA_TYPE_UINT16, mr.scales,
                       uint64_t(g.ldS), uint64_t(mr.N), uint64_t(g.ldS) * 2, 8, kBN,
                       CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B))
            return cudaErrorInvalidValue;
        if (g.fmt == EMB_Q6_0 &&
            !encode_2d(&p.high_map[i], CU_TENSOR_MAP_DATA_TYPE_UINT8, mr.high, uint64_t(g.K) / 4,
                       uint64_t(mr.N), uint64_t(g.K) / 4, 64, kBN, CU_TENSOR_MAP_SWIZZLE_NONE,
                       CU_TENSOR_MAP_L2_PROMOTION_L2_256B))
            return cudaErrorInvalidValue;
        p.Y[i] = mr.Y;
        p.N[i] = int32_t(mr.N);
        p.tile0[i] = tiles;
        tiles += int((mr.N + kBN - 1) / kBN);
    }
    p.tile0[g.n_mats] = tiles;
    p.n_mats = g.n_mats;
    p.M = int32_t(g.M);
    p.K = int32_t(g.K);
    p.X = g.X;
    p.T = T;
    p.P = P;
    p.stages = S;
    p.a_stages = a_stages_of(split, T, P);
    p.splits = splits;
    p.epi = g.epi;
    p.tmem_cols = kTmemCols;
    p.status = status;
    p.wait_first = pdl ? 0 : 1;
    if (pl.streamk) {
        if (g.fmt == EMB_Q8_0)
            return P == 2 ? launch_kernel<EMB_Q8_0, false, 2, true>(p, grid_x, grid_y, s)
                          : launch_kernel<EMB_Q8_0, false, 1, true>(p, grid_x, grid_y, s);
        if (g.fmt == EMB_Q4_0)
            return P == 2 ? launch_kernel<EMB_Q4_0, false, 2, true>(p, grid_x, grid_y, s)
                          : launch_kernel<EMB_Q4_0, false, 1, true>(p, grid_x, grid_y, s);
        return P == 2 ? launch_kernel<EMB_Q6_0, false, 2, true>(p, grid_x, grid_y, s)
                      : launch_kernel<EMB_Q6_0, false, 1, true>(p, grid_x, grid_y, s);
    }
    if (g.fmt == EMB_Q8_0)
        return split    ? launch_kernel<EMB_Q8_0, true, 1>(p, grid_x, grid_y, s)
               : P == 2 ? launch_kernel<EMB_Q8_0, false, 2>(p, grid_x, grid_y, s)
                        : launch_kernel<EMB_Q8_0, false, 1>(p, grid_x, grid_y, s);
    if (g.fmt == EMB_Q4_0)
        return split    ? launch_kernel<EMB_Q4_0, true, 1>(p, grid_x, grid_y, s)
               : P == 2 ? launch_kernel<EMB_Q4_0, false, 2>(p, grid_x, grid_y, s)
                        : launch_kernel<EMB_Q4_0, false, 1>(p, grid_x, grid_y, s);
    return split    ? launch_kernel<EMB_Q6_0, true, 1>(p, grid_x, grid_y, s)
           : P == 2 ? launch_kernel<EMB_Q6_0, false, 2>(p, grid_x, grid_y, s)
                    : launch_kernel<EMB_Q6_0, false, 1>(p, grid_x, grid_y, s);
}

}  // namespace

// Waves of clusters, each with its fill, its 64-k steps and, with a K split, the cluster's exchange, the
// drain of its tokens, and the codes' way from HBM. Fitted to 3060 launches of 17 to 64 tokens (rms 7 %).
double gemm_tc_chunk_us(const GroupRef& g) {
    const GemmPlan pl = plan_gemm(g, false);
    const Resident at_once = resident_clusters();
    int64_t rows = 0, tiles = 0;
    for (int i = 0; i < g.n_mats; ++i) {
        rows += g.mats[i].N;
        tiles += (g.mats[i].N + kBN - 1) / kBN;
    }
    const int64_t nr = (g.K + kKR - 1) / kKR, nk = (g.K + kKC - 1) / kKC;
    const double clusters = std::max(1, at_once.n[pl.splits == 8 ? 3 : pl.splits / 2]);
    const double waves = pl.splits > 1 ? std::ceil(double(tiles) / clusters) : std::max(1.0, double(tiles) / clusters);
    const double steps = double(std::min(nk, (nr + pl.splits - 1) / pl.splits * kStepsPerRaw));
    return -1.0 + waves * (1.52 + 0.28 * steps + (pl.splits > 1 ? 2.19 : 0.0) + 1.49 * pl.T / 64.0) +
           1.87e-7 * double(rows) * double(g.K);
}

size_t gemm_tc_workspace(const GroupRef& g) {
    if (!gemm_tc_supported(g)) return 0;
    return plan_gemm(g, true).ws_bytes;
}

// The stream-K schedule runs only with a caller workspace large enough for it (its size
// is what gemm_tc_workspace reports); without one the group takes the plan without it.
cudaError_t launch_gemm_tc(const GroupRef& g, bool pdl, int* status, cudaStream_t s) {
    GemmPlan pl = plan_gemm(g, g.ws != nullptr);
    if (pl.streamk && g.ws_bytes < pl.ws_bytes) pl = plan_gemm(g, false);
    return launch_plan(g, pl, pdl, status, s);
}

}  // namespace emb
