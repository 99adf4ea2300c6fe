// K2 for head_dim 128: the software-pipelined backward (see peagle_bwd.cu for the formulation and
// for the head_dim-64 kernel this one mirrors).  What differs at 128 elements per head:
//   - Tensor memory is full with S^T | dP^T | dK | dV (128 columns each), so K and V stay in shared
//     memory as the A operands of S^T and dP^T, and dQ = dS K is accumulated over the dP^T columns
//     once the compute warps hold dP^T in registers; dP^T of the next step follows when the drain
//     warps have read dQ out.
//   - Shared memory is full with K, V (one stage), the dS^T tile, two stages of Q, ONE stage of dO
//     (its last reader of a step, dV, runs early in the step and its first reader of the next
//     step, dP^T, late, so the reload fits between them) and two fp32 panels of 16 KB through which
//     dQ, dK and dV leave by tiled reduce-adds.  The fp32 reductions are what bounds the kernel: with
//     the dQ reduce-adds left out it takes 0.57 instead of 0.71 ms (16,384 tokens, 32 heads), so the
//     two panels alternate (one tile at a time, 64 columns of all warps together: 0.79 ms).  -LSE*log2e and -Delta of a step's rows (1 KB) come in with its Q tile; that
//     they fit at all takes the 1 KB usually kept as slack for aligning the tiles, so the kernel
//     requires a 1024-byte aligned base and reports an error otherwise.  Read from global memory
//     (broadcast loads, other rows every step) they cost 16 % of the kernel.  The packed metadata
//     of the rows, needed by the steps that are not FULL, is still read from global memory.
// Roles (512 threads): warps 0-7 compute (warp w key lanes 32 (w % 4) .. and half of the 128
// query columns), warp 8 issues S^T and dV (dV(i), S^T(i+1) while the compute warps form dS^T(i)), warp 10
// dQ, dK and dP^T (dQ(i), dK(i), then dP^T(i+1) while they form P^T(i+1)), warp 9 produces (TMA),
// warps 12-15 drain dQ per step and dK / dV per work item.
#include <math_constants.h>

#include "peagle_bwd_common.cuh"

namespace peagle {
using namespace sm100;

// Registers per thread after the roles re-split the CTA's allocation (512 threads x 128): two
// warpgroups of compute warps, the warpgroup of the issuing / producing warps, the drain warpgroup.
// The thread that issues the products wants its descriptors resident: with 56 (head_dim 128: 40)
// registers for its warpgroup the compiler spilled them and re-formed them per product, and the
// kernel was 9 (7) per cent slower than with 88.
#ifndef BWD128_COMPUTE_REGS
#define BWD128_COMPUTE_REGS 144
#define BWD128_ISSUE_REGS 88
#define BWD128_DRAIN_REGS 136
#endif
namespace {
constexpr int COMPUTE_REGS = BWD128_COMPUTE_REGS, ISSUE_REGS = BWD128_ISSUE_REGS, DRAIN_REGS = BWD128_DRAIN_REGS;
static_assert(256 * COMPUTE_REGS + 128 * ISSUE_REGS + 128 * DRAIN_REGS <= 512 * 128,
              "the re-split must fit the launch allocation, or setmaxnreg.inc waits for ever");
} // namespace

struct Bwd128Cfg {
    static constexpr int D = 128;
    static constexpr int NSQ = 2;
    static constexpr int PANEL_BYTES = 128 * 128;        // 128 rows x 64 bf16
    static constexpr int TILE_BYTES = 2 * PANEL_BYTES;   // 128 rows x 128 bf16, two panels
    static constexpr int OFF_K = 0;
    static constexpr int OFF_V = TILE_BYTES;
    static constexpr int OFF_DS = 2 * TILE_BYTES;                // [key][q 0..63], [key][q 64..127]
    static constexpr int OFF_Q = OFF_DS + TILE_BYTES;            // two stages of Q
    static constexpr int OFF_DO = OFF_Q + NSQ * TILE_BYTES;      // one stage of dO
    static constexpr int OFF_DQ = OFF_DO + TILE_BYTES;           // fp32 dQ half tile on its way out: 2 panels of 32 columns
    static constexpr int OFF_BAR = OFF_DQ + TILE_BYTES;
    static constexpr int N_BAR = 2 * NSQ + 14 + 4;               // the last four: work-queue slots
    static constexpr int OFF_MISC = OFF_BAR + N_BAR * 8;         // tensor-memory base, abort flag
    static constexpr int OFF_WQ = (OFF_MISC + 8 + 15) / 16 * 16; // work queue
    // per stage of Q: -LSE*log2e and -Delta of the step's 128 query rows (2 x 512 bytes)
    static constexpr int OFF_ROW = OFF_WQ + BWD_QUEUE_BYTES;
    static constexpr int ROW_BYTES = 1024;
    // No slack for alignment is left: the kernel declares its shared memory 1024-byte aligned and
    // leaves with an error if the base is not.
    static constexpr int SMEM_BYTES = OFF_ROW + NSQ * ROW_BYTES;
    static_assert(SMEM_BYTES <= 227 * 1024, "shared memory of one CTA");
    static constexpr int TM_S = 0, TM_DP = 128, TM_DQ = 128, TM_DK = 256, TM_DV = 384;
};

__global__ void __launch_bounds__(512, 1)
bwd128_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmdO,
              const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmV,
              const __grid_constant__ CUtensorMap tmDQ, const __grid_constant__ CUtensorMap tmDK,
             const __grid_constant__ CUtensorMap tmDV, const BwdParams P)
{
    using C = Bwd128Cfg;
    constexpr int D = 128, NSQ = C::NSQ, TB = C::TILE_BYTES, PB = C::PANEL_BYTES;
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    const uint32_t sb = smem_u32(smem_raw);
    uint8_t *sp = smem_raw;
    if (sb & 1023u) { // the swizzled tiles need this alignment; nothing has been set up yet
        pdl_wait();
        if (threadIdx.x == 0)
            atomicCAS(P.status, 0, PEAGLE_ERR_ALIGN);
        return;
    }
    const uint32_t bar0 = sb + C::OFF_BAR;
    auto BAR = [&](int i) { return bar0 + 8u * (uint32_t)i; };
    constexpr int B_QFULL = 0, B_QEMPTY = NSQ, B_KFULL = 2 * NSQ, B_KEMPTY = B_KFULL + 1,
                  B_SFULL = B_KFULL + 2, B_DPFULL = B_KFULL + 3, B_PFULL = B_KFULL + 4,
                  B_DSFULL = B_KFULL + 5, B_DQFULL = B_KFULL + 6, B_DQEMPTY = B_KFULL + 7,
                  B_ACCFREE = B_KFULL + 8, B_DOFULL = B_KFULL + 9, B_DOEMPTY = B_KFULL + 10,
                  B_ITEMDONE = B_KFULL + 11, B_VFULL = B_KFULL + 12, B_VEMPTY = B_KFULL + 13,
                  B_WQ = B_KFULL + 14;
    volatile uint32_t *tmem_slot = reinterpret_cast<volatile uint32_t *>(sp + C::OFF_MISC);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(sp + C::OFF_MISC + 4);
    uint8_t *wq = sp + C::OFF_WQ;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    if (threadIdx.x == 0) {
        *abort_flag = 0;
        for (int s = 0; s < NSQ; ++s) {
            mbar_init(BAR(B_QFULL + s), 1);
            mbar_init(BAR(B_QEMPTY + s), 1);
        }
        for (int s = 0; s < 4; ++s)
            mbar_init(BAR(B_WQ + s), 1);
        mbar_init(BAR(B_KFULL), 1);
        mbar_init(BAR(B_KEMPTY), 1);
        mbar_init(BAR(B_VFULL), 1);
        mbar_init(BAR(B_VEMPTY), 1);
        mbar_init(BAR(B_SFULL), 1);
        mbar_init(BAR(B_DPFULL), 1);
        mbar_init(BAR(B_PFULL), 8);   // one arrival per compute warp
        mbar_init(BAR(B_DSFULL), 8);
        mbar_init(BAR(B_DQFULL), 1);
        mbar_init(BAR(B_DQEMPTY), 4); // one arrival per drain warp
        mbar_init(BAR(B_ACCFREE), 4);
        mbar_init(BAR(B_DOFULL), 1);
        mbar_init(BAR(B_DOEMPTY), 2);  // dV and dP^T have read the tile
        mbar_init(BAR(B_ITEMDONE), 2); // dV and dK are complete
        fence_mbar_init();
    }
    if (warp == 8) {
        tmem_alloc(sb + C::OFF_MISC, 512);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    pdl_wait();
    pdl_trigger();

    if (warp >= 12) {
        // ------------------------------------------------------------ drain (warps 12-15)
        reg_set<DRAIN_REGS, 128>();
        const uint32_t lane_base = (uint32_t)((warp & 3) * 32) << 16;
        // A panel (this warp's 32 lanes, 32 columns) on its way out: registers -> swizzled fp32 tile
        // in shared memory -> tiled reduce-add.  Whole 128-byte row pieces reach L2 together, which
        // the L2 takes about 1.6 times faster than the same bytes as scattered 32-byte pieces.  The
        // panels take two places in turn: while the reduce-add of one reads shared memory the next is
        // written (a place is free once all but the warp's latest reduce-add have read theirs), and
        // no warp waits for another.
        auto send = [&](const uint32_t (&o)[32], float f, int slot, const CUtensorMap *map, int x, int y, int z) {
            if (lane == 0)
                bulk_wait_group_read<1>();
            __syncwarp();
            uint8_t *dst = sp + C::OFF_DQ + slot * PB + ((warp & 3) * 32 + lane) * 128;
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                float4 v;
                v.x = __uint_as_float(o[4 * c]) * f;
                v.y = __uint_as_float(o[4 * c + 1]) * f;
                v.z = __uint_as_float(o[4 * c + 2]) * f;
                v.w = __uint_as_float(o[4 * c + 3]) * f;
                *reinterpret_cast<float4 *>(dst + ((c ^ (lane & 7)) << 4)) = v;
            }
            fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) {
                tma_reduce_add_3d(map, sb + C::OFF_DQ + slot * PB + (warp & 3) * 4096, x, y, z + (warp & 3) * 32);
                bulk_commit_group();
            }
        };
        bool ok = true;
        int it = 0;
        BwdItem item;
        for (int w = 0; ok && bwd_take(wq, BAR(B_WQ), w, abort_flag, item); ++w) {
        unsigned em = item.mask & 0xffu;
        for (int i = 0, hh = 0; i < item.steps; ++i, ++it) {
            const int row0 = (item.qt0 + __ffs(em) - 1) * BM; // row of the partition
            const int h = item.h0 + hh;
            if (++hh == item.nh) {
                hh = 0;
                em &= em - 1;
            }
            ok = __all_sync(0xffffffffu, mbar_wait(BAR(B_DQFULL), it & 1, abort_flag));
            if (!ok)
                break;
            tc_fence_after();
            // dQ(it) (rows past the partition's end are clipped by the tensor map)
            uint32_t o[4][32];
#pragma unroll
            for (int pn = 0; pn < 4; ++pn)
                tmem_ld32(tmem + lane_base + C::TM_DQ + pn * 32, o[pn]);
            tmem_wait_ld();
            tc_fence_before();
            warp_arrive(BAR(B_DQEMPTY));
#pragma unroll
            for (int pn = 0; pn < 4; ++pn)
                send(o[pn], P.scale, pn & 1, &tmDQ, 32 * pn, h, row0);
        }
        if (!ok)
            break;
        // dK and dV of the work item
        ok = __all_sync(0xffffffffu, mbar_wait(BAR(B_ITEMDONE), w & 1, abort_flag));
        if (!ok)
            break;
        tc_fence_after();
        // Keys past a ragged tile's end are another range's, often another sequence's.  Their sums have weight
        // zero throughout, but a zero times an Inf or NaN of a row of Q or dO is not zero, so zeros are
        // what they get.  (The item is read again: carried through its steps these words would be
        // spilled; see the queue for why the slot still holds it.  A warp none of whose rows are the tile's
        // sends its zeros too: a branch around it costs 44 bytes of spills and 2 of 76 us at 391 positions,
        // 32 heads.)
        const BwdItem &done = *reinterpret_cast<const BwdItem *>(wq + (w & 3) * sizeof(BwdItem));
        const int k_start = done.k_start, g = done.g;
        const int rows = done.k_len - (warp & 3) * 32; // of this warp's 32 keys, how many are the tile's
#pragma unroll
        for (int pn = 0; pn < 8; ++pn) {
            uint32_t o[32];
            tmem_ld32(tmem + lane_base + C::TM_DK + pn * 32, o); // dK, then dV
            tmem_wait_ld();
            if (pn == 7) {
                tc_fence_before();
                warp_arrive(BAR(B_ACCFREE));
            }
            if (lane >= rows) {
#pragma unroll
                for (int i = 0; i < 32; ++i)
                    o[i] = 0;
            }
            const bool k = pn < 4;
            send(o, k ? P.scale : 1.f, pn & 1, k ? &tmDK : &tmDV, 32 * (pn % 4), g, k_start);
        }
        }
        if (lane == 0)
            bulk_wait_group<0>();
    } else if (warp >= 8) {
        reg_set<ISSUE_REGS, 128>();
        if (warp == 9) {
            // -------------------------------------------------------- producer
            if (lane == 0) {
                tma_prefetch_desc(&tmQ);
                tma_prefetch_desc(&tmdO);
                tma_prefetch_desc(&tmK);
                tma_prefetch_desc(&tmV);
            }
            const BwdSplit split = bwd_split(P);
            BwdItem item, nxt;
            int it = 0;
            bool more = bwd_draw(P, split, wq, BAR(B_WQ), 0, lane, item), ok = true;
            // waits for a place to be free, then loads a tile of two panels into it
            auto load = [&](int empty, uint32_t parity, int full, uint32_t extra, uint32_t dst, const CUtensorMap *map,
                            int y, int z) -> bool {
                if (!__all_sync(0xffffffffu, mbar_wait(BAR(empty), parity, abort_flag)))
                    return false;
                if (lane == 0) {
                    mbar_arrive_expect_tx(BAR(full), TB + extra);
                    for (int pn = 0; pn < 2; ++pn)
                        tma_load_3d(dst + pn * PB, map, BAR(full), pn * 64, y, z);
                }
                return true;
            };
            for (int w = 0; ok && more; ++w) {
                unsigned em = item.mask & 0xffu;
                for (int i = 0, hh = 0; i < item.steps; ++i, ++it) {
                    const int st = it % NSQ, ph = (it / NSQ) & 1;
                    const int qt = item.qt0 + __ffs(em) - 1, h = item.h0 + hh;
                    const int row0 = P.q_begin + qt * BM;
                    if (++hh == item.nh) {
                        hh = 0;
                        em &= em - 1;
                    }
                    // In the order in which the places become free: Q (two stages) after dK of the step
                    // before the last, V and dO (one stage) after dP^T and dV, K (one stage) after dQ of
                    // the last step.
                    ok = load(B_QEMPTY + st, ph ^ 1, B_QFULL + st, C::ROW_BYTES, sb + C::OFF_Q + st * TB, &tmQ, h, row0);
                    if (!ok)
                        break;
                    if (lane == 0) {
                        const uint32_t ra = sb + C::OFF_ROW + st * C::ROW_BYTES;
                        const size_t ri = (size_t)h * P.q_pad + (size_t)qt * BM;
                        bulk_load(ra, P.nl2 + ri, 512, BAR(B_QFULL + st));
                        bulk_load(ra + 512, P.nd + ri, 512, BAR(B_QFULL + st));
                    }
                    ok = (i > 0 || load(B_VEMPTY, (w & 1) ^ 1, B_VFULL, 0, sb + C::OFF_V, &tmV, item.g, item.k_start)) &&
                         load(B_DOEMPTY, (it & 1) ^ 1, B_DOFULL, 0, sb + C::OFF_DO, &tmdO, h, row0) &&
                         (i > 0 || load(B_KEMPTY, (w & 1) ^ 1, B_KFULL, 0, sb + C::OFF_K, &tmK, item.g, item.k_start));
                    if (!ok)
                        break;
                    if (i + 1 == item.steps)
                        more = bwd_draw(P, split, wq, BAR(B_WQ), w + 1, lane, nxt);
                }
                item = nxt;
            }
        } else if (warp == 8 || warp == 10) {
            // -------------------------------------------------------- MMA issue: two warps, each with
            // its own accumulators (products into one accumulator keep one thread's order): warp 8
            // S^T and dV, warp 10 dQ, dK and dP^T.  The whole warp walks the steps and waits, its
            // elected lane issues (see elect_one).
            const uint32_t lead = elect_one();
            constexpr uint32_t IDESC_S = idesc_bf16_f32(128, 128, 0, 0);
            constexpr uint32_t IDESC_KV = idesc_bf16_f32(128, D, 0, 1);
            constexpr uint32_t IDESC_DQ = idesc_bf16_f32(128, D, 1, 1);
            // Lower descriptor words (16-byte units).  "k" = K-major operand, "m" = MN-major
            // (its second 64-wide panel one PANEL_BYTES further on).
            const uint32_t k_k = desc_lo_sw128(sb + C::OFF_K, 16), k_m = desc_lo_sw128(sb + C::OFF_K, PB);
            const uint32_t v_k = desc_lo_sw128(sb + C::OFF_V, 16);
            const uint32_t ds_k = desc_lo_sw128(sb + C::OFF_DS, 16), ds_m = desc_lo_sw128(sb + C::OFF_DS, PB);
            const uint32_t q_k = desc_lo_sw128(sb + C::OFF_Q, 16), q_m = desc_lo_sw128(sb + C::OFF_Q, PB);
            const uint32_t do_k = desc_lo_sw128(sb + C::OFF_DO, 16), do_m = desc_lo_sw128(sb + C::OFF_DO, PB);
            constexpr uint32_t TBU = TB >> 4, PBU = PB >> 4;
            // slice k of a K-major operand: panel k / 4, 32 bytes per slice inside the 128-byte rows
            auto koff = [](int k) { return (uint32_t)((k / 4) * PBU + (k % 4) * 2); };
            auto issue_s = [&](uint32_t q) { // S^T = K Q^T
#pragma unroll
                for (int k = 0; k < D / 16; ++k)
                    if (lead) mma_ss_lo(tmem + C::TM_S, k_k + koff(k), q_k + q + koff(k), IDESC_S, k > 0);
                if (lead) tc_commit(BAR(B_SFULL));
            };
            auto issue_dp = [&]() { // dP^T = V dO^T
#pragma unroll
                for (int k = 0; k < D / 16; ++k)
                    if (lead) mma_ss_lo(tmem + C::TM_DP, v_k + koff(k), do_k + koff(k), IDESC_S, k > 0);
                if (lead) tc_commit(BAR(B_DPFULL));
                if (lead) tc_commit(BAR(B_DOEMPTY));
            };
            static_assert(NSQ == 2, "stage = step parity");
            bool ok = true;
            int it = 0;
            BwdItem item, nxt;
            bool have = bwd_take(wq, BAR(B_WQ), 0, abort_flag, item);
            // The steps of consecutive items follow one another like the steps of one item: the next
            // item's first S^T / dP^T is issued behind the last dV / dK of this one.
            if (warp == 8) {
                auto next_s = [&](int j, int w, bool first) { // S^T of step j, the first of item w or not
                    if ((first && !mbar_wait(BAR(B_KFULL), w & 1, abort_flag)) ||
                        !mbar_wait(BAR(B_QFULL + (j & 1)), (j >> 1) & 1, abort_flag))
                        return false;
                    tc_fence_after();
                    issue_s((j & 1) * TBU);
                    return true;
                };
                if (have)
                    ok = next_s(0, 0, true);
                for (int w = 0; ok && have; ++w) {
                    bool have_n = false;
                    for (int i = 0; i < item.steps; ++i, ++it) {
                        // ---- dV(it) once P^T(it) is in tensor memory (and dO in shared memory), then
                        // S^T(it+1)
                        ok = mbar_wait(BAR(B_PFULL), it & 1, abort_flag) && mbar_wait(BAR(B_DOFULL), it & 1, abort_flag);
                        if (ok && i == 0)
                            ok = mbar_wait(BAR(B_ACCFREE), (w & 1) ^ 1, abort_flag);
                        if (!ok)
                            break;
                        tc_fence_after();
#pragma unroll
                        for (int k = 0; k < 8; ++k) // query rows 16k..16k+15 of P^T (bf16 over S^T)
                            if (lead) mma_ts_lo(tmem + C::TM_DV, tmem + C::TM_S + (k / 4) * 64 + (k % 4) * 8,
                                      do_m + k * 128, IDESC_KV, i > 0 || k > 0);
                        if (lead) tc_commit(BAR(B_DOEMPTY));
                        const bool last = i + 1 == item.steps;
                        if (last) {
                            if (lead) tc_commit(BAR(B_ITEMDONE));
                            have_n = bwd_take(wq, BAR(B_WQ), w + 1, abort_flag, nxt);
                        }
                        if (!last || have_n)
                            ok = next_s(it + 1, w + 1, last);
                        if (!ok)
                            break;
                    }
                    item = nxt;
                    have = have_n;
                }
            } else {
                auto next_dp = [&](int j, int w, bool first) { // dP^T of step j, over the columns dQ(j-1) has left
                    if ((first && !mbar_wait(BAR(B_VFULL), w & 1, abort_flag)) ||
                        (j > 0 && !mbar_wait(BAR(B_DQEMPTY), (j - 1) & 1, abort_flag)) ||
                        !mbar_wait(BAR(B_DOFULL), j & 1, abort_flag))
                        return false;
                    tc_fence_after();
                    issue_dp();
                    return true;
                };
                if (have) {
                    ok = next_dp(0, 0, true);
                    if (item.steps == 1)
                        if (lead) tc_commit(BAR(B_VEMPTY));
                }
                for (int w = 0; ok && have; ++w) {
                    bool have_n = false;
                    for (int i = 0; i < item.steps; ++i, ++it) {
                        // ---- dQ(it), dK(it) once dS^T(it) is in shared memory (the compute warps then
                        // hold dP^T(it) in registers: dQ goes over its columns).  dQ first: dP^T(it+1)
                        // waits for the drain to read it out, dK runs meanwhile.
                        const bool last = i + 1 == item.steps;
                        ok = mbar_wait(BAR(B_DSFULL), it & 1, abort_flag);
                        if (ok && i == 0)
                            ok = mbar_wait(BAR(B_ACCFREE), (w & 1) ^ 1, abort_flag);
                        if (!ok)
                            break;
                        tc_fence_after();
#pragma unroll
                        for (int k = 0; k < 8; ++k)
                            if (lead) mma_ss_lo(tmem + C::TM_DQ, ds_m + k * 128, k_m + k * 128, IDESC_DQ, k > 0);
                        if (lead) tc_commit(BAR(B_DQFULL));
                        if (last)
                            if (lead) tc_commit(BAR(B_KEMPTY));
#pragma unroll
                        for (int k = 0; k < 8; ++k)
                            if (lead) mma_ss_lo(tmem + C::TM_DK, ds_k + koff(k), q_m + (it & 1) * TBU + k * 128, IDESC_KV,
                                      i > 0 || k > 0);
                        if (lead) tc_commit(BAR(B_QEMPTY + (it & 1)));
                        if (last) {
                            if (lead) tc_commit(BAR(B_ITEMDONE));
                            have_n = bwd_take(wq, BAR(B_WQ), w + 1, abort_flag, nxt);
                        }
                        if (!last || have_n) {
                            ok = next_dp(it + 1, w + 1, last);
                            // the item's last dP^T: V may be replaced behind it
                            if (last ? nxt.steps == 1 : i + 2 == item.steps)
                                if (lead) tc_commit(BAR(B_VEMPTY));
                        }
                        if (!ok)
                            break;
                    }
                    item = nxt;
                    have = have_n;
                }
            }
        }
    } else {
        reg_set<COMPUTE_REGS, 128>();
        // ------------------------------------------------------------ compute (warps 0-7)
        const int wg = warp >> 2;        // half of the query columns
        const uint32_t lane_sel = (uint32_t)((warp & 3) * 32) << 16;
        const uint32_t tS = tmem + lane_sel + C::TM_S + wg * 64;
        const uint32_t tDP = tmem + lane_sel + C::TM_DP + wg * 64;
        // row of the dS^T tile that this lane addresses in stmatrix_x4 (see there): its row of the
        // first 16, chunk added per store
        const uint32_t dsrow = sb + C::OFF_DS + wg * PB + ((warp & 3) * 32 + (lane & 15)) * 128;
        bool ok = true;
        int it = 0;
        BwdItem item;
        for (int w = 0; ok && bwd_take(wq, BAR(B_WQ), w, abort_flag, item); ++w) {
            int32_t mk[4]; // metadata of the keys of this thread's four lanes
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int kl = (warp & 3) * 32 + 8 * i + (lane >> 2);
                mk[i] = (kl < item.k_len) ? P.meta[item.k_start + kl] : META_NONE_K;
            }
            for (unsigned em = item.mask & 0xffu; ok && em; em &= em - 1) {
            const int qt = item.qt0 + __ffs(em) - 1;
            const bool full = (item.mask >> (7 + __ffs(em))) & 1u;
            for (int hh = 0; hh < item.nh; ++hh, ++it) {
            // per-row values of this step's 64 query columns
            const size_t rb = (size_t)qt * BM + wg * 64;
            const uint8_t *rowv = sp + C::OFF_ROW + (it % NSQ) * C::ROW_BYTES + wg * 256;
            const float4 *nl4 = reinterpret_cast<const float4 *>(rowv) + (lane & 3);
            const float4 *nd4 = reinterpret_cast<const float4 *>(rowv + 512) + (lane & 3);
            const int4 *mq4 = reinterpret_cast<const int4 *>(P.mqp + rb) + (lane & 3);
            // ---- P^T (the row values arrive with the step's Q tile).  A thread holds 4 key lanes x
            // 16 query columns, as in bwd64_kernel.
            // The row values came with the step's Q tile, which the products read: complete.
            ok = __all_sync(0xffffffffu, mbar_wait(BAR(B_SFULL), it & 1, abort_flag));
            if (!ok)
                break;
            tc_fence_after();
            float4 rv[4]; // row values of the thread's columns
#pragma unroll
            for (int m = 0; m < 4; ++m)
                rv[m] = nl4[4 * m];
            uint32_t sr[2][32];
            tmem_ld_16x256b_x8(tS, sr[0]);
            tmem_ld_16x256b_x8(tS + (16u << 16), sr[1]);
            tmem_wait_ld();
            float p[2][32];
#pragma unroll
            for (int m = 0; m < 4; ++m)
#pragma unroll
                for (int hf = 0; hf < 2; ++hf)
#pragma unroll
                    for (int e = 0; e < 8; e += 2) { // group 2m (e < 4) or 2m + 1, lane t/4 or t/4 + 8
                        const int c = 8 * m + e;
                        float a0, a1;
                        fma2(a0, a1, __uint_as_float(sr[hf][c]), __uint_as_float(sr[hf][c + 1]), P.scale_log2,
                             P.scale_log2, e < 4 ? rv[m].x : rv[m].z, e < 4 ? rv[m].y : rv[m].w);
                        p[hf][c] = fast_exp2(a0);
                        p[hf][c + 1] = fast_exp2(a1);
                    }
            if (!full) {
                // Where each of the warp's keys is a depth-0 token that all of its rows follow, nothing is
                // masked: so for six of the sixteen 32 x 32 blocks of a diagonal tile.
                int4 mq[4];
#pragma unroll
                for (int m = 0; m < 4; ++m)
                    mq[m] = __ldg(mq4 + 4 * m);
                int first = mq[0].x;
#pragma unroll
                for (int m = 0; m < 4; ++m)
                    first = min(min(first, min(mq[m].x, mq[m].y)), min(mq[m].z, mq[m].w));
                const int last = max(max(mk[0], mk[1]), max(mk[2], mk[3]));
                if (!__all_sync(0xffffffffu, last <= first && ((mk[0] | mk[1] | mk[2] | mk[3]) & 0xff) == 0)) {
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const uint32_t span = allowed_span(mk[k]);
#pragma unroll
                        for (int m = 0; m < 4; ++m)
#pragma unroll
                            for (int e = 0; e < 4; ++e) { // column 16m + 8 (e / 2) + 2 (lane % 4) + e % 2
                                const int row = e < 2 ? (e == 0 ? mq[m].x : mq[m].y) : (e == 2 ? mq[m].z : mq[m].w);
                                if ((uint32_t)(row - mk[k]) > span)
                                    p[k >> 1][8 * m + 4 * (e >> 1) + 2 * (k & 1) + (e & 1)] = 0.f;
                            }
                    }
                }
            }
#pragma unroll
            for (int hf = 0; hf < 2; ++hf) {
                uint32_t pk[16];
#pragma unroll
                for (int i = 0; i < 16; ++i)
                    pk[i] = pack_bf16x2(p[hf][2 * i], p[hf][2 * i + 1]);
                // packed P^T over the first half of this group's S^T columns
                tmem_st_16x128b_x8(tS + ((16u * hf) << 16), pk);
            }
            tmem_wait_st();
            tc_fence_before();
            warp_arrive(BAR(B_PFULL));
            // ---- dS^T
#pragma unroll
            for (int m = 0; m < 4; ++m)
                rv[m] = nd4[4 * m];
            // (and dQ and dK of the previous step have run: their warp issues dP^T behind them, so
            // the dS^T tile is free)
            ok = __all_sync(0xffffffffu, mbar_wait(BAR(B_DPFULL), it & 1, abort_flag));
            if (!ok)
                break;
            tc_fence_after();
            tmem_ld_16x256b_x8(tDP, sr[0]);
            tmem_ld_16x256b_x8(tDP + (16u << 16), sr[1]);
            tmem_wait_ld();
            tc_fence_before();
            uint32_t ds[2][16];
#pragma unroll
            for (int m = 0; m < 4; ++m)
#pragma unroll
                for (int hf = 0; hf < 2; ++hf)
#pragma unroll
                    for (int e = 0; e < 8; e += 2) {
                        const int c = 8 * m + e;
                        float t0, t1;
                        add2(t0, t1, __uint_as_float(sr[hf][c]), __uint_as_float(sr[hf][c + 1]),
                             e < 4 ? rv[m].x : rv[m].z, e < 4 ? rv[m].y : rv[m].w);
                        mul2(t0, t1, t0, t1, p[hf][c], p[hf][c + 1]);
                        ds[hf][c >> 1] = pack_bf16x2(t0, t1);
                    }
#pragma unroll
            for (int hf = 0; hf < 2; ++hf)
#pragma unroll
                for (int i = 0; i < 8; i += 2) // 16-byte chunks i, i + 1 of 16 rows
                    stmatrix_x4(dsrow + hf * 2048 + (((i + (lane >> 4)) ^ (lane & 7)) << 4), ds[hf][2 * i],
                                ds[hf][2 * i + 1], ds[hf][2 * i + 2], ds[hf][2 * i + 3]);
            fence_proxy_async_smem();
            warp_arrive(BAR(B_DSFULL));
            }
            }
        }
    }

    // ------------------------------------------------------------ teardown
    tc_fence_before();
    __syncthreads();
    if (*abort_flag) {
        if (threadIdx.x == 0)
            atomicCAS(P.status, 0, PEAGLE_ERR_TIMEOUT);
        const uint64_t t0 = globaltimer_ns();
        while (globaltimer_ns() - t0 < 200000ull) {
        }
        __syncthreads();
    }
    if (warp == 8) {
        __syncwarp();
        tc_fence_after();
        tmem_dealloc(tmem, 512);
    }
}

int launch_bwd128_main(const CUtensorMap &tmQ, const CUtensorMap &tmdO, const CUtensorMap &tmK,
                       const CUtensorMap &tmV, const CUtensorMap &tmDQ, const CUtensorMap &tmDK, const CUtensorMap &tmDV,
                       const BwdParams &P, int n_sm, cudaStream_t s)
{
    // per device, so set before every launch (host time only)
    if (cudaFuncSetAttribute(bwd128_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             Bwd128Cfg::SMEM_BYTES) != cudaSuccess)
        return PEAGLE_ERR_CUDA;
    launch_dependent(bwd128_kernel, n_sm, 512, Bwd128Cfg::SMEM_BYTES, s, tmQ, tmdO, tmK, tmV, tmDQ, tmDK, tmDV, P);
    return 1;
}

} // namespace peagle
