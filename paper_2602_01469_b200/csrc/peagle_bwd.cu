// K2: backward of one query partition on sm_100a (dQ, and fp32 accumulation of dK / dV).
//
// Key-tile-outer formulation.  A work item is one key tile (128 keys) of one KV head together
// with the non-skipped query tiles of one aligned chunk of BWD_CQ query tiles; for each of those
// query tiles the item visits the G query heads of the group (one "step" each).  dK and dV of the
// key tile stay in tensor memory for the whole item and are added to the caller's fp32
// accumulators once at its end; dQ of each step is added to an fp32 staging buffer and rounded to
// bf16 by a last kernel.
//
// All score-shaped matrices are held transposed (lanes = keys, columns = query rows) so that the
// probabilities can feed the dV product straight from tensor memory:
//   S^T  = K Q^T,  dP^T = V dO^T
//   P^T  = exp2(scale*log2e*S^T - LSE*log2e), masked entries 0;  dS^T = P^T o (dP^T - Delta)
//   dV  += P^T dO           P^T from tensor memory (bf16, over S^T), dO from shared memory (MN-major)
//   dK  += dS^T Q           Q MN-major
//   dQ   = dS K             dS^T read from shared memory as an MN-major A operand, K MN-major
// Two kernels with the same structure: bwd64_kernel (head_dim 64, below) and bwd128_kernel
// (head_dim 128, peagle_bwd128.cu).
#include <math_constants.h>

#include "peagle_bwd_common.cuh"

namespace peagle {
using namespace sm100;

int make_bf16_map(EncodeTiledFn enc, CUtensorMap *m, const void *base, int D, int H, int T);
int make_f32_map(EncodeTiledFn enc, CUtensorMap *m, float *base, int D, int H, int rows, int box_rows);
int launch_bwd128_main(const CUtensorMap &tmQ, const CUtensorMap &tmdO, const CUtensorMap &tmK,
                       const CUtensorMap &tmV, const CUtensorMap &tmDQ, const CUtensorMap &tmDK, const CUtensorMap &tmDV,
                       const BwdParams &P, int n_sm, cudaStream_t s);

// ---------------------------------------------------------------------------------------------
// head_dim 64.  The query columns of a step are two halves of 64, eight compute warps each, with
// barriers of their own, so that the halves drift apart and the exp2 unit serves one while the other
// does the rest of its step.  The products run one step ahead of the compute warps:
//   S^T(i+1) of a half behind its dV(i), once its P^T(i) is in tensor memory
//   dP^T(i+1) of a half behind its dK(i), once its dS^T(i) is
//   dQ(i) of both halves, once both dS^T(i) are in shared memory
// and are issued by three warps (S^T and dV; dP^T and dK; dQ), because one warp that waits for all of
// these in a fixed order leaves the tensor pipe idle behind every wait (one warp 3.74, three 3.05 ms
// on the headline shape).
// K and V of the item sit in tensor memory as bf16 (A operands of S^T and dP^T): a tensor-memory
// operand leaves half of the shared-memory bandwidth to the other warps, a shared-memory one 5 %.
// dS^T goes both over the dP^T columns (A operand of dK) and, swizzled, to shared memory (A operand
// of dQ).  Sixteen compute warps of 32 keys x 32 query columns: their time is the latency of waits,
// tensor-memory and shared-memory accesses more than arithmetic, so four warps per scheduler hide more
// of each other than two (with eight warps of 64 columns the kernel takes 8 % longer).  The scores are
// read as tcgen05.ld.16x256b gives them: a thread has 4 keys x 8 query columns, so that it needs 8
// instead of 32 of the row values -LSE and -Delta.
// What bounds it now is shared memory: a step moves about 250 KB through it (112 KB operands, 64 KB dQ on
// its way out, 34 KB Q / dO / row values, 32 KB dS^T), 1,950 of its 2,750 clocks; without the dQ tile's
// writes and reads it would take 12 % less time.
// The K tile of the next item is prefetched into a second shared-memory stage (V has one stage: it
// is only read when it is copied to tensor memory at the start of its item); Q / dO have three
// stages (with two, 10 % slower); the items come from a global cursor through a small queue.  768
// threads: warps 0-15 compute, warps 16, 18 and 19 issue MMAs, warp 17 produces, warps 20-23 drain dQ and,
// at the end of an item, dK / dV through fp32 panels in shared memory and tiled reduce-adds.
// The drain has warps of its own because a thread with reductions in flight stalls on its next
// proxy fence, which the compute warps need once per step for the dS^T hand-over.
// Registers per thread after the roles re-split the CTA's allocation (768 threads x 80): four warpgroups
// of compute warps, the warpgroup of the issuing / producing warps, the drain warpgroup.
#ifndef BWD64_COMPUTE_REGS
#define BWD64_COMPUTE_REGS 88
#define BWD64_ISSUE_REGS 48
#define BWD64_DRAIN_REGS 80
#endif
namespace {
constexpr int COMPUTE_REGS = BWD64_COMPUTE_REGS, ISSUE_REGS = BWD64_ISSUE_REGS, DRAIN_REGS = BWD64_DRAIN_REGS;
constexpr int THREADS = 768, LAUNCH_REGS = 80; // 24 warps
static_assert(512 * COMPUTE_REGS + 128 * ISSUE_REGS + 128 * DRAIN_REGS <= THREADS * LAUNCH_REGS,
              "the re-split must fit the launch allocation, or setmaxnreg.inc waits for ever");
} // namespace

struct Bwd64Cfg {
    static constexpr int D = 64;
    static constexpr int NSQ = 3;
    static constexpr int TILE_BYTES = 128 * 128;
    static constexpr int OFF_KV = 0;                              // K stage 0, K stage 1, V (one stage)
    static constexpr int OFF_DS = 3 * TILE_BYTES;                 // 2 panels
    static constexpr int OFF_DQ = OFF_DS + 2 * TILE_BYTES;        // fp32 dQ tile on its way out: 2 panels of 32 columns
    static constexpr int OFF_Q = OFF_DQ + 2 * TILE_BYTES;         // ring of (Q, dO)
    static constexpr int OFF_ROW = OFF_Q + NSQ * 2 * TILE_BYTES;  // ring of (-lse2[128], -delta[128], mq[128])
    static constexpr int ROW_BYTES = 3 * 128 * 4;
    static constexpr int OFF_BAR = OFF_ROW + NSQ * ROW_BYTES;
    static constexpr int N_BAR = 2 * NSQ + 17 + 4;  // the last four: work-queue slots
    static constexpr int OFF_MISC = OFF_BAR + N_BAR * 8; // tensor-memory base, abort flag
    static constexpr int OFF_WQ = (OFF_MISC + 8 + 15) / 16 * 16; // work queue
    static constexpr int SMEM_BYTES = OFF_WQ + BWD_QUEUE_BYTES + 1024;
    // tensor memory: S^T | dP^T | dQ | K (bf16) | V (bf16) | dK | dV.  P^T (bf16) overwrites the
    // first half of each group's S^T columns and dS^T (bf16) the first half of its dP^T columns.
    static constexpr int TM_S = 0, TM_DP = 128, TM_DQ = 256, TM_K = 320, TM_V = 352, TM_DK = 384,
                         TM_DV = 448;
};

__global__ void __launch_bounds__(THREADS, 1)
bwd64_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmdO,
             const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmV,
             const __grid_constant__ CUtensorMap tmDQ, const __grid_constant__ CUtensorMap tmDK,
             const __grid_constant__ CUtensorMap tmDV, const BwdParams P)
{
    using C = Bwd64Cfg;
    constexpr int D = 64, NSQ = C::NSQ, TB = C::TILE_BYTES;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t sb = (raw + 1023u) & ~1023u;
    uint8_t *sp = smem_raw + (sb - raw);
    const uint32_t bar0 = sb + C::OFF_BAR;
    auto BAR = [&](int i) { return bar0 + 8u * (uint32_t)i; };
    constexpr int B_QFULL = 0, B_QEMPTY = NSQ, B_KVFULL = 2 * NSQ, B_KVEMPTY = B_KVFULL + 2,
                  // per half of the query columns (compute warpgroup): [0], [1]
                  B_SFULL = B_KVFULL + 4, B_DPFULL = B_KVFULL + 6, B_PFULL = B_KVFULL + 8,
                  B_DSFULL = B_KVFULL + 10, B_DQFULL = B_KVFULL + 12, B_KVTFULL = B_KVFULL + 13,
                  B_DQEMPTY = B_KVFULL + 14, B_ACCFREE = B_KVFULL + 15,
                  B_ITEMDONE = B_KVFULL + 16;
    volatile uint32_t *tmem_slot = reinterpret_cast<volatile uint32_t *>(sp + C::OFF_MISC);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(sp + C::OFF_MISC + 4);
    uint8_t *wq = sp + C::OFF_WQ;
    constexpr int B_WQ = 2 * NSQ + 17;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    if (threadIdx.x == 0) {
        *abort_flag = 0;
        for (int s = 0; s < NSQ; ++s) {
            mbar_init(BAR(B_QFULL + s), 1);
            mbar_init(BAR(B_QEMPTY + s), 2); // the S^T / dV and the dP^T / dK issuer
        }
        for (int s = 0; s < 4; ++s)
            mbar_init(BAR(B_WQ + s), 1);
        for (int s = 0; s < 2; ++s) {
            mbar_init(BAR(B_KVFULL + s), 1);
            mbar_init(BAR(B_KVEMPTY + s), 1);
            mbar_init(BAR(B_SFULL + s), 1);
            mbar_init(BAR(B_DPFULL + s), 1);
            mbar_init(BAR(B_PFULL + s), 8); // one arrival per warp
            mbar_init(BAR(B_DSFULL + s), 8);
        }
        mbar_init(BAR(B_DQFULL), 1);
        mbar_init(BAR(B_KVTFULL), 16);
        mbar_init(BAR(B_DQEMPTY), 4);
        mbar_init(BAR(B_ITEMDONE), 2);
        mbar_init(BAR(B_ACCFREE), 4);
        fence_mbar_init();
    }
    if (warp == 16) {
        tmem_alloc(sb + C::OFF_MISC, 512);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    pdl_wait();
    pdl_trigger();

    if (warp >= 20) {
        // ------------------------------------------------------------ drain (warps 20-23)
        reg_set<DRAIN_REGS, LAUNCH_REGS>();
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
            uint8_t *dst = sp + C::OFF_DQ + slot * TB + ((warp & 3) * 32 + lane) * 128;
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
                tma_reduce_add_3d(map, sb + C::OFF_DQ + slot * TB + (warp & 3) * 4096, x, y, z + (warp & 3) * 32);
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
            ok = mbar_wait_warp(BAR(B_DQFULL), it & 1, abort_flag);
            if (!ok)
                break;
            tc_fence_after();
            // dQ(it) (rows past the partition's end are clipped by the tensor map)
            uint32_t o[2][32];
#pragma unroll
            for (int pn = 0; pn < 2; ++pn)
                tmem_ld32(tmem + lane_base + C::TM_DQ + pn * 32, o[pn]);
            tmem_wait_ld();
            tc_fence_before();
            warp_arrive(BAR(B_DQEMPTY));
#pragma unroll
            for (int pn = 0; pn < 2; ++pn)
                send(o[pn], P.scale, pn & 1, &tmDQ, 32 * pn, h, row0);
        }
        if (!ok)
            break;
        // dK and dV of the work item
        ok = mbar_wait_warp(BAR(B_ITEMDONE), w & 1, abort_flag);
        if (!ok)
            break;
        tc_fence_after();
        // Keys past a ragged tile's end are another range's, often another sequence's.  Their sums have weight
        // zero throughout, but a zero times an Inf or NaN of a row of Q or dO is not zero, so zeros are
        // what they get.
        const int rows = item.k_len - (warp & 3) * 32; // of this warp's 32 keys, how many are the tile's
#pragma unroll
        for (int t = 0; t < 2; ++t) { // dK, then dV
            uint32_t o[2][32];
            tmem_ld32(tmem + lane_base + (t ? C::TM_DV : C::TM_DK), o[0]);
            tmem_ld32(tmem + lane_base + (t ? C::TM_DV : C::TM_DK) + 32, o[1]);
            tmem_wait_ld();
            if (t) {
                tc_fence_before();
                warp_arrive(BAR(B_ACCFREE));
            }
            if (lane >= rows) {
#pragma unroll
                for (int i = 0; i < 32; ++i)
                    o[0][i] = o[1][i] = 0;
            }
            if (rows > 0) {
#pragma unroll
                for (int pn = 0; pn < 2; ++pn)
                    send(o[pn], t ? 1.f : P.scale, pn, t ? &tmDV : &tmDK, 32 * pn, item.g, item.k_start);
            }
        }
        }
        if (lane == 0)
            bulk_wait_group<0>();
    } else if (warp >= 16) {
        reg_set<ISSUE_REGS, LAUNCH_REGS>();
        if (warp == 17) {
            // -------------------------------------------------------- producer
            if (lane == 0) {
                tma_prefetch_desc(&tmQ);
                tma_prefetch_desc(&tmdO);
                tma_prefetch_desc(&tmK);
                tma_prefetch_desc(&tmV);
            }
            const BwdSplit split = bwd_split(P);
            BwdItem item, nxt;
            auto load_kv = [&](int w, const BwdItem &x) -> bool {
                bool ok = true;
                if (lane == 0) {
                    const int s = w & 1;
                    ok = mbar_wait(BAR(B_KVEMPTY + s), ((w >> 1) & 1) ^ 1, abort_flag) &&
                         (w == 0 || mbar_wait(BAR(B_KVTFULL), (w - 1) & 1, abort_flag));
                    if (ok) {
                        mbar_arrive_expect_tx(BAR(B_KVFULL + s), 2 * TB);
                        tma_load_3d(sb + C::OFF_KV + s * TB, &tmK, BAR(B_KVFULL + s), 0, x.g, x.k_start);
                        tma_load_3d(sb + C::OFF_KV + 2 * TB, &tmV, BAR(B_KVFULL + s), 0, x.g, x.k_start);
                    }
                }
                return __all_sync(0xffffffffu, ok);
            };
            int it = 0;
            bool more = bwd_draw(P, split, wq, BAR(B_WQ), 0, lane, item);
            bool ok = !more || load_kv(0, item);
            for (int w = 0; ok && more; ++w) {
                unsigned em = item.mask & 0xffu;
                for (int i = 0, hh = 0; i < item.steps; ++i, ++it) {
                    const int st = it % NSQ, ph = (it / NSQ) & 1;
                    const int qt = item.qt0 + __ffs(em) - 1, h = item.h0 + hh;
                    if (++hh == item.nh) {
                        hh = 0;
                        em &= em - 1;
                    }
                    ok = mbar_wait_warp(BAR(B_QEMPTY + st), ph ^ 1, abort_flag);
                    if (!ok)
                        break;
                    if (lane == 0) {
                        const int row0 = P.q_begin + qt * BM;
                        mbar_arrive_expect_tx(BAR(B_QFULL + st), 2 * TB + C::ROW_BYTES);
                        const uint32_t qa = sb + C::OFF_Q + st * 2 * TB;
                        tma_load_3d(qa, &tmQ, BAR(B_QFULL + st), 0, h, row0);
                        tma_load_3d(qa + TB, &tmdO, BAR(B_QFULL + st), 0, h, row0);
                        const uint32_t ra = sb + C::OFF_ROW + st * C::ROW_BYTES;
                        const size_t ri = (size_t)h * P.q_pad + (size_t)qt * BM;
                        bulk_load(ra, P.nl2 + ri, 512, BAR(B_QFULL + st));
                        bulk_load(ra + 512, P.nd + ri, 512, BAR(B_QFULL + st));
                        bulk_load(ra + 1024, P.mqp + (size_t)qt * BM, 512, BAR(B_QFULL + st));
                    }
                    // the next step's Q / dO tiles start towards L2 one step before their stage is
                    // free; the next item is drawn, and its K / V requested, with the last step
                    if (i + 1 < item.steps) {
                        if (lane == 0) {
                            const int row1 = P.q_begin + (item.qt0 + __ffs(em) - 1) * BM;
                            tma_prefetch_3d(&tmQ, 0, item.h0 + hh, row1);
                            tma_prefetch_3d(&tmdO, 0, item.h0 + hh, row1);
                        }
                    } else {
                        more = bwd_draw(P, split, wq, BAR(B_WQ), w + 1, lane, nxt);
                        if (more)
                            ok = load_kv(w + 1, nxt);
                    }
                }
                item = nxt;
            }
        } else {
            // -------------------------------------------------------- MMA issue: three warps, each
            // with its own accumulators (products into one accumulator keep one thread's order):
            // warp 16 S^T and dV, warp 18 dP^T and dK, warp 19 dQ.  The whole warp walks the steps
            // and waits, its elected lane issues (see elect_one).
            const uint32_t lead = elect_one();
            constexpr uint32_t IDESC_S = idesc_bf16_f32(128, 64, 0, 0);
            constexpr uint32_t IDESC_KV = idesc_bf16_f32(128, D, 0, 1);
            constexpr uint32_t IDESC_DQ = idesc_bf16_f32(128, D, 1, 1);
            // Lower descriptor words (16-byte units).  "k" = K-major operand, "m" = MN-major.
            const uint32_t ds_m = desc_lo_sw128(sb + C::OFF_DS, TB);
            const uint32_t kv_m = desc_lo_sw128(sb + C::OFF_KV, TB);
            constexpr uint32_t TBU = TB >> 4; // one tile in descriptor units
            // warp 16: Q for S^T, dO for dV; warp 18: dO for dP^T, Q for dK
            const uint32_t b_k = desc_lo_sw128(sb + C::OFF_Q, 16) + (warp == 16 ? 0 : TBU);
            const uint32_t b_m = desc_lo_sw128(sb + C::OFF_Q, TB) + (warp == 16 ? TBU : 0);
            const uint32_t t_sc = tmem + (warp == 16 ? C::TM_S : C::TM_DP), t_kv = tmem + (warp == 16 ? C::TM_K : C::TM_V),
                           t_acc = tmem + (warp == 16 ? C::TM_DV : C::TM_DK);
            const uint32_t bar_sc = BAR(warp == 16 ? B_SFULL : B_DPFULL), bar_in = BAR(warp == 16 ? B_PFULL : B_DSFULL);
            // The products of one step, by half h of its query columns (64 each, one compute
            // warpgroup's); q = offset of the step's Q / dO stage in descriptor units.
            auto issue_score = [&](uint32_t q, int h) { // S^T = K Q^T / dP^T = V dO^T, K / V in tensor memory
#pragma unroll
                for (int k = 0; k < D / 16; ++k)
                    if (lead) mma_ts_lo(t_sc + h * 64, t_kv + k * 8, b_k + q + h * 512 + k * 2, IDESC_S, k > 0);
                if (lead) tc_commit(bar_sc + 8 * h);
            };
            auto issue_acc = [&](uint32_t q, int h, bool acc) { // dV += P^T dO / dK += dS^T Q, 64 query rows
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    if (lead) mma_ts_lo(t_acc, t_sc + h * 64 + (k >> 1) * 32 + (k & 1) * 8, b_m + q + (h * 4 + k) * 128, IDESC_KV,
                              acc || k > 0);
            };
            bool ok = true;
            int it = 0, w = 0;
            BwdItem item;
            for (; bwd_take(wq, BAR(B_WQ), w, abort_flag, item); ++w) {
                const int n_cur = item.steps;
                const int ks = w & 1;
                if (warp == 19) {
                    const uint32_t kvo = ks * TBU;
                    for (int i = 0; ok && i < n_cur; ++i, ++it) {
                        ok = mbar_wait_warp(BAR(B_DSFULL), it & 1, abort_flag) &&
                             mbar_wait_warp(BAR(B_DSFULL + 1), it & 1, abort_flag) &&
                             mbar_wait_warp(BAR(B_DQEMPTY), (it & 1) ^ 1, abort_flag); // the accumulator has been read out
                        if (!ok)
                            break;
                        tc_fence_after();
#pragma unroll
                        for (int k = 0; k < 8; ++k)
                            if (lead) mma_ss_lo(tmem + C::TM_DQ, ds_m + k * 128, kv_m + kvo + k * 128, IDESC_DQ, k > 0);
                        if (lead) tc_commit(BAR(B_DQFULL));
                    }
                    if (!ok)
                        break;
                    if (lead) tc_commit(BAR(B_KVEMPTY + ks));
                    continue;
                }
                // K / V of this item are in tensor memory
                ok = mbar_wait_warp(BAR(B_KVTFULL), w & 1, abort_flag) &&
                     mbar_wait_warp(BAR(B_QFULL + it % 3), (it / 3) & 1, abort_flag);
                if (!ok)
                    break;
                tc_fence_after();
                issue_score((it % 3) * 2 * TBU, 0);
                issue_score((it % 3) * 2 * TBU, 1);
                for (int i = 0; ok && i < n_cur; ++i, ++it) {
                    const int st = it % 3, nst = (it + 1) % 3;
                    const uint32_t qo = st * 2 * TBU, nqo = nst * 2 * TBU;
                    const bool first = i == 0, last = i == n_cur - 1;
                    ok = mbar_wait_warp(bar_in, it & 1, abort_flag);
                    if (ok && first)
                        ok = mbar_wait_warp(BAR(B_ACCFREE), (w & 1) ^ 1, abort_flag);
                    if (!ok)
                        break;
                    tc_fence_after();
                    issue_acc(qo, 0, !first);
                    if (!last) {
                        ok = mbar_wait_warp(BAR(B_QFULL + nst), ((it + 1) / 3) & 1, abort_flag);
                        if (!ok)
                            break;
                        tc_fence_after();
                        issue_score(nqo, 0);
                    }
                    ok = mbar_wait_warp(bar_in + 8, it & 1, abort_flag);
                    if (!ok)
                        break;
                    tc_fence_after();
                    issue_acc(qo, 1, true);
                    if (lead) tc_commit(BAR(B_QEMPTY + st));
                    if (!last)
                        issue_score(nqo, 1);
                }
                if (!ok)
                    break;
                if (lead) tc_commit(BAR(B_ITEMDONE));
            }
        }
    } else {
        reg_set<COMPUTE_REGS, LAUNCH_REGS>();
        // ------------------------------------------------------------ compute (warps 0-15)
        const int wg = warp >> 3;       // half of the query columns
        const int ch = (warp >> 2) & 1; // 32 of its 64 columns
        const int r = (warp & 3) * 32 + lane;
        const uint32_t lane_sel = (uint32_t)((warp & 3) * 32) << 16;
        const uint32_t tS = tmem + lane_sel + C::TM_S + wg * 64 + ch * 32;
        const uint32_t tDP = tmem + lane_sel + C::TM_DP + wg * 64 + ch * 32;
        // row of the dS^T tile that this lane addresses in stmatrix_x4 (see there): its row of the
        // first 16, chunk added per store
        const uint32_t dsrow = sb + C::OFF_DS + wg * TB + ((warp & 3) * 32 + (lane & 15)) * 128;
        bool ok = true;
        int it = 0, st = 0; // step of this CTA, its Q / dO stage
        BwdItem item;
        for (int w = 0; ok && bwd_take(wq, BAR(B_WQ), w, abort_flag, item); ++w) {
            int32_t mk[4]; // metadata of the keys of this thread's four lanes
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int kl = (warp & 3) * 32 + 8 * i + (lane >> 2);
                mk[i] = (kl < item.k_len) ? P.meta[item.k_start + kl] : META_NONE_K;
            }
            {
                // New work item: a bf16 copy of K (group 0) / V (group 1) goes to tensor memory,
                // half a row per thread.  Every S^T / dP^T product of the previous item is complete
                // (their results were consumed in its last step), so the old copy is not in use.
                const int ks = w & 1;
                // (The other group's last S^T / dP^T must be complete as well.)
                ok = mbar_wait_warp(BAR(B_KVFULL + ks), (w >> 1) & 1, abort_flag) &&
                     (it == 0 || mbar_wait_warp(BAR(wg == 0 ? B_SFULL + 1 : B_DPFULL), (it - 1) & 1, abort_flag));
                if (!ok)
                    break;
                const uint8_t *src = sp + C::OFF_KV + (wg == 0 ? ks : 2) * TB + r * 128;
                uint32_t kvw[16];
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const uint4 v = *reinterpret_cast<const uint4 *>(src + (((4 * ch + c) ^ (r & 7)) << 4));
                    kvw[4 * c] = v.x;
                    kvw[4 * c + 1] = v.y;
                    kvw[4 * c + 2] = v.z;
                    kvw[4 * c + 3] = v.w;
                }
                tmem_st16(tmem + lane_sel + (wg == 0 ? C::TM_K : C::TM_V) + ch * 16, kvw);
                tmem_wait_st();
                tc_fence_before();
                warp_arrive(BAR(B_KVTFULL));
            }
            for (unsigned em = item.mask & 0xffu; ok && em; em &= em - 1) {
            const bool full = (item.mask >> (7 + __ffs(em))) & 1u;
            for (int hh = 0; hh < item.nh; ++hh, ++it, st = st == NSQ - 1 ? 0 : st + 1) {
            const float *rowbuf = reinterpret_cast<const float *>(sp + C::OFF_ROW + st * C::ROW_BYTES);
            const float4 *nl4 = reinterpret_cast<const float4 *>(rowbuf + wg * 64 + ch * 32) + (lane & 3);
            const float4 *nd4 = reinterpret_cast<const float4 *>(rowbuf + 128 + wg * 64 + ch * 32) + (lane & 3);
            const int4 *mq4 = reinterpret_cast<const int4 *>(rowbuf + 256 + wg * 64 + ch * 32) + (lane & 3);
            // ---- P^T.  A thread holds 4 key lanes x 8 query columns (tmem_ld_16x256b_x4): for each
            // group i of 8 columns the columns 8i + 2 (lane % 4) and the next one.
            // The row values came with the step's Q tile, which the products read: complete.
            ok = mbar_wait_warp(BAR(B_SFULL + wg), it & 1, abort_flag);
            if (!ok)
                break;
            tc_fence_after();
            float4 rv[2]; // row values of the thread's columns
#pragma unroll
            for (int m = 0; m < 2; ++m)
                rv[m] = nl4[4 * m];
            uint32_t sr[2][16];
            tmem_ld_16x256b_x4(tS, sr[0]);
            tmem_ld_16x256b_x4(tS + (16u << 16), sr[1]);
            tmem_wait_ld();
            float p[2][16];
#pragma unroll
            for (int m = 0; m < 2; ++m)
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
                int4 mq[2];
#pragma unroll
                for (int m = 0; m < 2; ++m)
                    mq[m] = mq4[4 * m];
                int first = mq[0].x;
#pragma unroll
                for (int m = 0; m < 2; ++m)
                    first = min(min(first, min(mq[m].x, mq[m].y)), min(mq[m].z, mq[m].w));
                const int last = max(max(mk[0], mk[1]), max(mk[2], mk[3]));
                if (!__all_sync(0xffffffffu, last <= first && ((mk[0] | mk[1] | mk[2] | mk[3]) & 0xff) == 0)) {
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const uint32_t span = allowed_span(mk[k]);
#pragma unroll
                        for (int m = 0; m < 2; ++m)
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
            for (int m = 0; m < 2; ++m)
                rv[m] = nd4[4 * m]; // used by dS^T, requested ahead of the hand-over
#pragma unroll
            for (int hf = 0; hf < 2; ++hf) {
                uint32_t pk[8];
#pragma unroll
                for (int i = 0; i < 8; ++i)
                    pk[i] = pack_bf16x2(p[hf][2 * i], p[hf][2 * i + 1]);
                // packed P^T over the first half of this warp's S^T columns
                tmem_st_16x128b_x4(tS + ((16u * hf) << 16), pk);
            }
            tmem_wait_st();
            tc_fence_before();
            warp_arrive(BAR(B_PFULL + wg));
            // ---- dS^T
            // (and dQ of the previous step has run, so that the dS^T panel is free)
            ok = mbar_wait_warp(BAR(B_DPFULL + wg), it & 1, abort_flag) &&
                 (it == 0 || mbar_wait_warp(BAR(B_DQFULL), (it - 1) & 1, abort_flag));
            if (!ok)
                break;
            tc_fence_after();
            tmem_ld_16x256b_x4(tDP, sr[0]);
            tmem_ld_16x256b_x4(tDP + (16u << 16), sr[1]);
            tmem_wait_ld();
            tc_fence_before();
            uint32_t ds[2][8];
#pragma unroll
            for (int m = 0; m < 2; ++m)
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
            // the same dS^T goes over this group's dP^T columns (operand of dK) and to shared memory
#pragma unroll
            for (int hf = 0; hf < 2; ++hf)
                tmem_st_16x128b_x4(tDP + ((16u * hf) << 16), ds[hf]);
#pragma unroll
            for (int hf = 0; hf < 2; ++hf)
#pragma unroll
                for (int i = 0; i < 4; i += 2) // 16-byte chunks 4 ch + i, + 1 of 16 rows
                    stmatrix_x4(dsrow + hf * 2048 + (((4 * ch + i + (lane >> 4)) ^ (lane & 7)) << 4), ds[hf][2 * i],
                                ds[hf][2 * i + 1], ds[hf][2 * i + 2], ds[hf][2 * i + 3]);
            tmem_wait_st();
            fence_proxy_async_smem();
            tc_fence_before();
            warp_arrive(BAR(B_DSFULL + wg));
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
    if (warp == 16) {
        __syncwarp();
        tc_fence_after();
        tmem_dealloc(tmem, 512);
    }
}

__global__ void bwd_finish_dq(const float *__restrict__ dq_acc, __nv_bfloat16 *__restrict__ dQ,
                              size_t n8)
{
    pdl_wait();
    pdl_trigger();
    const size_t gid = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (gid >= n8)
        return;
    const float4 a = reinterpret_cast<const float4 *>(dq_acc)[2 * gid];
    const float4 b = reinterpret_cast<const float4 *>(dq_acc)[2 * gid + 1];
    uint4 v;
    v.x = pack_bf16x2(a.x, a.y);
    v.y = pack_bf16x2(a.z, a.w);
    v.z = pack_bf16x2(b.x, b.y);
    v.w = pack_bf16x2(b.z, b.w);
    reinterpret_cast<uint4 *>(dQ)[gid] = v;
}

__global__ void cast_grads_kernel(const float *__restrict__ a, const float *__restrict__ b,
                                  __nv_bfloat16 *__restrict__ oa, __nv_bfloat16 *__restrict__ ob,
                                  size_t n8)
{
    pdl_wait();
    pdl_trigger();
    const size_t gid = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (gid >= 2 * n8)
        return;
    const float *src = gid < n8 ? a : b;
    __nv_bfloat16 *dst = gid < n8 ? oa : ob;
    const size_t i = gid < n8 ? gid : gid - n8;
    const float4 x = reinterpret_cast<const float4 *>(src)[2 * i];
    const float4 y = reinterpret_cast<const float4 *>(src)[2 * i + 1];
    uint4 v;
    v.x = pack_bf16x2(x.x, x.y);
    v.y = pack_bf16x2(x.z, x.w);
    v.z = pack_bf16x2(y.x, y.y);
    v.w = pack_bf16x2(y.z, y.w);
    reinterpret_cast<uint4 *>(dst)[i] = v;
}

template <int D>
static int launch_bwd_t(const Plan &p, const BwdArgs &a, EncodeTiledFn enc, int n_sm, cudaStream_t s,
                        cudaEvent_t ev0, cudaEvent_t ev1)
{
    // Q and dO maps end at the partition's last row so that rows past it read as zeros.
    CUtensorMap tmQ, tmdO, tmK, tmV;
    if (make_bf16_map(enc, &tmQ, a.Q, D, a.Hq, p.q_end) || make_bf16_map(enc, &tmdO, a.dO, D, a.Hq, p.q_end) ||
        make_bf16_map(enc, &tmK, a.K, D, a.Hkv, p.T) || make_bf16_map(enc, &tmV, a.V, D, a.Hkv, p.T))
        return PEAGLE_ERR_CUDA;
    const int q_len = p.q_end - p.q_begin;
    const int q_pad = p.n_qt * BM;
    // fp32 sums as tensors for tiled reduce-adds, 32 columns x 32 rows: the dQ staging
    // [q_len][Hq][D] and the caller's dK / dV [T][Hkv][D]
    CUtensorMap tmDQ, tmDK, tmDV;
    if (make_f32_map(enc, &tmDQ, a.dq_acc, D, a.Hq, q_len, 32) || make_f32_map(enc, &tmDK, a.dK_acc, D, a.Hkv, p.T, 32) ||
        make_f32_map(enc, &tmDV, a.dV_acc, D, a.Hkv, p.T, 32))
        return PEAGLE_ERR_CUDA;
    const size_t n8 = (size_t)q_len * a.Hq * (D / 8);
    int launches = 0;
    if (p.n_kt > 0) {
        BwdParams P;
        P.ktile = p.ktile;
        P.bitems = p.bitems;
        P.counters = p.counters;
        P.cursor = p.counters + CNT_BWD_CURSOR;
        P.meta = p.meta;
        P.status = p.status;
        P.n_qt = p.n_qt;
        P.n_kt = p.n_kt;
        P.q_begin = p.q_begin;
        P.nl2 = a.nl2;
        P.nd = a.nd;
        P.mqp = a.mqp;
        P.q_pad = q_pad;
        P.dq_acc = a.dq_acc;
        P.dK_acc = a.dK_acc;
        P.dV_acc = a.dV_acc;
        P.Hq = a.Hq;
        P.Hkv = a.Hkv;
        P.scale = a.scale;
        P.scale_log2 = a.scale * 1.4426950408889634f;
        // per device, so set before every launch (host time only)
        if (D == 64 && cudaFuncSetAttribute(bwd64_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                            Bwd64Cfg::SMEM_BYTES) != cudaSuccess)
            return PEAGLE_ERR_CUDA;
        if (ev0)
            cudaEventRecord(ev0, s);
        if (D == 64)
            launch_dependent(bwd64_kernel, n_sm, THREADS, Bwd64Cfg::SMEM_BYTES, s, tmQ, tmdO, tmK, tmV, tmDQ, tmDK, tmDV, P);
        else if (launch_bwd128_main(tmQ, tmdO, tmK, tmV, tmDQ, tmDK, tmDV, P, n_sm, s) < 0)
            return PEAGLE_ERR_CUDA;
        if (ev1)
            cudaEventRecord(ev1, s);
        ++launches;
    }
    if (p.allow_single) {
        const int n = launch_finish_single(p, a, s);
        return n < 0 ? n : launches + n;
    }
    launch_dependent(
        bwd_finish_dq, (unsigned)((n8 + 255) / 256), 256, 0, s, a.dq_acc, static_cast<__nv_bfloat16 *>(a.dQ) + (size_t)p.q_begin * a.Hq * D, n8);
    return launches + 1;
}

int launch_bwd(const Plan &p, const BwdArgs &a, EncodeTiledFn enc, int n_sm, cudaStream_t s,
               cudaEvent_t ev0, cudaEvent_t ev1)
{
    if (p.n_qt == 0)
        return 0;
    return a.D == 64 ? launch_bwd_t<64>(p, a, enc, n_sm, s, ev0, ev1)
                     : launch_bwd_t<128>(p, a, enc, n_sm, s, ev0, ev1);
}

// One fp32 array of n elements (a multiple of 8) rounded to bf16.
int launch_cast_one(const float *src, void *dst, size_t n, cudaStream_t s)
{
    const size_t n8 = n / 8;
    if (n8 == 0)
        return 0;
    // the kernel takes two arrays of n8 pieces; here both are the one array, and the grid covers it
    // once (threads past n8 in the last block repeat the first pieces with the same values)
    launch_dependent(
        cast_grads_kernel, (unsigned)((n8 + 255) / 256), 256, 0, s, src, src, static_cast<__nv_bfloat16 *>(dst), static_cast<__nv_bfloat16 *>(dst), n8);
    return 1;
}

int launch_cast_grads(const float *dK_acc, const float *dV_acc, void *dK, void *dV, size_t n,
                      cudaStream_t s)
{
    const size_t n8 = n / 8;
    launch_dependent(
        cast_grads_kernel, (unsigned)((2 * n8 + 255) / 256), 256, 0, s, dK_acc, dV_acc, static_cast<__nv_bfloat16 *>(dK), static_cast<__nv_bfloat16 *>(dV), n8);
    return 1;
}

} // namespace peagle
