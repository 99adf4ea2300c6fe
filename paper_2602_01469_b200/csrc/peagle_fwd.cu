// K1: forward of one query partition on sm_100a.
//
// A work item is one query tile (128 rows) for two query heads of the same KV group (or one head
// when the group size is odd), so both tiles share the K/V tiles staged in shared memory and the
// same mask.  The kernel is persistent: one CTA per SM (it takes all of tensor memory and of the
// register file) draws items from a global counter, longest query tiles first, and its
// barriers, K / V ring and tensor memory carry on from item to item, so that the loads and the
// first S product of the next item run under the last softmax and the epilogue of the current
// one.  Roles (384 threads):
//   warps 0-3  softmax of tile A (one query row per thread; online softmax in the log2 domain,
//              log-sum-exp bookkeeping, final normalisation and store)
//   warps 4-7  softmax of tile B
//              (rows of O leave through shared memory: at head_dim 64 by one tiled store per tile, at 128
//              32 rows by 32 columns at a time; not as 32 scattered 16-byte pieces per store instruction)
//   warp  8    allocates tensor memory; its elected lane issues the MMAs of tile A
//   warp  10   its elected lane issues the MMAs of tile B
//   warp  9    producer: draws the items; TMA loads of Q per item and of the K / V tiles
//              through a ring, plus the packed metadata of each key tile for the implicit mask
// Tensor memory (512 columns x 128 lanes, fp32): S_A | S_B (128 columns each), O_A | O_B
// (head_dim each) and, for head_dim 64, P_A | P_B (bf16 probabilities, 64 columns each) so that
// S(j+1) is computed while the softmax of S(j) runs; for head_dim 128 tensor memory is full and
// the probabilities overwrite the first 64 columns of their own S.
// S = Q K^T takes both operands from shared memory (K-major, 128-byte swizzle); O += P V takes
// P from tensor memory and V from shared memory (MN-major).
// Only tiles the classifier kept are visited; FULL tiles skip the per-element predicate; SINGLE
// entries (windows with one allowed key per row) pass through the same ring first and are done on the CUDA
// cores in two passes, scores and weighted values, their result seeding the running (m, l, O).
#include <math_constants.h>

#include <algorithm>

#include "peagle_internal.h"
#include "sm100_ptx.cuh"

namespace peagle {
using namespace sm100;

struct FwdParams {
    const int2 *klist;
    const int *kcount;
    const int *qorder;
    const int32_t *meta;
    int *status;
    int *cursor;  // next work item (zero at launch)
    int n_items;  // query tiles x head blocks
    int n_kt, q_begin, q_end, T;
    __nv_bfloat16 *O;
    float *LSE;
    int Hq, Hkv;
    int two; // 1: two heads per CTA
    float scale_log2;
    // SINGLE tiles (one allowed key per row), handled pair by pair before the tile loop
    const int *scount;
    const uint8_t *scs;  // [n_qt][MAX_SINGLE][BM] key of row r in entry i's window, or NO_COL
    const int *sbase;    // [n_qt][MAX_SINGLE] first token of entry i's window
    // Optional hand-over to the backward of the same partition (the driver knows dO when the
    // forward runs): per (head, row) -LSE * log2(e) and -Delta = -<dO, O>, [Hq][q_pad] each, and
    // the rows' packed metadata [q_pad], neutral values for the rows past the partition's end.
    const __nv_bfloat16 *dO; // null: nothing is handed over
    float *nl2, *nd;
    int32_t *mqp;
    int q_pad;
};

template <int D>
struct FwdCfg {
    static constexpr int NS = (D == 64) ? 3 : 2;
    // SINGLE entries per pass: at head_dim 64 as many as the ring holds, so that the next ones' K arrives under
    // these ones' V and their V under that K (4,096 positions, 64 heads: 1,617 us, all at once 1,650); at 128, where
    // the ring holds two and O would go through tensor memory between them, all (2,048 positions, 32
    // heads: 365 us, as many as the ring holds 378).
    static constexpr int CHUNK = (D == 64) ? NS : MAX_SINGLE;
    static constexpr bool ONE_CHUNK = CHUNK >= MAX_SINGLE;
    static constexpr int PANELS = D / 64;
    static constexpr int PANEL_BYTES = 128 * 128; // 128 rows of 128 bytes
    static constexpr int TILE_BYTES = PANELS * PANEL_BYTES;
    static constexpr int OFF_Q = 0;
    static constexpr int OFF_K = 2 * TILE_BYTES;
    static constexpr int OFF_V = OFF_K + NS * TILE_BYTES;
    // head_dim 64: the finished O tiles leave through shared memory and a tiled store (a thread
    // that writes its own row puts 32 separate 16-byte pieces into every store instruction of its
    // warp); head_dim 128 has no room for the two staging tiles: its rows pass through 2 KB per warp
    // and leave by plain stores of four neighbouring lanes to a row
    static constexpr bool O_STAGED = (D == 64);
    static constexpr int OFF_OST = OFF_V + NS * TILE_BYTES;
    // ZERO_ROWS x 32 fp32 zeros, the source of the stores that clear the backward's dQ staging
    static constexpr int ZERO_ROWS = (D == 64) ? 128 : 64;
    static constexpr int OFF_ZERO = OFF_OST + (O_STAGED ? 2 * TILE_BYTES : 0);
    // SINGLE entries of the item: the rows' keys [entry][row]; and 2 KB per softmax warp, the scores [entry][lane],
    // at head_dim 128 in the epilogue 32 rows of 32 columns of dO or O on their way
    static constexpr int OFF_COL = OFF_ZERO + ZERO_ROWS * 128;
    static constexpr int OFF_SCORE = OFF_COL + MAX_SINGLE * BM;
    static constexpr int WARP_BYTES = MAX_SINGLE * 32 * 4;
    static constexpr int OFF_META = OFF_SCORE + 8 * WARP_BYTES;
    static constexpr int OFF_BAR = OFF_META + NS * BN * 4;
    static constexpr int N_BAR = 1 + 4 * NS + 10 + 9 + 8;
    static constexpr int OFF_MISC = (OFF_BAR + N_BAR * 8 + 15) / 16 * 16; // tmem slot, abort flag; item queue
    static constexpr int SMEM_BYTES = OFF_MISC + 16 + 4 * 16 + 1024;      // + slack for 1024-byte alignment
    static constexpr int TM_S = 0;      // S_A at 0, S_B at 128
    static constexpr int TM_O = 256;    // O_A at 256, O_B at 256 + D
    // head_dim 64 leaves 128 columns for the bf16 probabilities (64 columns per tile), so the next
    // S can be computed while the softmax of the current one runs.  head_dim 128 fills tensor
    // memory with S and O, and P overwrites the first 64 columns of its own S.
    static constexpr bool P_SEPARATE = (D == 64);
    static constexpr int TM_P = P_SEPARATE ? 384 : 0;   // P_A, then P_B at + P_STRIDE
    static constexpr int P_STRIDE = P_SEPARATE ? 64 : 128;
    // P is handed over in two halves where S(j+1) waits for P V(j): P V starts under the second half of the
    // exponentials (2,048 positions, 32 heads of 128: 398 -> 388 us).  With S in columns of its own P V has time,
    // and the extra hand-over costs (3,891 positions, 64 heads of 64: 1,633 -> 1,723 us).
    static constexpr bool P_HALVES = !P_SEPARATE;
};

// The n lowest bits (none below 1, all from 32 on).
__device__ __forceinline__ uint32_t bits_below(int n)
{
    uint32_t r;
    asm("shl.b32 %0, 1, %1;" : "=r"(r) : "r"(max(n, 0))); // clamps: 32 and more give 0
    return r - 1u;
}
// The keys that row mq allows of a PARTIAL tile with KLIST_EVEN, a bit per key.  In a run of one kind whose anchors
// follow one another they are neighbours, depth-0 keys up to mq or the keys of the row's own chain up to mq, and
// their places are subtractions.  A warp then passes over the 32 columns that all its rows see.  (The predicate
// for every element takes 2,200 clocks of a tile, as much as all else in it: forward of 500 positions, 64 heads
// of 64, 114.4 -> 106.7 us; 3,891 positions 1,714 -> 1,648.  For the other tiles, of COD sets or anchor-major
// orders, it stays: searches of eight dependent reads in sorted runs, or bits from the predicate, were slower.)
__device__ __forceinline__ void row_mask(const int32_t *mk, int word, int32_t mq, uint32_t (&see)[4])
{
    const int split = klist_split(word), len = klist_len(word);
    auto first_above = [&](int lo, int end, int w) { // first key of lo .. end - 1 above w
        return lo + min(max(((w - mk[lo]) >> 8) + 1, 0), end - lo);
    };
    const int own = (mq & ~0xff) - 1; // below the row's chain
    const int e0 = first_above(0, split, mq), b0 = word & KLIST_RUN0 ? 0 : first_above(0, split, own);
    int e1 = split, b1 = split;
    if (split < len) {
        e1 = first_above(split, len, mq);
        if (!(word & KLIST_RUN1))
            b1 = first_above(split, len, own);
    }
#pragma unroll
    for (int c = 0; c < 4; ++c)
        see[c] = (bits_below(e0 - 32 * c) & ~bits_below(b0 - 32 * c)) |
                 (bits_below(e1 - 32 * c) & ~bits_below(b1 - 32 * c));
}

template <int D>
__global__ void __launch_bounds__(384, 1)
fwd_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
           const __grid_constant__ CUtensorMap tmV, const __grid_constant__ CUtensorMap tmO,
           const __grid_constant__ CUtensorMap tmZ, const FwdParams P)
{
    using C = FwdCfg<D>;
    constexpr int NS = C::NS;
    constexpr int STAGE_ARRIVALS = 4;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t sb = (raw + 1023u) & ~1023u;
    uint8_t *sp = smem_raw + (sb - raw);

    const uint32_t bar0 = sb + C::OFF_BAR;
    auto BAR = [&](int i) { return bar0 + 8u * (uint32_t)i; };
    // barrier indices
    constexpr int B_QFULL = 0, B_KFULL = 1, B_KEMPTY = 1 + NS, B_VFULL = 1 + 2 * NS,
                  B_VEMPTY = 1 + 3 * NS, B_SFULL = 1 + 4 * NS, B_PVDONE = B_SFULL + 2, B_SREAD = B_SFULL + 4,
                  B_PFULL = B_SFULL + 6, // [half of the columns, where P is handed over in halves][tile]
                  B_WQFULL = B_SFULL + 10,
                  B_WQFREE = B_WQFULL + 4, B_QEMPTY = B_WQFREE + 4, B_TURN = B_QEMPTY + 1;
    volatile uint32_t *tmem_slot = reinterpret_cast<volatile uint32_t *>(sp + C::OFF_MISC);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(sp + C::OFF_MISC + 4);
    int4 *wq = reinterpret_cast<int4 *>(sp + C::OFF_MISC + 16); // 4 slots
    int32_t *smeta = reinterpret_cast<int32_t *>(sp + C::OFF_META);

    // The warp index read through a shuffle is a value the compiler knows to be the same in every
    // lane, so what depends on it (tensor-memory addresses, barrier addresses) moves to the uniform
    // datapath.  Measured, not reasoned: 3,891 positions, 64 heads of 64, 1,794 -> 1,675 us without it and with.
    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0);
    const int lane = threadIdx.x & 31;
    const int ntile = P.two ? 2 : 1;
    const int n_hb = P.two ? P.Hq / 2 : P.Hq;
    // Work item w of this CTA = (query tile, head block), handed out by a global counter in the
    // order of the schedule (query tiles with the most key tiles first).  The producer warp draws
    // the index, looks the item up and passes it to the other roles through a four-slot queue in shared
    // memory: query tile (negative: no more items), head block, key tiles, SINGLE entries.
    const int heads = ntile; // of a block
    // Every warp of the other roles: item w, query tile -1 at the end, GONE when a wait ran out.  Each of them hands the
    // slot back, the issuing warps too: items without keys take no phase of Q, so nothing else keeps the
    // producer from drawing past a warp that has yet to read the slot.
    constexpr int GONE = -2;
    auto take = [&](int w) {
        const int slot = w & 3;
        if (!mbar_wait_warp(BAR(B_WQFULL + slot), (w >> 2) & 1, abort_flag))
            return make_int4(GONE, 0, 0, 0);
        const int4 e = wq[slot];
        warp_arrive(BAR(B_WQFREE + slot));
        return e;
    };

    if (threadIdx.x == 0) {
        *abort_flag = 0;
        mbar_init(BAR(B_QFULL), 1);
        for (int s = 0; s < NS; ++s) {
            mbar_init(BAR(B_KFULL + s), 1);
            // a stage is free when, for each tile, a commit of the issuing warp and STAGE_ARRIVALS more
            // have arrived: for a key tile the issuing warp's own, for a SINGLE entry one per softmax
            // warp (and the issuing warp, which only has to see the phase pass, in place of the commit)
            mbar_init(BAR(B_KEMPTY + s), ntile * (1 + STAGE_ARRIVALS));
            mbar_init(BAR(B_VFULL + s), 1);
            mbar_init(BAR(B_VEMPTY + s), ntile * (1 + STAGE_ARRIVALS));
        }
        for (int x = 0; x < 2; ++x) {
            mbar_init(BAR(B_SFULL + x), 1);
            mbar_init(BAR(B_PFULL + x), 4);   // one arrival per softmax warp of the tile
            mbar_init(BAR(B_PFULL + 2 + x), 4);
            mbar_init(BAR(B_PVDONE + x), 1);
            mbar_init(BAR(B_SREAD + x), 4);
            for (int i = 0; i < 4; ++i)
                mbar_init(BAR(B_TURN + 4 * x + i), 1);
        }
        for (int i = 0; i < 4; ++i) {
            mbar_init(BAR(B_WQFULL + i), 1);
            mbar_init(BAR(B_WQFREE + i), 5 * ntile); // one arrival per softmax and issuing warp
        }
        // Q may be overwritten once the MMA threads are done with it and every softmax warp has
        // read its rows (or has no use for them).  Items without any key load no Q and have no phase here;
        // for the others no warp arrives for an item before the issuing warps have taken it, or the
        // arrivals of two items could mix.
        mbar_init(BAR(B_QEMPTY), 5 * ntile);
        fence_mbar_init();
    }
    if (warp == 8) {
        tmem_alloc(sb + C::OFF_MISC, 512);
        tmem_relinquish();
    }
    if (P.dO) {
        for (int i = threadIdx.x; i < C::ZERO_ROWS * 8; i += 384)
            reinterpret_cast<uint4 *>(sp + C::OFF_ZERO)[i] = make_uint4(0, 0, 0, 0);
        fence_proxy_async_smem();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    pdl_wait();
    pdl_trigger();

    // Warps 8-11 hand most of their registers to the eight softmax warps.
    if (warp >= 8)
        reg_dec<56>();
    if (warp == 9) {
        // ------------------------------------------------------------ producer
        if (lane == 0) {
            tma_prefetch_desc(&tmQ);
            tma_prefetch_desc(&tmK);
            tma_prefetch_desc(&tmV);
        }
        uint32_t kpos = 0; // position in the K / V ring, running over the items
        bool live = true;
        // Draws item w once the queue slot's last readers (four items ago) are done.  A chain of an atomic and two
        // dependent loads, 2,000 clocks, so it is started ahead of the last key tile of the item before.
        auto draw = [&](int w) {
            int4 e = make_int4(-1, 0, 0, 0);
            if (mbar_wait_warp(BAR(B_WQFREE + (w & 3)), ((w >> 2) & 1) ^ 1, abort_flag) && lane == 0) {
                const int idx = atomicAdd(P.cursor, 1);
                if (idx < P.n_items) {
                    e.x = P.qorder[idx / n_hb];
                    e.y = idx % n_hb;
                    e.z = P.kcount[e.x];
                    e.w = P.scount[e.x];
                }
                wq[w & 3] = e;
                mbar_arrive(BAR(B_WQFULL + (w & 3)));
            }
            return make_int4(__shfl_sync(0xffffffffu, e.x, 0), __shfl_sync(0xffffffffu, e.y, 0),
                             __shfl_sync(0xffffffffu, e.z, 0), __shfl_sync(0xffffffffu, e.w, 0));
        };
        int4 item = draw(0), next = make_int4(-1, 0, 0, 0);
        int qn = 0; // items with keys
        for (int w = 0; live && item.x >= 0; ++w, item = next) {
            const int qt = item.x, h0 = item.y * heads, cnt = item.z, n_single = item.w;
            const int g = h0 / (P.Hq / P.Hkv), row0 = P.q_begin + qt * BM;
            const int2 *klist = P.klist + (size_t)qt * P.n_kt;
            const int window = lane < n_single ? P.sbase[qt * MAX_SINGLE + lane] : 0; // first token of entry `lane`
            auto load = [&](int off, const CUtensorMap *map, int full, uint32_t pos, int start) { // one K or V tile
                const int st = pos % NS;
                if (lane == 0) {
                    mbar_arrive_expect_tx(BAR(full + st), C::TILE_BYTES);
                    for (int pn = 0; pn < C::PANELS; ++pn)
                        tma_load_3d(sb + off + st * C::TILE_BYTES + pn * C::PANEL_BYTES, map, BAR(full + st), pn * 64, g,
                                    start);
                }
                __syncwarp();
            };
            auto stage_free = [&](int empty, uint32_t pos) {
                return mbar_wait_warp(BAR(empty + pos % NS), ((pos / NS) & 1) ^ 1, abort_flag);
            };
            if (cnt + n_single > 0)
                live = mbar_wait_warp(BAR(B_QEMPTY), (qn++ & 1) ^ 1, abort_flag);
            if (cnt + n_single > 0 && live && lane == 0) {
                mbar_arrive_expect_tx(BAR(B_QFULL), ntile * C::TILE_BYTES + n_single * BM);
                for (int x = 0; x < ntile; ++x)
                    for (int pn = 0; pn < C::PANELS; ++pn)
                        tma_load_3d(sb + C::OFF_Q + x * C::TILE_BYTES + pn * C::PANEL_BYTES, &tmQ, BAR(B_QFULL), pn * 64,
                                    h0 + x, row0);
                if (n_single > 0)
                    bulk_load(sb + C::OFF_COL, P.scs + (size_t)qt * MAX_SINGLE * BM, n_single * BM, BAR(B_QFULL));
            }
            __syncwarp();
            // The key tiles of the SINGLE entries go through the same K / V ring first, CHUNK at a time, K of all of them and
            // then V (where a chunk is longer than the ring, the first V beside K); the softmax warps read their
            // rows from shared memory.
            for (int c0 = 0; live && c0 < n_single; c0 += C::CHUNK) {
                const int c1 = min(c0 + C::CHUNK, n_single), beside = C::CHUNK > NS ? min(c1, NS) : c0;
                for (int i = c0; live && i < c1; ++i) {
                    const int start = __shfl_sync(0xffffffffu, window, i);
                    live = stage_free(B_KEMPTY, kpos + i);
                    if (live)
                        load(C::OFF_K, &tmK, B_KFULL, kpos + i, start);
                    if (live && i < beside) {
                        live = stage_free(B_VEMPTY, kpos + i);
                        if (live)
                            load(C::OFF_V, &tmV, B_VFULL, kpos + i, start);
                    }
                }
                for (int i = beside; live && i < c1; ++i) {
                    const int start = __shfl_sync(0xffffffffu, window, i);
                    live = stage_free(B_VEMPTY, kpos + i);
                    if (live)
                        load(C::OFF_V, &tmV, B_VFULL, kpos + i, start);
                }
            }
            // List entries and key metadata are fetched one key tile ahead, so that no global
            // load latency sits between a stage becoming free and its TMA loads.
            auto tile_meta = [&](int2 e, int32_t (&mv)[BN / 32]) {
                const int start = e.x, len = klist_len(e.y);
                const bool need = klist_class(e.y) != TILE_FULL; // FULL tiles skip the predicate
#pragma unroll
                for (int i = 0; i < BN / 32; ++i) {
                    const int t = lane + 32 * i;
                    mv[i] = (need && t < len) ? P.meta[start + t] : META_NONE_K;
                }
            };
            int2 e_cur = cnt > 0 ? klist[0] : make_int2(0, 0);
            int2 e_nxt = cnt > 1 ? klist[1] : e_cur;
            int32_t m_cur[BN / 32], m_nxt[BN / 32];
            if (cnt > 0)
                tile_meta(e_cur, m_cur);
            for (int j = 0; live && j < cnt; ++j) {
                const uint32_t pos = kpos + n_single + j;
                const int st = pos % NS;
                const int start = e_cur.x;
                const int2 e_nn = j + 2 < cnt ? klist[j + 2] : e_nxt;
                if (j + 1 < cnt)
                    tile_meta(e_nxt, m_nxt);
                live = stage_free(B_KEMPTY, pos);
                if (!live)
                    break;
                load(C::OFF_K, &tmK, B_KFULL, pos, start);
                live = stage_free(B_VEMPTY, pos);
                if (!live)
                    break;
#pragma unroll
                for (int i = 0; i < BN / 32; ++i)
                    smeta[st * BN + lane + 32 * i] = m_cur[i];
                __syncwarp();
                load(C::OFF_V, &tmV, B_VFULL, pos, start);
                if (j + 2 == cnt && cnt > NS)
                    next = draw(w + 1);
                e_cur = e_nxt;
                e_nxt = e_nn;
#pragma unroll
                for (int i = 0; i < BN / 32; ++i)
                    m_cur[i] = m_nxt[i];
            }
            if (live && cnt <= NS) // short items: no load waits for it
                next = draw(w + 1);
            kpos += (uint32_t)(n_single + cnt);
            // Hand-over to the backward: the item's rows of the fp32 dQ staging are cleared here, where
            // the memory system is idle (the map ends at the partition's last row).
            if (P.dO && live && lane == 0) {
                for (int x = 0; x < ntile; ++x)
                    for (int pn = 0; pn < D / 32; ++pn)
                        for (int rr = 0; rr < BM && row0 + rr < P.q_end; rr += C::ZERO_ROWS)
                            tma_store_3d(&tmZ, sb + C::OFF_ZERO, pn * 32, h0 + x, qt * BM + rr);
                bulk_commit_group();
            }
        }
        if (lane == 0)
            bulk_wait_group<0>();
    } else if (warp == 8 || warp == 10) {
        // ------------------------------------------------------------ MMA issue
        // One lane of warp 8 issues every MMA of tile A, one of warp 10 those of tile B: the two
        // tiles are independent instruction streams (they only share the K / V stages, which are
        // released once both threads have committed), and two threads issue twice as fast as one.
        const int x = (warp - 8) >> 1;
        // the whole warp walks the items and waits, its elected lane issues (see elect_one)
        const uint32_t lead = elect_one();
        if (x < ntile) {
            constexpr uint32_t IDESC_S = idesc_bf16_f32(128, BN, 0, 0);
            constexpr uint32_t IDESC_O = idesc_bf16_f32(128, D, 0, 1);
            constexpr uint32_t TU = C::TILE_BYTES >> 4, PU = C::PANEL_BYTES >> 4;
            // lower descriptor words in 16-byte units (see desc_lo_sw128)
            const uint32_t q_lo = desc_lo_sw128(sb + C::OFF_Q, 16) + x * TU;
            const uint32_t k_lo = desc_lo_sw128(sb + C::OFF_K, 16);
            const uint32_t v_lo = desc_lo_sw128(sb + C::OFF_V, C::PANEL_BYTES);
            const uint32_t tS = tmem + C::TM_S + x * 128, tO = tmem + C::TM_O + x * D;
            const uint32_t tP = tmem + C::TM_P + x * C::P_STRIDE;
            auto issue_s = [&](int st) {
                const uint32_t kb = k_lo + st * TU;
#pragma unroll
                for (int k = 0; k < D / 16; ++k) {
                    const uint32_t off = (k / 4) * PU + (k % 4) * 2;
                    if (lead) mma_ss_lo(tS, q_lo + off, kb + off, IDESC_S, k > 0);
                }
                if (lead) tc_commit(BAR(B_SFULL + x));
                if (lead) mbar_arrive_n(BAR(B_KEMPTY + st), STAGE_ARRIVALS);
                if (lead) tc_commit(BAR(B_KEMPTY + st));
            };
            auto issue_pv = [&](int st, int half, bool acc) { // 64 keys
                const uint32_t vb = v_lo + st * TU + half * 512, pb = tP + half * 32;
                if (lead) mma_ts_lo(tO, pb, vb, IDESC_O, acc);
#pragma unroll
                for (int k = 1; k < BN / 32; ++k)
                    if (lead) mma_ts_lo(tO, pb + k * 8, vb + k * 128, IDESC_O, 1);
                if (half == 0)
                    return;
                if (lead) tc_commit(BAR(B_PVDONE + x));
                if (lead) mbar_arrive_n(BAR(B_VEMPTY + st), STAGE_ARRIVALS);
                if (lead) tc_commit(BAR(B_VEMPTY + st));
            };
            uint32_t kpos = 0; // position in the K / V ring, running over the items
            uint32_t t = 0;    // key tiles of this thread's tile so far (phases of S, P, PV)
            int qn = 0;        // items with keys so far (phases of Q)
            bool ok = true;
            for (int w = 0; ok; ++w) {
                const int4 item = take(w);
                if (item.x < 0)
                    break;
                const int cnt = item.z, n_single = item.w;
                if (cnt + n_single == 0)
                    continue;
                ok = mbar_wait_warp(BAR(B_QFULL), qn++ & 1, abort_flag);
                if (ok && cnt == 0)
                    if (lead) mbar_arrive(BAR(B_QEMPTY)); // no product reads this Q
                // The SINGLE entries come first in the ring, CHUNK at a time, K and then V.  This warp waits for their phases
                // one by one in that order, and a stage is not refilled before it has: a parity wait is only
                // meaningful on the phase that follows the last one seen.
                for (int c0 = 0; ok && c0 < n_single; c0 += C::CHUNK) {
                    const int c1 = min(c0 + C::CHUNK, n_single);
                    for (int i = c0; ok && i < c1; ++i) {
                        const uint32_t pos = kpos + i;
                        ok = mbar_wait_warp(BAR(B_KFULL + pos % NS), (pos / NS) & 1, abort_flag);
                        if (ok && lead) mbar_arrive(BAR(B_KEMPTY + pos % NS));
                    }
                    for (int i = c0; ok && i < c1; ++i) {
                        const uint32_t pos = kpos + i;
                        ok = mbar_wait_warp(BAR(B_VFULL + pos % NS), (pos / NS) & 1, abort_flag);
                        if (ok && lead) mbar_arrive(BAR(B_VEMPTY + pos % NS));
                    }
                }
                if (ok && cnt > 0) {
                    const uint32_t p0 = kpos + n_single;
                    // S of the previous item's last key tile must be in the softmax registers
                    ok = mbar_wait_warp(BAR(B_KFULL + p0 % NS), (p0 / NS) & 1, abort_flag) &&
                         (t == 0 || mbar_wait_warp(BAR(B_SREAD + x), (t - 1) & 1, abort_flag));
                    if (ok) {
                        tc_fence_after();
                        issue_s(p0 % NS);
                        if (cnt == 1)
                            if (lead) tc_commit(BAR(B_QEMPTY));
                    }
                }
                for (int j = 0; ok && j < cnt; ++j) {
                    const uint32_t pos = kpos + n_single + j, tt = t + j;
                    const int st = pos % NS, ph = (pos / NS) & 1;
                    const int nst = (pos + 1) % NS, nph = ((pos + 1) / NS) & 1;
                    const bool more = j + 1 < cnt;
                    if constexpr (C::P_SEPARATE) {
                        // S(j+1) as soon as the softmax warps hold S(j) in registers
                        if (more) {
                            ok = mbar_wait_warp(BAR(B_KFULL + nst), nph, abort_flag) &&
                                 mbar_wait_warp(BAR(B_SREAD + x), tt & 1, abort_flag);
                            if (!ok)
                                break;
                            tc_fence_after();
                            issue_s(nst);
                            if (j + 2 == cnt)
                                if (lead) tc_commit(BAR(B_QEMPTY)); // the item's last product with Q
                        }
                    }
                    ok = mbar_wait_warp(BAR(B_VFULL + st), ph, abort_flag) &&
                         mbar_wait_warp(BAR(B_PFULL + x), tt & 1, abort_flag);
                    if (!ok)
                        break;
                    tc_fence_after();
                    issue_pv(st, 0, j > 0 || n_single > 0);
                    if constexpr (C::P_HALVES) {
                        ok = mbar_wait_warp(BAR(B_PFULL + 2 + x), tt & 1, abort_flag);
                        if (!ok)
                            break;
                        tc_fence_after();
                    }
                    issue_pv(st, 1, true);
                    if constexpr (!C::P_SEPARATE) {
                        // P overwrote S(j): S(j+1) can only follow the P V product that reads it
                        if (more) {
                            ok = mbar_wait_warp(BAR(B_KFULL + nst), nph, abort_flag);
                            if (!ok)
                                break;
                            issue_s(nst);
                            if (j + 2 == cnt)
                                if (lead) tc_commit(BAR(B_QEMPTY));
                        }
                    }
                }
                kpos += (uint32_t)(n_single + cnt);
                t += (uint32_t)cnt;
            }
        }
    } else if (warp < 4 * ntile) {
        reg_inc<224>();
        // ------------------------------------------------------------ softmax of tile x
        const int x = warp >> 2;
        const int r = threadIdx.x & 127;
        const uint32_t lane_sel = (uint32_t)((warp & 3) * 32) << 16;
        const uint32_t tS = tmem + lane_sel + C::TM_S + x * 128;
        const uint32_t tO = tmem + lane_sel + C::TM_O + x * D;
        const uint32_t tP = tmem + lane_sel + C::TM_P + x * C::P_STRIDE;
        uint32_t kpos = 0; // position in the K / V ring, running over the items
        uint32_t t = 0;    // key tiles of this tile so far (phases of S, P, PV)
        int qn = 0;        // items with keys so far (phases of Q)
        uint32_t n_turn = 0; // items with key tiles so far
        // Item w, and its row's metadata, are fetched ahead of the epilogue of item w - 1 (two dependent reads of
        // global memory and the draw itself, 1,500 to 3,500 clocks per item before the queue carried the item).
        auto fetch = [&](int w, int32_t &meta) {
            const int4 e = take(w);
            const int row = P.q_begin + e.x * BM + r;
            meta = e.x >= 0 && row < P.q_end ? P.meta[row] : META_NONE_Q;
            return e;
        };
        // At head_dim 64 a tile's four warps meet at named barriers, which know no limit.  So once per item they agree,
        // at such a barrier, whether all of them go on to the next: one whose wait ran out would leave the others
        // there for good.
        auto together = [&](bool on) {
            __syncwarp();
            return C::O_STAGED ? bar_and(1 + x, 128, on) : on;
        };
        int32_t mq;
        int4 item = fetch(0, mq);
        bool ok = together(item.x != GONE);
        for (int w = 0; ok && item.x >= 0; ++w) {
        const int qt = item.x, h0 = item.y * heads, cnt = item.z, n_single = item.w;
        const int2 *klist = P.klist + (size_t)qt * P.n_kt;
        const int h = h0 + x;
        const int row0 = P.q_begin + qt * BM, row = row0 + r;
        const bool row_ok = row < P.q_end;
        if (mq == META_NONE_K)
            mq = META_NONE_Q;
        float m = -CUDART_INF_F, l = 0.f;
        if (P.dO && row_ok) { // the epilogue reads this row of dO
            const __nv_bfloat16 *pre = P.dO + ((size_t)row * P.Hq + h) * D;
            asm volatile("prefetch.global.L2 [%0];" ::"l"(pre));
            if (D == 128)
                asm volatile("prefetch.global.L2 [%0];" ::"l"(pre + 64));
        }
        if (n_single > 0) {
            // One allowed key per row and entry, on the CUDA cores from the staged K / V rows, CHUNK entries at a time:
            // their scores, then the softmax over them and the weighted values, whose sums become the starting
            // (m, l, O) of the tile loop.  A row of Q and a row of O are then not held at the same time, and
            // each of the two passes needs K or V only.  Bound by unpacking bf16 (a row's element is two
            // instructions, one of them packed).  (One pass with an online softmax, O in tensor memory at
            // head_dim 128, and a barrier of the tile's warps after every entry: 1,900 clocks per entry at
            // head_dim 64, 3,300 at 128.)
            ok = mbar_wait_warp(BAR(B_QFULL), qn & 1, abort_flag);
            const uint8_t *cols = sp + C::OFF_COL + r;
            float *score = reinterpret_cast<float *>(sp + C::OFF_SCORE + warp * C::WARP_BYTES) + lane;
            auto row_piece = [&](uint32_t off, int rr, int c) { // elements 8c .. 8c + 7 of row rr of a staged tile
                return *reinterpret_cast<const uint4 *>(sp + off + (c >> 3) * C::PANEL_BYTES + rr * 128 +
                                                        (((c & 7) ^ (rr & 7)) << 4));
            };
            auto pair = [](uint32_t w2) { return f2(__uint_as_float(w2 << 16), __uint_as_float(w2 & 0xffff0000u)); };
#pragma unroll 1
            for (int c0 = 0; ok && c0 < (C::ONE_CHUNK ? 1 : n_single); c0 += C::CHUNK) {
                const int c1 = min(c0 + C::CHUNK, n_single);
                const bool again = !C::ONE_CHUNK && c0 > 0;
                float cm = -CUDART_INF_F; // largest of these scores
                {
                    F2 q[D / 2];
#pragma unroll
                    for (int c = 0; c < D / 8; ++c) {
                        const uint4 v = row_piece(C::OFF_Q + x * C::TILE_BYTES, r, c);
                        q[4 * c] = pair(v.x);
                        q[4 * c + 1] = pair(v.y);
                        q[4 * c + 2] = pair(v.z);
                        q[4 * c + 3] = pair(v.w);
                    }
#pragma unroll 1
                    for (int i = c0; ok && i < c1; ++i) {
                        const uint32_t pos = kpos + i;
                        const int st = pos % NS;
                        const int col = cols[i * BM];
                        ok = mbar_wait_warp(BAR(B_KFULL + st), (pos / NS) & 1, abort_flag);
                        if (!ok)
                            break;
                        float s2 = -CUDART_INF_F;
                        if (col != NO_COL && row_ok) {
                            F2 acc[4]; // four chains of dependent adds
#pragma unroll
                            for (int c = 0; c < D / 8; ++c) {
                                const uint4 v = row_piece(C::OFF_K + st * C::TILE_BYTES, col, c);
                                const uint32_t kw[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                                for (int k = 0; k < 4; ++k)
                                    acc[k] = c == 0 ? mul_f2(q[k], pair(kw[k])) : fma_f2(q[4 * c + k], pair(kw[k]), acc[k]);
                            }
                            const float2 a = unf2(add_f2(add_f2(acc[0], acc[1]), add_f2(acc[2], acc[3])));
                            s2 = (a.x + a.y) * P.scale_log2;
                        }
                        score[(i - c0) * 32] = s2;
                        cm = fmaxf(cm, s2);
                        warp_arrive(BAR(B_KEMPTY + st)); // this warp is done with the rows
                    }
                }
                const float m_new = fmaxf(m, cm), neg_m = m_new == -CUDART_INF_F ? 0.f : -m_new;
                const float alpha = fast_exp2(m + neg_m); // of the sums so far; 0 while there are none
                m = m_new;
                l *= alpha;
                F2 o[D / 2];
#pragma unroll
                for (int c = 0; c < D / 32; ++c) {
                    uint32_t ov[32];
                    if (again) {
                        tmem_ld32(tO + c * 32, ov);
                        tmem_wait_ld();
                    }
#pragma unroll
                    for (int i = 0; i < 16; ++i)
                        o[16 * c + i] = again ? mul_f2(f2(__uint_as_float(ov[2 * i]), __uint_as_float(ov[2 * i + 1])), f2(alpha, alpha))
                                               : f2(0.f, 0.f);
                }
#pragma unroll 1
                for (int i = c0; ok && i < c1; ++i) {
                    const uint32_t pos = kpos + i;
                    const int st = pos % NS;
                    const int col = cols[i * BM];
                    const float pr = fast_exp2(score[(i - c0) * 32] + neg_m);
                    ok = mbar_wait_warp(BAR(B_VFULL + st), (pos / NS) & 1, abort_flag);
                    if (!ok)
                        break;
                    if (col != NO_COL && row_ok) {
                        l += pr;
                        const F2 pp = f2(pr, pr);
#pragma unroll
                        for (int c = 0; c < D / 8; ++c) {
                            const uint4 v = row_piece(C::OFF_V + st * C::TILE_BYTES, col, c);
                            o[4 * c] = fma_f2(pp, pair(v.x), o[4 * c]);
                            o[4 * c + 1] = fma_f2(pp, pair(v.y), o[4 * c + 1]);
                            o[4 * c + 2] = fma_f2(pp, pair(v.z), o[4 * c + 2]);
                            o[4 * c + 3] = fma_f2(pp, pair(v.w), o[4 * c + 3]);
                        }
                    }
                    warp_arrive(BAR(B_VEMPTY + st));
                }
#pragma unroll
                for (int c = 0; c < D / 32; ++c) {
                    uint32_t ov[32];
#pragma unroll
                    for (int i = 0; i < 16; ++i) {
                        const float2 v = unf2(o[16 * c + i]);
                        ov[2 * i] = __float_as_uint(v.x);
                        ov[2 * i + 1] = __float_as_uint(v.y);
                    }
                    tmem_st32(tO + c * 32, ov);
                }
                tmem_wait_st(); // ordered before the first P V product by the P hand-over below
            }
            // Q and the entries' columns are done with (the issuing warps need Q for longer anyway)
            warp_arrive(BAR(B_QEMPTY));
        }
        int word_nxt = cnt > 0 ? klist[0].y : 0;
        for (int j = 0; ok && j < cnt; ++j) {
            const uint32_t pos = kpos + n_single + j, tt = t + j;
            const int st = pos % NS, ph = (pos / NS) & 1;
            const int word = word_nxt;
            if (j + 1 < cnt)
                word_nxt = klist[j + 1].y; // used one key tile later
            ok = mbar_wait_warp(BAR(B_SFULL + x), tt & 1, abort_flag);
            if (!ok)
                break;
            tc_fence_after();
            uint32_t xr[4][32];
#pragma unroll
            for (int c = 0; c < 4; ++c)
                tmem_ld32(tS + c * 32, xr[c]);
            tmem_wait_ld();
            // S(j) is in registers: its columns may be overwritten by S(j+1)
            tc_fence_before();
            warp_arrive(BAR(B_SREAD + x));
            if (klist_class(word) != TILE_FULL) {
                ok = mbar_wait_warp(BAR(B_VFULL + st), ph, abort_flag);
                if (!ok)
                    break;
                if (word & KLIST_EVEN) {
                    uint32_t see[4];
                    row_mask(smeta + st * BN, word, mq, see);
#pragma unroll
                    for (int c = 0; c < 4; ++c)
                        if (!__all_sync(0xffffffffu, see[c] == ~0u)) {
#pragma unroll
                            for (int i = 0; i < 32; ++i)
                                if (!(see[c] >> i & 1u)) xr[c][i] = 0xff800000u;
                        }
                } else {
                    const int4 *mk4 = reinterpret_cast<const int4 *>(smeta + st * BN);
#pragma unroll
                    for (int c = 0; c < 4; ++c)
#pragma unroll
                        for (int i = 0; i < 32; i += 4) {
                            const int4 mk = mk4[(c * 32 + i) >> 2];
                            if (!allowed_packed(mq, mk.x)) xr[c][i + 0] = 0xff800000u;
                            if (!allowed_packed(mq, mk.y)) xr[c][i + 1] = 0xff800000u;
                            if (!allowed_packed(mq, mk.z)) xr[c][i + 2] = 0xff800000u;
                            if (!allowed_packed(mq, mk.w)) xr[c][i + 3] = 0xff800000u;
                        }
                }
            }
            float mx4[4]; // four independent chains of three-input maxima
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                mx4[c] = -CUDART_INF_F;
#pragma unroll
                for (int i = 0; i < 32; i += 2)
                    mx4[c] = max3(mx4[c], __uint_as_float(xr[c][i]), __uint_as_float(xr[c][i + 1]));
            }
            float mx = fmaxf(fmaxf(mx4[0], mx4[1]), fmaxf(mx4[2], mx4[3]));
            mx *= P.scale_log2; // scale > 0, so the max commutes with the scaling
            const float m_new = fmaxf(m, mx);
            if (j == 0 && n_single == 0) {
                m = m_new;
            } else {
                // P V of the previous key tile must be done before O or P are touched
                if (j > 0) {
                    ok = mbar_wait_warp(BAR(B_PVDONE + x), (tt - 1) & 1, abort_flag);
                    if (!ok)
                        break;
                    tc_fence_after();
                }
                // Rescale the running output only when the maximum grew by more than 2^8; until
                // then the stale maximum keeps every probability below 256.
                const bool grow = m_new > m + 8.f;
                if (__any_sync(0xffffffffu, grow)) {
                    const float alpha = (m_new == -CUDART_INF_F) ? 1.f : fast_exp2(m - m_new);
                    l *= alpha;
                    m = m_new;
#pragma unroll
                    for (int c = 0; c < D / 32; ++c) {
                        uint32_t o[32];
                        tmem_ld32(tO + c * 32, o);
                        tmem_wait_ld();
#pragma unroll
                        for (int i = 0; i < 32; ++i)
                            o[i] = __float_as_uint(__uint_as_float(o[i]) * alpha);
                        tmem_st32(tO + c * 32, o);
                    }
                    tmem_wait_st();
                }
            }
            // Left alone the two tiles' warps of a scheduler fall into step: both do exponentials at once and both wait
            // at once, with the exp2 unit idle for half of the time.  It is enough that tile B's first
            // exponentials of an item start behind tile A's: the distance lasts, and a hand-over per tile costs more
            // than it gives (one set of inputs again and again, 3,891 positions, 64 heads of 64: 1,660 us in step,
            // 1,547 apart, 1,737 with a turn per tile; 2,048 positions, 32 heads of 128: 346 with turns, 336 so).
            // Tile A waits for tile B's first turn of the item before, which is long past, so that no warp is ever
            // two phases ahead of another's wait.
            if (P.two && j == 0 && (x == 1 || n_turn > 0)) {
                ok = mbar_wait_warp(BAR(B_TURN + 4 * x + (warp & 3)), (x == 1 ? n_turn : n_turn - 1) & 1, abort_flag);
                if (!ok)
                    break;
            }
            const float neg_m = (m == -CUDART_INF_F) ? 0.f : -m;
            // A quarter of the exponentials goes to the FMA pipe: the last two columns of every eight, so
            // that arguments, exponentials and sums all stay packed pairs (every fourth column: 190 more
            // instructions per tile, 3,891 positions, 64 heads of 64: 1,815 against 1,633 us; three
            // eighths 1,790).  The cubic is 7e-5 off at argument 0, so which columns take it decides how
            // exact the first rows of a sequence are, whose few keys stand in the first columns: depth-0 rows of
            // up to six keys that begin a tile are exact to fp32 rounding.
            const F2 scale2 = f2(P.scale_log2, P.scale_log2), nm2 = f2(neg_m, neg_m);
            F2 sum2[2] = {f2(0.f, 0.f), f2(0.f, 0.f)};
#pragma unroll
            for (int hf = 0; hf < 2; ++hf) {
                uint32_t pk[32];
#pragma unroll
                for (int i = 0; i < 32; ++i) { // columns 64 hf + 2i, + 1
                    const int c = 2 * hf + (i >> 4), e = 2 * (i & 15);
                    F2 v = fma_f2(f2(__uint_as_float(xr[c][e]), __uint_as_float(xr[c][e + 1])), scale2, nm2);
                    float2 w = unf2(v);
                    v = (i & 3) == 3 ? exp2_fma2(v) : f2(fast_exp2(w.x), fast_exp2(w.y));
                    sum2[i & 1] = add_f2(sum2[i & 1], v);
                    w = unf2(v);
                    pk[i] = pack_bf16x2(w.x, w.y);
                }
                tmem_st32(tP + hf * 32, pk);
                if (C::P_HALVES && hf == 0) {
                    tmem_wait_st();
                    tc_fence_before();
                    warp_arrive(BAR(B_PFULL + x));
                }
            }
            if (P.two && lane == 0 && j == 0)
                mbar_arrive(BAR(B_TURN + 4 * (x ^ 1) + (warp & 3))); // the other tile's turn
            const float2 s0 = unf2(sum2[0]), s1 = unf2(sum2[1]);
            l += (s0.x + s0.y) + (s1.x + s1.y);
            tmem_wait_st();
            tc_fence_before();
            warp_arrive(BAR(B_PFULL + (C::P_HALVES ? 2 : 0) + x));
        }
        if (ok && cnt > 0 && n_single == 0 && lane == 0)
            mbar_arrive(BAR(B_QEMPTY)); // this warp reads no row of Q; not ahead of the issuing warp, see Q's phases
        __syncwarp();
        int32_t mq_next = META_NONE_Q;
        const int4 item_next = fetch(w + 1, mq_next);
        // ---- epilogue: normalise, store O and LSE
        // Delta of the row needs the row of dO: requested here, ahead of the wait for the last P V product (the rows
        // were sent towards L2 when the item began).  The warp's 32 rows are read together, D / 2 bytes or more of a
        // row by neighbouring lanes, and dealt out through shared memory: a lane that reads (or writes) its own
        // row makes every access of the warp 32 pieces of 16 bytes, and at head_dim 128 O left that way too.
        // (Forward of a step, 4,096 positions, 64 heads of 64: 1,722 -> 1,701 us; 2,048 positions, 32 heads of
        // 128: 2 to 5 per cent.)
        constexpr int ROW_PIECES = C::O_STAGED ? 8 : 4; // 16-byte pieces of a row that are taken together
        const int wrow = row0 + (warp & 3) * 32;
        auto own_piece = [&](int k, int &rr, int &c) { // piece k of this lane: row of the warp, piece of the row
            rr = (k * 32 + lane) / ROW_PIECES;
            c = (k * 32 + lane) % ROW_PIECES;
        };
        uint4 dov[D / 8];
        if (P.dO && cnt + n_single > 0) {
#pragma unroll
            for (int k = 0; k < D / 8; ++k) {
                int rr, c;
                own_piece(k % ROW_PIECES, rr, c);
                const uint4 *src = reinterpret_cast<const uint4 *>(P.dO + ((size_t)(wrow + rr) * P.Hq + h) * D);
                dov[k] = wrow + rr < P.q_end ? __ldg(src + k / ROW_PIECES * ROW_PIECES + c) : make_uint4(0, 0, 0, 0);
            }
        } else { // never read, but see the compiler keep the registers through the item without it
#pragma unroll
            for (int k = 0; k < D / 8; ++k)
                dov[k] = make_uint4(0, 0, 0, 0);
        }
        // rows of the padded partition are numbered from its first row
        const size_t hand = (size_t)h * P.q_pad + (size_t)row_slot(qt * BM + r);
        if (P.dO && x == 0 && h0 == 0)
            P.mqp[row_slot(qt * BM + r)] = mq;
        if (cnt == 0 && n_single == 0) {
            if (row_ok) {
                uint4 z = make_uint4(0, 0, 0, 0);
                uint4 *dst = reinterpret_cast<uint4 *>(P.O + ((size_t)row * P.Hq + h) * D);
                for (int i = 0; i < D / 8; ++i)
                    dst[i] = z;
                P.LSE[(size_t)h * P.T + row] = -CUDART_INF_F;
            }
            if (P.dO) {
                P.nl2[hand] = -CUDART_INF_F;
                P.nd[hand] = 0.f;
            }
            ok = together(item_next.x != GONE);
        } else if ([&] {
                       const bool fin = ok && item_next.x != GONE &&
                                        (cnt == 0 || mbar_wait_warp(BAR(B_PVDONE + x), (t + cnt - 1) & 1, abort_flag));
                       // the staging tile of the previous item must have left shared memory
                       if (C::O_STAGED && r == 0)
                           bulk_wait_group_read<0>();
                       return together(fin);
                   }()) {
            tc_fence_after();
            // A row with no key in any of its tiles has m = -inf, but not l = 0: the cubic never goes below
            // 2^-126.  Its O is zero all the same.
            const bool seen = m > -CUDART_INF_F && l > 0.f;
            const float inv = seen ? 1.f / l : 0.f;
            float delta = 0.f;
            auto dot8 = [&](const uint4 w, const uint32_t *o8) {
                const uint32_t ww[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    delta = fmaf(__uint_as_float(ww[k] << 16), __uint_as_float(o8[2 * k]), delta);
                    delta = fmaf(__uint_as_float(ww[k] & 0xffff0000u), __uint_as_float(o8[2 * k + 1]), delta);
                }
            };
            if constexpr (C::O_STAGED) {
                // rows -> swizzled bf16 tile in shared memory -> one tiled store; the map ends at
                // the partition's last row, so rows past it are not written
                uint8_t *orow = sp + C::OFF_OST + x * C::TILE_BYTES + r * 128;
                if (P.dO) { // the warp's rows of dO in the places that its rows of O will take
#pragma unroll
                    for (int k = 0; k < D / 8; ++k) {
                        int rr, c;
                        own_piece(k, rr, c);
                        *reinterpret_cast<uint4 *>(orow + (rr - lane) * 128 + ((c ^ (rr & 7)) << 4)) = dov[k];
                    }
                    __syncwarp();
                }
#pragma unroll
                for (int c = 0; c < D / 32; ++c) {
                    uint32_t o[32];
                    tmem_ld32(tO + c * 32, o);
                    tmem_wait_ld();
#pragma unroll
                    for (int i = 0; i < 32; i += 8) {
                        if (P.dO)
                            dot8(*reinterpret_cast<const uint4 *>(orow + (((c * 4 + (i >> 3)) ^ (r & 7)) << 4)), o + i);
                        uint4 v;
                        v.x = pack_bf16x2(__uint_as_float(o[i + 0]) * inv, __uint_as_float(o[i + 1]) * inv);
                        v.y = pack_bf16x2(__uint_as_float(o[i + 2]) * inv, __uint_as_float(o[i + 3]) * inv);
                        v.z = pack_bf16x2(__uint_as_float(o[i + 4]) * inv, __uint_as_float(o[i + 5]) * inv);
                        v.w = pack_bf16x2(__uint_as_float(o[i + 6]) * inv, __uint_as_float(o[i + 7]) * inv);
                        const int j = c * 4 + (i >> 3); // 16-byte chunk of the row
                        *reinterpret_cast<uint4 *>(orow + ((j ^ (r & 7)) << 4)) = v;
                    }
                }
                fence_proxy_async_smem();
                asm volatile("bar.sync %0, 128;" ::"r"(1 + x) : "memory");
                if (r == 0) {
                    tma_store_3d(&tmO, sb + C::OFF_OST + x * C::TILE_BYTES, 0, h, row0);
                    bulk_commit_group();
                }
            } else {
                uint8_t *stage = sp + C::OFF_SCORE + warp * C::WARP_BYTES; // 32 rows of 64 bytes
                auto slot = [&](int rr, int c) {
                    return reinterpret_cast<uint4 *>(stage + rr * 64 + ((c ^ ((rr >> 1) & 3)) << 4));
                };
#pragma unroll
                for (int q4 = 0; q4 < D / 32; ++q4) { // 32 columns
                    uint32_t o[32];
                    tmem_ld32(tO + q4 * 32, o);
                    if (P.dO) {
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            int rr, c;
                            own_piece(k, rr, c);
                            *slot(rr, c) = dov[4 * q4 + k];
                        }
                        __syncwarp();
                    }
                    tmem_wait_ld();
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        const uint32_t *o8 = o + 8 * c;
                        if (P.dO)
                            dot8(*slot(lane, c), o8);
                        uint4 v;
                        v.x = pack_bf16x2(__uint_as_float(o8[0]) * inv, __uint_as_float(o8[1]) * inv);
                        v.y = pack_bf16x2(__uint_as_float(o8[2]) * inv, __uint_as_float(o8[3]) * inv);
                        v.z = pack_bf16x2(__uint_as_float(o8[4]) * inv, __uint_as_float(o8[5]) * inv);
                        v.w = pack_bf16x2(__uint_as_float(o8[6]) * inv, __uint_as_float(o8[7]) * inv);
                        *slot(lane, c) = v;
                    }
                    __syncwarp();
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        int rr, c;
                        own_piece(k, rr, c);
                        if (wrow + rr < P.q_end)
                            reinterpret_cast<uint4 *>(P.O + ((size_t)(wrow + rr) * P.Hq + h) * D)[4 * q4 + c] = *slot(rr, c);
                    }
                    __syncwarp(); // before the next columns take the places
                }
            }
            const float lse2 = seen ? m + log2f(l) : -CUDART_INF_F;
            if (row_ok)
                P.LSE[(size_t)h * P.T + row] = lse2 * 0.6931471805599453f;
            if (P.dO) { // the accumulator is not normalised: Delta = inv * <dO, O_acc>
                P.nl2[hand] = (row_ok && seen) ? -lse2 : -CUDART_INF_F;
                P.nd[hand] = row_ok ? -delta * inv : 0.f;
            }
        } else {
            ok = false; // a wait ran out
        }
        kpos += (uint32_t)(n_single + cnt);
        t += (uint32_t)cnt;
        qn += cnt + n_single > 0;
        n_turn += cnt > 0;
        item = item_next;
        mq = mq_next;
        } // items
    }

    // ------------------------------------------------------------ teardown
    if (C::O_STAGED && warp < 8 && (threadIdx.x & 127) == 0)
        bulk_wait_group<0>(); // this thread's tile stores are complete
    tc_fence_before();
    __syncthreads();
    if (*abort_flag) {
        if (threadIdx.x == 0)
            atomicCAS(P.status, 0, PEAGLE_ERR_TIMEOUT);
        // give copies and MMAs that may still be in flight time to land before the CTA's
        // shared and tensor memory are released
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

static int make_map(EncodeTiledFn enc, CUtensorMap *m, const void *base, int D, int H, int T)
{
    cuuint64_t dims[3] = {(cuuint64_t)D, (cuuint64_t)H, (cuuint64_t)T};
    cuuint64_t strides[2] = {(cuuint64_t)D * 2, (cuuint64_t)H * D * 2};
    cuuint32_t box[3] = {64, 1, 128};
    cuuint32_t estr[3] = {1, 1, 1};
    CUresult r = enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void *>(base), dims, strides,
                     box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                     CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? 0 : -1;
}

int make_bf16_map(EncodeTiledFn enc, CUtensorMap *m, const void *base, int D, int H, int T)
{
    return make_map(enc, m, base, D, H, T);
}

// Tensor map of fp32 sums [rows][H][D]: 32 columns x box_rows rows, for tiled reduce-adds and stores.
int make_f32_map(EncodeTiledFn enc, CUtensorMap *m, float *base, int D, int H, int rows, int box_rows)
{
    cuuint64_t dims[3] = {(cuuint64_t)D, (cuuint64_t)H, (cuuint64_t)rows};
    cuuint64_t strides[2] = {(cuuint64_t)D * 4, (cuuint64_t)H * D * 4};
    cuuint32_t box[3] = {32, 1, (cuuint32_t)box_rows};
    cuuint32_t estr[3] = {1, 1, 1};
    return enc(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, base, dims, strides, box, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS
               ? 0
               : -1;
}

template <int D>
static int launch_fwd_t(const Plan &p, const FwdArgs &a, EncodeTiledFn enc, int n_sm,
                        cudaStream_t s, cudaEvent_t ev0, cudaEvent_t ev1)
{
    // the O map ends at the partition's last row: a tiled store does not write past it
    CUtensorMap tmQ, tmK, tmV, tmO;
    if (make_map(enc, &tmQ, a.Q, D, a.Hq, p.T) || make_map(enc, &tmK, a.K, D, a.Hkv, p.T) ||
        make_map(enc, &tmV, a.V, D, a.Hkv, p.T) || make_map(enc, &tmO, a.O, D, a.Hq, p.q_end))
        return PEAGLE_ERR_CUDA;
    CUtensorMap tmZ = tmO;
    if (a.dO && make_f32_map(enc, &tmZ, a.dq_acc, D, a.Hq, p.q_end - p.q_begin, FwdCfg<D>::ZERO_ROWS))
        return PEAGLE_ERR_CUDA;
    FwdParams P;
    P.klist = p.klist;
    P.kcount = p.kcount;
    P.qorder = p.qorder;
    P.meta = p.meta;
    P.status = p.status;
    P.cursor = p.counters + CNT_FWD_CURSOR;
    P.n_kt = p.n_kt;
    P.q_begin = p.q_begin;
    P.q_end = p.q_end;
    P.T = p.T;
    P.O = static_cast<__nv_bfloat16 *>(a.O);
    P.LSE = a.LSE;
    P.Hq = a.Hq;
    P.Hkv = a.Hkv;
    P.two = ((a.Hq / a.Hkv) % 2 == 0) ? 1 : 0;
    P.scale_log2 = a.scale * 1.4426950408889634f;
    P.scount = p.scount;
    P.scs = p.scs;
    P.sbase = p.sbase;
    P.dO = static_cast<const __nv_bfloat16 *>(a.dO);
    P.nl2 = a.nl2;
    P.nd = a.nd;
    P.mqp = a.mqp;
    P.q_pad = p.n_qt * BM;
    // the attribute belongs to the current device's copy of the function: set before every launch
    // (host time only), so that a process that drives several GPUs gets it on each of them
    if (cudaFuncSetAttribute(fwd_kernel<D>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             FwdCfg<D>::SMEM_BYTES) != cudaSuccess)
        return PEAGLE_ERR_CUDA;
    const int n_hb = P.two ? a.Hq / 2 : a.Hq;
    P.n_items = p.n_qt * n_hb;
    if (ev0)
        cudaEventRecord(ev0, s);
    launch_dependent(fwd_kernel<D>, std::min(P.n_items, n_sm), 384, FwdCfg<D>::SMEM_BYTES, s, tmQ, tmK, tmV, tmO, tmZ, P);
    if (ev1)
        cudaEventRecord(ev1, s);
    return 1;
}

int launch_fwd(const Plan &p, const FwdArgs &a, EncodeTiledFn enc, int n_sm, cudaStream_t s,
               cudaEvent_t ev0, cudaEvent_t ev1)
{
    if (p.n_qt == 0)
        return 0;
    return a.D == 64 ? launch_fwd_t<64>(p, a, enc, n_sm, s, ev0, ev1)
                     : launch_fwd_t<128>(p, a, enc, n_sm, s, ev0, ev1);
}

} // namespace peagle
