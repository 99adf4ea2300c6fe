// Shared by the backward kernels: launch parameters and the walk over a CTA's work items.
#pragma once
#include "peagle_internal.h"
#include "sm100_ptx.cuh"

namespace peagle {

struct BwdParams {
    const int2 *ktile;
    const int2 *bitems;
    const int *counters;
    int *cursor; // device counter, zero at launch: next (work item, KV head) index to hand out
    const int32_t *meta;
    int *status;
    int n_qt, n_kt, q_begin;
    const float *nl2, *nd; // [Hq][q_pad] -LSE*log2(e) and -Delta, padded rows (-inf, 0)
    const int32_t *mqp;    // [q_pad] packed metadata of the partition's rows
    int q_pad;             // n_qt * BM
    // The sums' addresses are in the tensor maps and no kernel reads these.  They stay because of the
    // compiler: without them it spills 20 bytes more in bwd64_kernel, in the wrong place (4,096 positions, 64
    // heads of 64: 3.10 -> 3.31 ms).
    float *dq_acc;         // [q_len][Hq][D]
    float *dK_acc, *dV_acc;
    int Hq, Hkv;
    float scale, scale_log2;
};

// Work items are handed out dynamically: the producer warp takes the next index from a global cursor
// and publishes what the other roles need of the item in a four-slot queue in shared memory.  A CTA that
// falls behind therefore takes fewer items, and the CTAs running at any time work on a contiguous window
// of the chunk-major item list (their shared Q / dO rows and dQ staging rows stay in L2), instead of
// drifting apart as with a static round-robin.
// Slot w & 3 has the CTA's item w.  The producer writes it with the last step of item w - 1, when every
// role has taken item w - 4, also where items are single steps:
//   bwd64_kernel   K of item w - 1 was requested before, so the K stage of item w - 3 was free
//                  (B_KVEMPTY): dQ of its last step was complete, which follows that step's dS^T
//                  (compute warps, S^T and dP^T issuers) and the drain's read of dQ of the step before
//                  (B_DQEMPTY), in item w - 4 or later.  The drain may still be sending dK / dV of item
//                  w - 4, from its registers.
//   bwd128_kernel  K of item w - 1 was requested before, so K of item w - 2 was free (B_KEMPTY): dQ of its
//                  last step was complete, behind that step's dP^T, which followed the drain's read of dQ
//                  of the step before, in item w - 3 or later.  The drain is therefore through with item
//                  w - 4 altogether, and may read its slot again at the item's end.
// One index = (work item of K0, KV head, part of the group's heads): one key tile against the query
// tiles of a chunk, one head after the other; every (query tile, head) is a step.
struct BwdItem {
    int k_start, k_len; // key tile
    int qt0;            // first query tile of the chunk
    unsigned mask;      // bit b: query tile qt0 + b takes part; bit 8 + b: its tile is FULL
    int h0, nh;         // heads h0 .. h0 + nh - 1
    int g;              // KV head; negative: no more items
    int steps;
};
constexpr int BWD_QUEUE_BYTES = 4 * (int)sizeof(BwdItem);

// How finely the work items of K0 are cut, from the steps a CTA gets on average: with whole groups a
// small problem keeps few SMs busy for up to BWD_CQ x group steps, but every item costs a K / V load,
// a start of the pipeline and two fp32 tiles added to dK / dV (about two steps in all).  The heads of a
// group are dealt out in parts of a twelfth of a CTA's steps (times up to BWD_CQ query tiles per
// item), so a CTA draws three items or more; with less than three steps per CTA every step is an
// item of its own.  Measured, backward kernel: 512 tokens, 4 heads of 64 (one KV head) 39 -> 15 us;
// 3,128 tokens, 32 heads of 128 99 -> 76 us; divisors from 8 to 16 within 2 per cent of each other,
// 24 up to 12 per cent slower between 5,600 and 11,200 tokens.
struct BwdSplit {
    int parts, nh; // parts of a KV group, heads per part
    int count[BWD_CQ]; // work items of K0 with 1 .. BWD_CQ query tiles
    int cap;           // places for the items of a size
    int tiles;     // 1: whole chunks, BWD_CQ: one query tile per item
    int total;     // indexes to draw
};
__device__ __forceinline__ BwdSplit bwd_split(const BwdParams &P)
{
    const int G = P.Hq / P.Hkv;
    BwdSplit s;
    int items = 0;
    long long steps = 0;
#pragma unroll
    for (int i = 0; i < BWD_CQ; ++i) {
        s.count[i] = P.counters[CNT_ITEMS + i];
        items += s.count[i];
        steps += (long long)(i + 1) * s.count[i] * P.Hq;
    }
    s.cap = (P.n_qt + BWD_CQ - 1) / BWD_CQ * P.n_kt;
    const int avg = (int)min(steps / gridDim.x, (long long)(1 << 20));
    s.nh = min(G, max(1, avg / 12));
    s.parts = (G + s.nh - 1) / s.nh;
    s.nh = (G + s.parts - 1) / s.parts;
    s.parts = (G + s.nh - 1) / s.nh;
    s.tiles = avg < 3 ? BWD_CQ : 1;
    s.total = items * P.Hkv * s.parts * s.tiles;
    return s;
}

// Producer warp (convergent): draws the next item and publishes it as item w.
__device__ __forceinline__ bool bwd_draw(const BwdParams &P, const BwdSplit &sp, uint8_t *queue, uint32_t queue_bar,
                                         int w, int lane, BwdItem &out)
{
    const int G = P.Hq / P.Hkv;
    out.g = -1;
    while (true) {
        int v = 0;
        if (lane == 0)
            v = atomicAdd(P.cursor, 1);
        v = __shfl_sync(0xffffffffu, v, 0);
        if (v >= sp.total)
            break;
        const int tile = v % sp.tiles, rest = v / sp.tiles;
        const int part = rest % sp.parts, ig = rest / sp.parts;
        int at = ig / P.Hkv, base = 0; // the items with most query tiles come first
#pragma unroll
        for (int i = BWD_CQ - 1; i >= 0; --i) {
            if (at >= 0 && at < sp.count[i]) {
                base = i * sp.cap + at;
                at = -1;
            } else if (at >= 0) {
                at -= sp.count[i];
            }
        }
        const int2 item = P.bitems[base];
        unsigned mask = item_mask(item);
        if (sp.tiles > 1)
            mask &= 0x101u << tile;
        if ((mask & 0xffu) == 0)
            continue; // this query tile of the chunk is skipped by the key tile
        const int2 kt = P.ktile[item.x];
        out.g = ig % P.Hkv;
        out.k_start = kt.x;
        out.k_len = kt.y;
        out.qt0 = item_chunk(item) * BWD_CQ;
        out.mask = mask;
        out.h0 = out.g * G + part * sp.nh;
        out.nh = min(sp.nh, G - part * sp.nh);
        out.steps = __popc(mask & 0xffu) * out.nh;
        break;
    }
    if (lane == 0) {
        *reinterpret_cast<BwdItem *>(queue + (w & 3) * sizeof(BwdItem)) = out;
        sm100::mbar_arrive(queue_bar + 8u * (w & 3));
    }
    return out.g >= 0;
}
// The other roles: item w, or false at the end (or when a wait ran out).
__device__ __forceinline__ bool bwd_take(uint8_t *queue, uint32_t queue_bar, int w, volatile int *abort, BwdItem &out)
{
    const bool ok = sm100::mbar_wait(queue_bar + 8u * (w & 3), (w >> 2) & 1, abort);
    if (!__all_sync(0xffffffffu, ok))
        return false;
    out = *reinterpret_cast<const BwdItem *>(queue + (w & 3) * sizeof(BwdItem));
    return out.g >= 0;
}

} // namespace peagle
