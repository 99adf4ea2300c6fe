// K0: implicit mask evaluator, tile classifier and scheduler.
//
// The parallel-prediction mask (paper Section 3 / 3.2) is a function of per-token metadata only,
// so it is evaluated from a packed word per token (anchor << 8 | depth) and never stored.  For
// one call (a query partition and the key ranges it may see) two kernels
//   k0_tiles  pack and validate the metadata, lay out the key tiles of the visible ranges, summarise
//             every query tile and key tile (min/max anchor and depth of its first run of equal depth
//             and of the rest: in a depth-major layout a tile on the border of two depths holds the
//             last anchors of one and the first of the next, and one summary would decide nothing);
//   k0_plan   one block per query tile: classify its (query tile, key tile) pairs as SKIP / PARTIAL /
//             FULL -- from the summaries where they decide, else exactly, by the keys each query row
//             allows -- and compact the non-skipped ones into its key list; the last block of a chunk
//             of query tiles cuts the backward's (key tile, chunk) work items, the last block of all
//             orders the query tiles.
// Everything runs on the caller's stream; nothing returns to the host.  The work is integer and small:
// what it costs is launches and the latency of dependent steps, hence two kernels and not one per
// step (eight kernels before: 24 us for 512 tokens, 47 us for 32,768, 95 us for the COD example).
#include <cuda_bf16.h>
#include <math_constants.h>

#include "peagle_internal.h"
#include "sm100_ptx.cuh"

namespace peagle {

__device__ __forceinline__ void set_status(int *status, int err)
{
    atomicCAS(status, 0, err);
}

__device__ __forceinline__ int pack_meta(int a, int d, int K)
{
    return a < 0 || a >= (1 << 23) || d < 0 || d >= K ? META_NONE_K : (a << 8) | d;
}

// Beside the length of the first run in ksplit, for each run: it is in ascending order; its anchors follow one
// another; its keys are all depth-0 tokens; all deeper ones.
constexpr int KRUN0_SORTED = 1 << 8, KRUN1_SORTED = 1 << 9, KRUN0_EVEN = 1 << 10, KRUN1_EVEN = 1 << 11;
constexpr int KRUN0_REAL = 1 << 12, KRUN1_REAL = 1 << 13, KRUN0_CHAIN = 1 << 14, KRUN1_CHAIN = 1 << 15;

// ---- 1. pack metadata, lay out and summarise tiles ---------------------------------------------
// Block b packs tokens 128 b .. of the sequence and summarises tile b (query tiles first).
__global__ void __launch_bounds__(128) k0_tiles(Plan p, const int32_t *__restrict__ anchor,
                                                const int32_t *__restrict__ depth, int K, int seq_begin,
                                                int seq_end, RangeList ranges)
{
    sm100::pdl_wait();
    sm100::pdl_trigger();
    const int tile = blockIdx.x;
    const int t = seq_begin + tile * 128 + threadIdx.x;
    if (t < seq_end) {
        const int m = pack_meta(anchor[t], depth[t], K);
        if (m == META_NONE_K)
            set_status(p.status, PEAGLE_ERR_BAD_META);
        p.meta[t] = m;
    }
    if (tile == 0 && threadIdx.x < PLAN_COUNTERS)
        p.counters[threadIdx.x] = 0;
    if (threadIdx.x == 0 && tile * BWD_CQ < p.n_qt)
        p.cdone[tile] = 0;
    if (tile >= p.n_qt + p.n_kt)
        return;
    int b, e;
    int4 *out;
    if (tile < p.n_qt) {
        b = p.q_begin + tile * BM;
        e = min(b + BM, p.q_end);
        out = p.qsum + 2 * tile;
    } else {
        int kt = tile - p.n_qt, i = 0; // key tiles are numbered through the visible ranges
        while (kt >= (ranges.end[i] - ranges.begin[i] + BN - 1) / BN)
            kt -= (ranges.end[i] - ranges.begin[i] + BN - 1) / BN, ++i;
        b = ranges.begin[i] + kt * BN;
        e = min(b + BN, ranges.end[i]);
        out = p.ksum + 2 * (tile - p.n_qt);
        if (threadIdx.x == 0)
            p.ktile[tile - p.n_qt] = make_int2(b, e - b);
    }
    const bool in_tile = b + (int)threadIdx.x < e;
    const int m = in_tile ? pack_meta(anchor[b + threadIdx.x], depth[b + threadIdx.x], K) : META_NONE_K;
    const int dn = m == META_NONE_K ? -1 : m & 0xff; // depth -1: no token, or not a valid one
    __shared__ int split, not_so, word[128];
    __shared__ int4 part[2][4];
    word[threadIdx.x] = m;
    if (threadIdx.x == 0) {
        split = e - b;
        not_so = 0;
    }
    __syncthreads();
    const int first_depth = word[0] == META_NONE_K ? -1 : word[0] & 0xff;
    if (in_tile && dn != first_depth)
        atomicMin(&split, (int)threadIdx.x);
    __syncthreads();
#pragma unroll
    for (int run = 0; run < 2; ++run) {
        const bool in = dn >= 0 && ((int)threadIdx.x < split) == (run == 0);
        const int a0 = __reduce_min_sync(0xffffffffu, in ? m >> 8 : INT_MAX);
        const int a1 = __reduce_max_sync(0xffffffffu, in ? m >> 8 : -1);
        const int d0 = __reduce_min_sync(0xffffffffu, in ? dn : INT_MAX);
        const int d1 = __reduce_max_sync(0xffffffffu, in ? dn : -1);
        if ((threadIdx.x & 31) == 0)
            part[run][threadIdx.x >> 5] = make_int4(a0, a1, d0, d1);
    }
    // runs in ascending order of their packed words can be searched instead of read through
    const int nx = threadIdx.x + 1;
    if (nx < e - b && nx != split && word[nx] != word[threadIdx.x] + 256)
        atomicOr(&not_so, (nx < split ? KRUN0_EVEN : KRUN1_EVEN) |
                              (word[threadIdx.x] <= word[nx] ? 0 : nx < split ? KRUN0_SORTED : KRUN1_SORTED));
    __syncthreads();
    if (threadIdx.x < 2) {
        int4 r = part[threadIdx.x][0];
        for (int w = 1; w < 4; ++w) {
            const int4 o = part[threadIdx.x][w];
            r.x = min(r.x, o.x);
            r.y = max(r.y, o.y);
            r.z = min(r.z, o.z);
            r.w = max(r.w, o.w);
        }
        out[threadIdx.x] = r;
        int kinds = (r.w == 0 ? KRUN0_REAL : 0) | (r.z >= 1 ? KRUN0_CHAIN : 0);
        kinds |= __shfl_down_sync(3u, kinds, 1) << 1; // the second run's bits follow the first's
        if (threadIdx.x == 0 && tile >= p.n_qt)
            p.ksplit[tile - p.n_qt] =
                split | kinds | ((KRUN0_SORTED | KRUN1_SORTED | KRUN0_EVEN | KRUN1_EVEN) & ~not_so);
    }
}

// ---- 2. the plan -----------------------------------------------------------------------------
constexpr int PLAN_THREADS = 512;
constexpr int PLAN_GROUPS = PLAN_THREADS / BM; // pairs classified exactly at a time
constexpr int PAIR_CACHE = 256;                // undecided pairs of a query tile kept in shared memory
constexpr int RAW_SINGLE = 2 * MAX_SINGLE;     // one-key-per-row tiles kept before neighbours are joined
constexpr int SORT_BUCKETS = 4096;

// Class of a run of query rows and a run of keys from their summaries (min anchor, max anchor, min
// depth, max depth; max anchor < 0: no token), or -1 where the summaries do not decide.
__device__ __forceinline__ int classify_runs(const int4 q, const int4 k)
{
    if (k.w == 0) { // every key is a depth-0 (real context) token
        if (k.y <= q.x)
            return TILE_FULL;
        if (k.x > q.y)
            return TILE_SKIP;
    } else if (k.z >= 1) { // no depth-0 key: only same-anchor, not-deeper chain tokens can match
        if (k.x > q.y || k.y < q.x || k.z > q.w)
            return TILE_SKIP;
    }
    return -1;
}
// Class of a tile pair, or -1: len keys, the first run has `split` of them.
__device__ __forceinline__ int classify_quick(const int4 (&q)[2], const int4 *k2, int len, int split)
{
    // skip: some row does not allow some key; full: a run pair is FULL, full2: with two keys or more
    bool skip = false, full = false, full2 = false, open = false;
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        const int4 k = k2[j];
        if (k.y < 0)
            continue;
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            if (q[i].y < 0)
                continue;
            const int c = classify_runs(q[i], k);
            skip |= c == TILE_SKIP;
            full |= c == TILE_FULL;
            full2 |= c == TILE_FULL && (j == 0 ? split : len - split) >= 2;
            // an undecided pair may still be FULL only if all its rows belong to the chain of its keys
            open |= c < 0;
            skip |= c < 0 && !(k.w > 0 && q[i].x == q[i].y);
        }
    }
    if (!open && !full)
        return TILE_SKIP; // also: no valid token
    if (!open && !skip)
        return len == BN ? TILE_FULL : TILE_PARTIAL;
    return full2 && skip ? TILE_PARTIAL : -1;
}

__device__ __forceinline__ void group_sync(int group)
{
    asm volatile("bar.sync %0, %1;" ::"r"(1 + group), "n"(BM) : "memory");
}

// Compacts the elements o = 0 .. n - 1 with pred(o) in ascending order: calls emit(o, position).
// Every thread of the block takes part.
template <class Pred, class Emit>
__device__ __forceinline__ int block_compact(int n, int *warp_cnt, Pred pred, Emit emit)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int base = 0;
    for (int o0 = 0; o0 < n; o0 += PLAN_THREADS) {
        const int o = o0 + threadIdx.x;
        const bool mine = o < n && pred(o);
        const unsigned bal = __ballot_sync(0xffffffffu, mine);
        __syncthreads(); // the counts of the previous round have been read
        if (lane == 0)
            warp_cnt[wid] = __popc(bal);
        __syncthreads();
        int off = base, all = 0;
        for (int w = 0; w < PLAN_THREADS / 32; ++w) {
            const int c = warp_cnt[w];
            off += w < wid ? c : 0;
            all += c;
        }
        if (mine)
            emit(o, off + __popc(bal & ((1u << lane) - 1u)));
        base += all;
    }
    return base;
}

// Sorts the query tiles by bucket(i), 0 .. SORT_BUCKETS - 1, ascending; the order inside a bucket is
// arbitrary.  Every thread of the block takes part.  Up to one tile per thread the ranks are counted
// directly (n reads of shared memory each); beyond that a counting sort over the buckets.
template <class Bucket>
__device__ __forceinline__ void block_sort(int n, int *hist, int *warp_sum, int *out, Bucket bucket)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    __syncthreads();
    if (n <= PLAN_THREADS) {
        const int mine = (int)threadIdx.x < n ? bucket(threadIdx.x) * PLAN_THREADS + (int)threadIdx.x : INT_MAX;
        hist[threadIdx.x] = mine;
        __syncthreads();
        if ((int)threadIdx.x < n) {
            int rank = 0;
            for (int j = 0; j < n; j += 4) { // entries past n hold INT_MAX
                const int4 v = *reinterpret_cast<const int4 *>(hist + j);
                rank += (int)(v.x < mine) + (int)(v.y < mine) + (int)(v.z < mine) + (int)(v.w < mine);
            }
            out[rank] = threadIdx.x;
        }
        return;
    }
    constexpr int PER = SORT_BUCKETS / PLAN_THREADS;
    for (int i = threadIdx.x; i < SORT_BUCKETS; i += PLAN_THREADS)
        hist[i] = 0;
    __syncthreads();
    for (int i = threadIdx.x; i < n; i += PLAN_THREADS)
        atomicAdd(&hist[bucket(i)], 1);
    __syncthreads();
    int sum = 0;
    for (int j = 0; j < PER; ++j)
        sum += hist[threadIdx.x * PER + j];
    int scan = sum; // inclusive over the warp
    for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, scan, o);
        scan += lane >= o ? v : 0;
    }
    if (lane == 31)
        warp_sum[wid] = scan;
    __syncthreads();
    int at = scan - sum;
    for (int w = 0; w < wid; ++w)
        at += warp_sum[w];
    for (int j = 0; j < PER; ++j) {
        const int c = hist[threadIdx.x * PER + j];
        hist[threadIdx.x * PER + j] = at;
        at += c;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < n; i += PLAN_THREADS)
        out[atomicAdd(&hist[bucket(i)], 1)] = i;
}

// The backward's inputs for the q_pad = n_qt * BM rows that the query tiles cover: -LSE * log2(e), -Delta with
// Delta[h][r] = <dO[q,h,:], O[q,h,:]>, and the packed metadata, with neutral values for the rows past the
// partition's end; and a cleared fp32 dQ staging.  D / 8 neighbouring lanes per (row, head), 8 elements each.
// Bound by memory (8 bytes per element of O).  Beside the plan rather than as a kernel of its own: the
// plan is a chain of dependent steps on a few SMs (two partitions of 4,000 tokens, 64 heads of 64, forward and
// backward calls: 768 us with a kernel behind the plan, 725 us this way).
__device__ __forceinline__ void prepare_rows(const Plan &p, const PlanSide &a, int block, int blocks)
{
    const int tpr = a.D / 8, q_len = p.q_end - p.q_begin;
    const size_t q_pad = (size_t)p.n_qt * BM, n = q_pad * a.Hq * tpr; // a multiple of 32: warps stay whole
    for (size_t gid = (size_t)block * PLAN_THREADS + threadIdx.x; gid < n; gid += (size_t)blocks * PLAN_THREADS) {
        const size_t rh = gid / tpr, r = rh / a.Hq, h = rh % a.Hq;
        const bool real = r < (size_t)q_len;
        float acc = 0.f;
        if (real) {
            const size_t src = ((size_t)p.q_begin * a.Hq * tpr + gid);
            const uint4 x4 = reinterpret_cast<const uint4 *>(a.O)[src], y4 = reinterpret_cast<const uint4 *>(a.dO)[src];
            const __nv_bfloat162 *pa = reinterpret_cast<const __nv_bfloat162 *>(&x4);
            const __nv_bfloat162 *pb = reinterpret_cast<const __nv_bfloat162 *>(&y4);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float2 x = __bfloat1622float2(pa[i]), y = __bfloat1622float2(pb[i]);
                acc += x.x * y.x + x.y * y.y;
            }
            float4 *z = reinterpret_cast<float4 *>(a.dq_acc) + 2 * gid;
            z[0] = make_float4(0.f, 0.f, 0.f, 0.f);
            z[1] = make_float4(0.f, 0.f, 0.f, 0.f);
        }
        for (int o = tpr / 2; o > 0; o >>= 1)
            acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if (gid % tpr == 0) {
            float l = -CUDART_INF_F;
            int mq = META_NONE_Q;
            if (real) {
                const float lse = a.LSE[h * (size_t)p.T + p.q_begin + r];
                if (lse != -CUDART_INF_F)
                    l = -lse * 1.4426950408889634f;
                mq = p.meta[p.q_begin + r];
                if (mq == META_NONE_K)
                    mq = META_NONE_Q;
            }
            a.nl2[h * q_pad + row_slot((int)r)] = l;
            a.nd[h * q_pad + row_slot((int)r)] = real ? -acc : 0.f;
            if (h == 0)
                a.mqp[row_slot((int)r)] = mq;
        }
    }
}

// PREP: the side blocks prepare rows.  (In one kernel for both uses, plans that do not were 1 to 2 us slower.)
template <bool PREP>
__global__ void __launch_bounds__(PLAN_THREADS) k0_plan(Plan p, int seq_begin, int seq_end, int for_bwd,
                                                        const PlanSide side)
{
    __shared__ __align__(16) int hist[SORT_BUCKETS];
    __shared__ int warp_cnt[PLAN_THREADS / 32];
    __shared__ __align__(16) int mk[PLAN_GROUPS][BN];
    __shared__ int2 part[PLAN_GROUPS][BM / 32];       // (allowed pairs, most keys of a row) per warp
    __shared__ int slot_of[PLAN_GROUPS];
    __shared__ uint8_t raw_col[RAW_SINGLE][BM];       // one-key-per-row tiles in arrival order
    __shared__ int raw_kt[RAW_SINGLE], raw_start[RAW_SINGLE], raw_ord[RAW_SINGLE], raw_conflict[RAW_SINGLE];
    __shared__ int raw_min[RAW_SINGLE], raw_max[RAW_SINGLE];
    __shared__ int4 pairs[PAIR_CACHE];                // (key tile, first token, length, first run | flags)
    __shared__ int2 entry[RAW_SINGLE];                // sorted raw tiles of an entry: first, last
    __shared__ int n_undecided, n_raw, n_entry, flag;
    sm100::pdl_wait();
    sm100::pdl_trigger();
    const int qt = blockIdx.x, tid = threadIdx.x;
    // The blocks past the query tiles work on the side (PlanSide), while memory is idle and the others wait
    // for one dependent step after another.  Clearing the fp32 sums that the backward adds to, as a fill of its
    // own, is a launch that cannot overlap its neighbours (512 tokens, 4 heads: 46.2 -> 45.1 us a step; 3,128
    // tokens, 32 heads of 128: 220 -> 213 us).
    if (qt >= p.n_qt) {
        const int block = qt - p.n_qt, blocks = gridDim.x - p.n_qt;
        float4 *zero = reinterpret_cast<float4 *>(side.zero);
        for (size_t i = (size_t)block * PLAN_THREADS + tid; i < side.zero_n / 4; i += (size_t)blocks * PLAN_THREADS)
            zero[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        if constexpr (PREP)
            prepare_rows(p, side, block, blocks);
        return;
    }
    const int lane = tid & 31;
    uint8_t *cls = p.cls + (size_t)qt * p.n_kt;
    int2 *klist = p.klist + (size_t)qt * p.n_kt;
    int *undecided = reinterpret_cast<int *>(klist); // done with when the key list is written
    if (tid == 0) {
        n_undecided = 0;
        n_raw = 0;
    }
    __syncthreads();
    // ---- classes from the summaries
    const int4 q[2] = {p.qsum[2 * qt], p.qsum[2 * qt + 1]};
    for (int kt = tid; kt < p.n_kt; kt += PLAN_THREADS) {
        const int2 k = p.ktile[kt];
        const int split = p.ksplit[kt];
        const int c = classify_quick(q, p.ksum + 2 * kt, k.y, split & 0xff);
        cls[kt] = (uint8_t)c;
        if (c < 0) {
            const int at = atomicAdd(&n_undecided, 1);
            undecided[at] = kt;
            if (at < PAIR_CACHE)
                pairs[at] = make_int4(kt, k.x, k.y, split);
        }
    }
    __syncthreads();
    // ---- exact classes of the rest, PLAN_GROUPS pairs at a time, a thread per query row
    const int r0 = p.q_begin + qt * BM, r1 = min(r0 + BM, p.q_end);
    const int group = tid / BM, row = tid % BM;
    int mq = r0 + row < r1 ? p.meta[r0 + row] : META_NONE_Q;
    if (mq == META_NONE_K)
        mq = META_NONE_Q;
    auto pair_at = [&](int w) {
        if (w < PAIR_CACHE)
            return pairs[w];
        const int kt = undecided[w];
        const int2 k = p.ktile[kt];
        return make_int4(kt, k.x, k.y, p.ksplit[kt]);
    };
    // this thread's key of pair w, requested one pair ahead of its use
    auto key_of = [&](int w) {
        if (w >= n_undecided)
            return META_NONE_K;
        const int4 pr = pair_at(w);
        return row < pr.z ? p.meta[pr.y + row] : META_NONE_K;
    };
    int key = key_of(group);
    for (int w = group; w < n_undecided; w += PLAN_GROUPS) {
        const int4 pr = pair_at(w);
        const int kt = pr.x;
        const int2 ktile = make_int2(pr.y, pr.z);
        mk[group][row] = key;
        group_sync(group);
        key = key_of(w + PLAN_GROUPS);
        // A row allows the keys of its own chain up to its depth, words [anchor << 8, mq], and the
        // depth-0 keys up to its anchor, words up to mq: in a sorted run of one of the two kinds these
        // are neighbours, and where the run's anchors follow one another their place is a subtraction.  (With
        // searches throughout, and the kinds of the runs read from memory pair by pair, this was half of a plan of
        // 18 us for 391 positions.)
        int mine = 0, col = NO_COL;
#pragma unroll
        for (int run = 0; run < 2; ++run) {
            const int lo = run == 0 ? 0 : pr.w & 0xff, hi = run == 0 ? pr.w & 0xff : ktile.y;
            if (lo >= hi)
                continue;
            const int flags = pr.w >> run; // the first run's bits are this run's
            if ((flags & KRUN0_SORTED) && (flags & (KRUN0_REAL | KRUN0_CHAIN))) {
                auto first_above = [&](int word) { // first key of the run whose word is above `word`
                    if (flags & KRUN0_EVEN)
                        return lo + min(max(((word - mk[group][lo]) >> 8) + 1, 0), hi - lo);
                    int a = lo, b = hi;
                    while (a < b) {
                        const int m = (a + b) >> 1;
                        if (mk[group][m] <= word)
                            a = m + 1;
                        else
                            b = m;
                    }
                    return a;
                };
                const int end = first_above(mq);
                const int beg = flags & KRUN0_REAL ? lo : first_above((mq & ~0xff) - 1);
                if (end > beg) {
                    mine += end - beg;
                    col = end - 1;
                }
            } else {
                for (int c = lo; c < hi; ++c)
                    if (allowed_packed(mq, mk[group][c])) {
                        ++mine;
                        col = c;
                    }
            }
        }
        const int cnt = __reduce_add_sync(0xffffffffu, mine), most = __reduce_max_sync(0xffffffffu, mine);
        if (lane == 0)
            part[group][row >> 5] = make_int2(cnt, most);
        group_sync(group);
        if (row == 0) {
            int total = 0, mx = 0, slot = -1;
            for (int i = 0; i < BM / 32; ++i) {
                total += part[group][i].x;
                mx = max(mx, part[group][i].y);
            }
            uint8_t c = TILE_PARTIAL;
            if (total == 0) {
                c = TILE_SKIP;
            } else if (ktile.y == BN && total == (r1 - r0) * BN) {
                c = TILE_FULL;
            } else if (p.allow_single && mx <= 1) {
                c = TILE_SINGLE;
                slot = atomicAdd(&n_raw, 1);
                if (slot < RAW_SINGLE) {
                    raw_kt[slot] = kt;
                    raw_start[slot] = ktile.x;
                    raw_min[slot] = INT_MAX;
                    raw_max[slot] = -1;
                } else {
                    slot = -1;
                }
            }
            cls[kt] = c;
            slot_of[group] = slot;
        }
        group_sync(group);
        const int slot = slot_of[group];
        if (slot >= 0) {
            raw_col[slot][row] = (uint8_t)col;
            const int lo = __reduce_min_sync(0xffffffffu, col == NO_COL ? INT_MAX : ktile.x + col);
            const int hi = __reduce_max_sync(0xffffffffu, col == NO_COL ? -1 : ktile.x + col);
            if (lane == 0) {
                atomicMin(&raw_min[slot], lo);
                atomicMax(&raw_max[slot], hi);
            }
        }
    }
    __syncthreads();
    // More one-key-per-row tiles than there are places (from 33 depths on).  Which of them came first
    // differs from run to run, so the lowest are taken, and looked at once more; the rest goes to the
    // tensor cores.
    if (n_raw > RAW_SINGLE) {
        block_compact(
            p.n_kt, warp_cnt, [&](int kt) { return cls[kt] == TILE_SINGLE; },
            [&](int kt, int at) {
                if (at < RAW_SINGLE) {
                    raw_kt[at] = kt;
                    raw_start[at] = p.ktile[kt].x;
                    raw_min[at] = INT_MAX;
                    raw_max[at] = -1;
                } else {
                    cls[kt] = TILE_PARTIAL;
                }
            });
        __syncthreads();
#pragma unroll 1
        for (int i = group; i < RAW_SINGLE; i += PLAN_GROUPS) {
            const int2 k = p.ktile[raw_kt[i]];
            int col = NO_COL;
#pragma unroll 1
            for (int c = 0; c < k.y; ++c)
                if (allowed_packed(mq, p.meta[k.x + c]))
                    col = c;
            raw_col[i][row] = (uint8_t)col;
            if (col != NO_COL) {
                atomicMin(&raw_min[i], k.x + col);
                atomicMax(&raw_max[i], k.x + col);
            }
        }
        __syncthreads();
    }
    // ---- one-key-per-row tiles: ascending by key tile (they were numbered in arrival order, and the
    // order of the per-pair sums shall not change from run to run)
    const int nr = min(n_raw, RAW_SINGLE);
    if (tid < nr) {
        int rank = 0;
        for (int j = 0; j < nr; ++j)
            rank += raw_kt[j] < raw_kt[tid];
        raw_ord[rank] = tid;
        raw_conflict[rank] = 0;
    }
    __syncthreads();
    // Two neighbours become one entry when their keys lie within 128 tokens and no row has a key in
    // both: the chain keys of 128 consecutive anchors are 128 consecutive tokens, which straddle two
    // key tiles unless the anchors per depth are a multiple of 128.  (391 anchors, 8 depths, 32 heads of
    // 128: forward 94 -> 72 us, the pairs' backward 76 -> 49 us.)
    for (int i = group; i + 1 < nr; i += PLAN_GROUPS)
        if (raw_col[raw_ord[i]][row] != NO_COL && raw_col[raw_ord[i + 1]][row] != NO_COL)
            raw_conflict[i] = 1;
    __syncthreads();
    if (tid == 0) {
        int n = 0;
        for (int i = 0; i < nr; ++i, ++n) {
            const bool join = i + 1 < nr && !raw_conflict[i] &&
                              raw_max[raw_ord[i + 1]] - raw_min[raw_ord[i]] < BN;
            if (n == MAX_SINGLE) { // no room: this tile and the rest go to the tensor cores
                for (; i < nr; ++i)
                    cls[raw_kt[raw_ord[i]]] = TILE_PARTIAL;
                break;
            }
            entry[n] = make_int2(i, join ? i + 1 : i);
            i += join;
        }
        n_entry = n;
        p.scount[qt] = n;
    }
    __syncthreads();
    const int ns = n_entry;
    for (int i = group; i < ns; i += PLAN_GROUPS) {
        const int2 e = entry[i];
        const int first = raw_ord[e.x], last = raw_ord[e.y];
        const int base = raw_min[first];
        int col = raw_col[first][row], start = raw_start[first];
        if (col == NO_COL && e.y != e.x) {
            col = raw_col[last][row];
            start = raw_start[last];
        }
        if (col != NO_COL)
            col = start + col - base;
        p.scs[((size_t)qt * MAX_SINGLE + i) * BM + row] = (uint8_t)col;
        if (row == 0)
            p.sbase[qt * MAX_SINGLE + i] = base;
    }
    // ---- the query tile's key list, ascending (SINGLE tiles are handled outside it)
    const int listed = block_compact(
        p.n_kt, warp_cnt, [&](int kt) { const uint8_t c = cls[kt]; return c != TILE_SKIP && c != TILE_SINGLE; },
        [&](int kt, int at) {
            const int2 k = p.ktile[kt];
            int word = k.y | ((int)cls[kt] << 16);
            if (cls[kt] == TILE_PARTIAL) {
                const int split = p.ksplit[kt];
                const bool even = (split & KRUN0_EVEN) && (split & KRUN1_EVEN) &&
                                  (split & (KRUN0_REAL | KRUN0_CHAIN)) && (split & (KRUN1_REAL | KRUN1_CHAIN));
                word |= (split & 0xff) << 8 | (split & KRUN0_REAL ? KLIST_RUN0 : 0) |
                        (split & KRUN1_REAL ? KLIST_RUN1 : 0) | (even ? KLIST_EVEN : 0);
            }
            klist[at] = make_int2(k.x, word);
        });
    if (tid == 0)
        p.kcount[qt] = listed;

    // ---- backward work items, by the last block of a chunk of BWD_CQ consecutive query tiles: a key
    // tile together with the chunk's query tiles that do not skip it.  Items of a chunk stay together,
    // so that the CTAs running at the same time work on the same few query tiles (their Q / dO rows
    // and their fp32 dQ staging rows then stay in L2), and are kept by size: the backward takes the
    // full-size ones first and ends on small ones, so that the CTAs finish together.
    __threadfence();
    __syncthreads();
    if (for_bwd) {
        const int c = qt / BWD_CQ, nq = min(BWD_CQ, p.n_qt - c * BWD_CQ);
        if (tid == 0)
            flag = atomicAdd(&p.cdone[c], 1) == nq - 1;
        __syncthreads();
        if (flag) {
            __threadfence();
            auto word = [&](int kt) { // bit b: query tile c * BWD_CQ + b is not skipped, bit 8 + b: FULL
                unsigned m = 0;
                for (int b = 0; b < nq; ++b) {
                    const uint8_t cl = __ldcg(p.cls + (size_t)(c * BWD_CQ + b) * p.n_kt + kt);
                    if (cl != TILE_SKIP && cl != TILE_SINGLE)
                        m |= 1u << b;
                    if (cl == TILE_FULL)
                        m |= 1u << (8 + b);
                }
                return m;
            };
            const size_t cap = (size_t)((p.n_qt + BWD_CQ - 1) / BWD_CQ) * p.n_kt; // per size
            if (tid < 2 * BWD_CQ)
                hist[tid] = 0;
            __syncthreads();
            unsigned m = 0; // the word of this thread's first key tile, kept for the second pass
            for (int kt = tid; kt < p.n_kt; kt += PLAN_THREADS) {
                const unsigned mm = word(kt);
                m = kt == tid ? mm : m;
                if (mm)
                    atomicAdd(&hist[__popc(mm & 0xffu) - 1], 1);
            }
            __syncthreads();
            if (tid < BWD_CQ && hist[tid])
                hist[BWD_CQ + tid] = atomicAdd(&p.counters[CNT_ITEMS + tid], hist[tid]);
            __syncthreads();
            for (int kt = tid; kt < p.n_kt; kt += PLAN_THREADS) {
                const unsigned mm = kt == tid ? m : word(kt);
                if (mm) {
                    const int sz = __popc(mm & 0xffu);
                    const int at = atomicAdd(&hist[BWD_CQ + sz - 1], 1);
                    p.bitems[(size_t)(sz - 1) * cap + at] = pack_item(kt, c, mm);
                }
            }
        }
    }
    // ---- orders of the query tiles, by the last block of all
    __syncthreads();
    if (tid == 0)
        flag = atomicAdd(&p.counters[CNT_DONE], 1) == p.n_qt - 1;
    __syncthreads();
    if (!flag)
        return;
    __threadfence();
    // what both sorts need of this thread's first tile, requested at once
    int kc = 0, sc = 0, sb = 0;
    if (tid < p.n_qt) {
        kc = __ldcg(p.kcount + tid);
        sc = __ldcg(p.scount + tid);
        sb = __ldcg(p.sbase + tid * MAX_SINGLE); // not set, and not used, without entries
    }
    // the forward takes the longest query tiles first
    block_sort(p.n_qt, hist, warp_cnt, p.qorder, [&](int i) {
        const int n = i == tid ? 2 * kc + sc : 2 * __ldcg(p.kcount + i) + __ldcg(p.scount + i);
        return SORT_BUCKETS - 1 - min(SORT_BUCKETS - 1, n);
    });
    // The SINGLE-tile backward takes them by the first token of their lowest SINGLE entry (tiles
    // without such entries last).  In the depth-major layout the chain tiles of one block of anchors
    // at depths 1, 2, .. then run one after the other, and the fp32 dK / dV rows they all add to are
    // still in L2 (one trip to memory per key row instead of one per depth).
    int shift = 7;
    while (((seq_end - seq_begin) >> shift) >= SORT_BUCKETS - 1)
        ++shift;
    if (for_bwd)
        block_sort(p.n_qt, hist, warp_cnt, p.sperm, [&](int i) {
            const int n = i == tid ? sc : __ldcg(p.scount + i);
            const int first = i == tid ? sb : __ldcg(p.sbase + i * MAX_SINGLE);
            return n > 0 ? (first - seq_begin) >> shift : SORT_BUCKETS - 1;
        });
}

// ---- test hook: the mask as the device predicate sees it -----------------------------------
__global__ void k0_mask_dense(Plan p, RangeList ranges, uint8_t *out)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    const int q = p.q_begin + blockIdx.y;
    if (k >= p.T)
        return;
    bool vis = false;
    for (int i = 0; i < ranges.n; ++i)
        vis |= (k >= ranges.begin[i] && k < ranges.end[i]);
    const int mq = p.meta[q], mk = p.meta[k];
    out[(size_t)blockIdx.y * p.T + k] =
        (uint8_t)(vis && mq != META_NONE_K && allowed_packed(mq, mk));
}

int launch_plan(const Plan &p, const int32_t *anchor, const int32_t *depth, int K, int seq_begin,
                int seq_end, const RangeList &ranges, bool for_bwd, cudaStream_t s, const PlanSide &side)
{
    if (p.n_qt == 0)
        return 0;
    const int n_seq = seq_end - seq_begin;
    const int blocks = (n_seq + 127) / 128 > p.n_qt + p.n_kt ? (n_seq + 127) / 128 : p.n_qt + p.n_kt;
    launch_dependent(k0_tiles, blocks, 128, 0, s, p, anchor, depth, K, seq_begin, seq_end, ranges);
    // A side block clears 64 KB or prepares 1,024 pieces of 8 elements, more where there are more than 256 or
    // 1,184 blocks (the plan's own come first; four are resident on an SM).  Preparation of two partitions of
    // 4,000 tokens, 64 heads of 64, with at most 296 / 444 / 592 / 1,184 blocks or any number: the case takes
    // 747 / 730 / 734 / 729 / 729 us.
    const size_t prep = side.O ? (size_t)p.n_qt * BM * side.Hq * (side.D / 8) : 0;
    const size_t want = side.zero_n * 4 / 65536 + (side.zero_n > 0) + (prep + 1023) / 1024, most = side.O ? 1184 : 256;
    launch_dependent(side.O ? k0_plan<true> : k0_plan<false>, p.n_qt + (unsigned)(want < most ? want : most),
                     PLAN_THREADS, 0, s, p, seq_begin, seq_end, for_bwd ? 1 : 0, side);
    return 2;
}

// ---- self-test of the bounded waits ----------------------------------------------------------
// One CTA waits, with the kernels' own mbar_wait, on a barrier that nothing ever arrives at; the
// wait gives up after `limit_ns`, the CTA records PEAGLE_ERR_TIMEOUT exactly as the attention
// kernels do, and returns.  Nothing faults and nothing spins without a limit.
__global__ void k0_wait_expiry(int *status, unsigned long long limit_ns, int *reached_end)
{
    __shared__ __align__(8) uint64_t bar;
    __shared__ int abort_flag;
    const uint32_t b = sm100::smem_u32(&bar);
    if (threadIdx.x == 0) {
        abort_flag = 0;
        sm100::mbar_init(b, 1);
        sm100::fence_mbar_init();
    }
    __syncthreads();
    // every thread waits; the first to run out of time raises the CTA's abort flag, the others
    // leave on seeing it
    const bool ok = sm100::mbar_wait(b, 0, &abort_flag, limit_ns);
    __syncthreads();
    if (threadIdx.x == 0) {
        if (!ok || abort_flag)
            atomicCAS(status, 0, PEAGLE_ERR_TIMEOUT);
        *reached_end = 1;
    }
}

int launch_wait_expiry(int *status, unsigned long long limit_ns, int *reached_end, cudaStream_t s)
{
    k0_wait_expiry<<<1, 64, 0, s>>>(status, limit_ns, reached_end);
    return 1;
}

int launch_mask_dense(const Plan &p, const RangeList &ranges, uint8_t *out, cudaStream_t s)
{
    const int q_len = p.q_end - p.q_begin;
    if (q_len <= 0)
        return 0;
    k0_mask_dense<<<dim3((p.T + 255) / 256, q_len), 256, 0, s>>>(p, ranges, out);
    return 1;
}

} // namespace peagle
