// The last pass of a partition's backward (head_dim 64 and 128): the SINGLE entries -- windows of keys in
// which every query row allows at most one key, such as the chain tiles of the depth-major layout --
// and the rounding of dQ.  On the tensor cores such a window costs a full 128 x 128 step for 128 useful
// pairs, so the pairs are done one by one on the CUDA cores.
// For a pair (query row q of head h, key k of its KV head), with the forward's LSE and
// Delta = <dO, O> (Section 3.2's backward, same formulas as the tile kernel):
//   s = <Q[q,h], K[k]>,  p = exp(scale * s - LSE),  dp = <dO[q,h], V[k]>,  ds = p * (dp - Delta)
//   dQ[q,h] += scale * ds * K[k]      dK[k] += scale * ds * Q[q,h]      dV[k] += p * dO[q,h]
// One kernel, query-major so that no reverse (key -> queries) list is needed: a unit of D / 8 lanes per
// (query row, KV head); for every head of the group it adds to the row's dQ and to per-key dK / dV sums
// kept in registers across the heads (one fp32 add
// per key row at the end).  It runs after the tile kernel: its own part of dQ is added to the fp32
// staging row that the tile kernel left, which is read once and leaves as bf16.  (Before the tile
// kernel, as the initial value of the staging, the same pairs took a write of the staging of
// their own and a separate rounding pass: headline shape 0.44 + 0.12 ms, together 0.40 ms.)
#include <math_constants.h>

#include <algorithm>

#include "peagle_internal.h"
#include "sm100_ptx.cuh"

namespace peagle {
using namespace sm100;

struct SingleParams {
    const int *scount;
    const uint8_t *scs;  // [n_qt][MAX_SINGLE][BM] key of row r in entry i's window, or NO_COL
    const int *sbase;    // [n_qt][MAX_SINGLE] first token of entry i's window
    const int *sperm;    // [n_qt] order in which the blocks take the query tiles
    const __nv_bfloat16 *Q, *K, *V, *dO;
    const float *nl2, *nd; // [Hq][q_pad] -LSE * log2(e) and -Delta
    const float *dq_acc;   // [q_len][Hq][D] what the tile kernel left
    __nv_bfloat16 *dQ;
    float *dK_acc, *dV_acc;
    int *status;
    int q_begin, q_end, q_pad, Hq, Hkv, rows_per_block;
    float scale, scale_log2;
};

// A row of D elements is spread over LANES = D / 8 consecutive lanes of a warp, a unit: lane `sub` holds the
// elements 4 sub .. 4 sub + 3 of each half of the row, as fp32 in neighbouring pairs.  (With 8 sub ..
// 8 sub + 7, one load of bf16, the fp32 rows were read, written and added to with 32 bytes between the
// lanes' 16: two-way bank conflicts in shared memory and half-used sectors in the adds to dK and dV.
// 2,048 positions, 32 heads of 128: 240 -> 219 us; 4,096, 64 heads of 64: 435 -> 421 us.)
struct Chunk {
    F2 v[4];
};
__device__ __forceinline__ Chunk unpack_chunk(const uint4 t)
{
    const uint32_t w[4] = {t.x, t.y, t.z, t.w};
    Chunk c;
#pragma unroll
    for (int i = 0; i < 4; ++i)
        c.v[i] = f2(__uint_as_float(w[i] << 16), __uint_as_float(w[i] & 0xffff0000u));
    return c;
}
template <int D>
__device__ __forceinline__ Chunk load_chunk(const __nv_bfloat16 *row, int sub)
{
    const uint2 a = reinterpret_cast<const uint2 *>(row)[sub], b = reinterpret_cast<const uint2 *>(row + D / 2)[sub];
    return unpack_chunk(make_uint4(a.x, a.y, b.x, b.y));
}
__device__ __forceinline__ float dot_chunk(const Chunk &a, const Chunk &b)
{
    F2 acc = mul_f2(a.v[0], b.v[0]);
#pragma unroll
    for (int i = 1; i < 4; ++i)
        acc = fma_f2(a.v[i], b.v[i], acc);
    const float2 r = unf2(acc);
    return r.x + r.y;
}
// acc += x * (w, w)
__device__ __forceinline__ void axpy_chunk(Chunk &acc, const Chunk &x, float w)
{
    const F2 ww = f2(w, w);
#pragma unroll
    for (int i = 0; i < 4; ++i)
        acc.v[i] = fma_f2(x.v[i], ww, acc.v[i]);
}
__device__ __forceinline__ void zero_chunk(Chunk &c)
{
#pragma unroll
    for (int i = 0; i < 4; ++i)
        c.v[i] = f2(0.f, 0.f);
}
// adds this lane's piece of a row (dst = the row's first element) scaled by f
template <int D>
__device__ __forceinline__ void red_chunk(float *dst, int sub, const Chunk &x, float f)
{
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        const float2 a = unf2(x.v[2 * j]), b = unf2(x.v[2 * j + 1]);
        asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(dst + 4 * sub + D / 2 * j), "f"(a.x * f),
                     "f"(a.y * f), "f"(b.x * f), "f"(b.y * f)
                     : "memory");
    }
}

// This lane's dQ values of row r, head h, rounded to bf16.
template <int D>
__device__ __forceinline__ void store_dq(const SingleParams &P, int r, int h, int sub, const float4 a, const float4 b)
{
    __nv_bfloat16 *row = P.dQ + ((size_t)(P.q_begin + r) * P.Hq + h) * D;
    reinterpret_cast<uint2 *>(row)[sub] = make_uint2(pack_bf16x2(a.x, a.y), pack_bf16x2(a.z, a.w));
    reinterpret_cast<uint2 *>(row + D / 2)[sub] = make_uint2(pack_bf16x2(b.x, b.y), pack_bf16x2(b.z, b.w));
}

constexpr int KEYS = 2; // keys per pass: their dK / dV sums are kept in registers across the heads

struct KeyRows {
    int tok[KEYS];           // -1: none
    uint4 k[KEYS], v[KEYS]; // this lane's elements of the keys' rows, packed bf16
};
// Takes the next KEYS keys of the row (bits of `keys`: entries, ascending; at least one) and requests their
// rows.
// Lane `sub` of a unit has the key of entry sub in t0 and, with 8 lanes, that of entry sub + 8 in t1.
template <int D>
__device__ __forceinline__ void next_keys(const SingleParams &P, unsigned &keys, int t0, int t1, int sub, unsigned um,
                                          int ub, int g, KeyRows &out)
{
#pragma unroll
    for (int i = 0; i < KEYS; ++i) {
        const int at = __ffs(keys) - 1;
        out.tok[i] = -1;
        if (at >= 0)
            out.tok[i] = __shfl_sync(um, at < D / 8 ? t0 : t1, ub + at % (D / 8));
        keys &= keys - 1;
        // an absent key takes the row of the first one, which the query sees: with weight zero it is
        // harmless unless the row has an Inf or NaN, and then the result has one anyway
        const size_t kr = ((size_t)(out.tok[i] >= 0 ? out.tok[i] : out.tok[0]) * P.Hkv + g) * D;
        auto row_of = [&](const __nv_bfloat16 *row) {
            const uint2 a = __ldg(reinterpret_cast<const uint2 *>(row) + sub);
            const uint2 b = __ldg(reinterpret_cast<const uint2 *>(row + D / 2) + sub);
            return make_uint4(a.x, a.y, b.x, b.y);
        };
        out.k[i] = row_of(P.K + kr);
        out.v[i] = row_of(P.V + kr);
    }
}

template <int D, bool LAST>
__device__ __forceinline__ void single_pass(const SingleParams &P, const KeyRows &rows, int sub, unsigned um, int r,
                                            int g, int G, const __nv_bfloat16 *sq, const __nv_bfloat16 *sdo,
                                            float *sdq, const float *snl2, const float *snd)
{
    static_assert(KEYS == 2, "the reduction below deals two keys");
    const int (&tok)[KEYS] = rows.tok;
    Chunk k[KEYS], v[KEYS], dk[KEYS], dv[KEYS];
#pragma unroll
    for (int i = 0; i < KEYS; ++i) {
        k[i] = unpack_chunk(rows.k[i]);
        v[i] = unpack_chunk(rows.v[i]);
        zero_chunk(dk[i]);
        zero_chunk(dv[i]);
    }
    const bool odd = sub & 1, second = sub & 2; // which of the four sums this lane ends up with
    const bool mine = tok[0] >= 0 && (!second || tok[1] >= 0);
    for (int hh = 0; hh < G; ++hh) {
        const int h = g * G + hh;
        const Chunk q = load_chunk<D>(sq + (size_t)h * D, sub);
        const Chunk dO = load_chunk<D>(sdo + (size_t)h * D, sub);
        const float nl2 = snl2[h], nd = snd[h];
        // The four sums <q, k0>, <q, k1>, <dO, v0>, <dO, v1> over the unit's lanes: halve what a lane
        // carries with every exchange (even lanes keep the scores, odd lanes dp; then one key each), so
        // 4 shuffles instead of 12 for 8 lanes; a lane then has one key's p and ds and gets the other's.
        const float s0 = dot_chunk(q, k[0]), s1 = dot_chunk(q, k[1]);
        const float e0 = dot_chunk(dO, v[0]), e1 = dot_chunk(dO, v[1]);
        const float a0 = (odd ? e0 : s0) + __shfl_xor_sync(um, odd ? s0 : e0, 1);
        const float a1 = (odd ? e1 : s1) + __shfl_xor_sync(um, odd ? s1 : e1, 1);
        float a = (second ? a1 : a0) + __shfl_xor_sync(um, second ? a0 : a1, 2);
#pragma unroll
        for (int o = 4; o < D / 8; o <<= 1)
            a += __shfl_xor_sync(um, a, o);
        const float b = __shfl_xor_sync(um, a, 1);
        // an absent key takes part with weight zero, so that the keys' chains of dependent
        // instructions interleave instead of branching around each other
        const float p = fast_exp2(fmaf(odd ? b : a, P.scale_log2, mine ? nl2 : -CUDART_INF_F)); // nl2 = -inf: p = 0
        const float ds = p * ((odd ? a : b) + nd);
        const float p_other = __shfl_xor_sync(um, p, 2), ds_other = __shfl_xor_sync(um, ds, 2);
        const float p0 = second ? p_other : p, p1 = second ? p : p_other;
        const float ds0 = second ? ds_other : ds, ds1 = second ? ds : ds_other;
        axpy_chunk(dk[0], q, ds0);
        axpy_chunk(dk[1], q, ds1);
        axpy_chunk(dv[0], dO, p0);
        axpy_chunk(dv[1], dO, p1);
        float4 *acc = reinterpret_cast<float4 *>(sdq + (size_t)h * D) + sub;
        const float4 x = acc[0], y = acc[D / 8];
        Chunk dq;
        dq.v[0] = f2(x.x, x.y);
        dq.v[1] = f2(x.z, x.w);
        dq.v[2] = f2(y.x, y.y);
        dq.v[3] = f2(y.z, y.w);
        axpy_chunk(dq, k[0], ds0 * P.scale);
        axpy_chunk(dq, k[1], ds1 * P.scale);
        const float2 d0 = unf2(dq.v[0]), d1 = unf2(dq.v[1]), d2 = unf2(dq.v[2]), d3 = unf2(dq.v[3]);
        const float4 lo = make_float4(d0.x, d0.y, d1.x, d1.y), hi = make_float4(d2.x, d2.y, d3.x, d3.y);
        if (LAST) {
            store_dq<D>(P, r, h, sub, lo, hi);
        } else {
            acc[0] = lo;
            acc[D / 8] = hi;
        }
    }
#pragma unroll
    for (int i = 0; i < KEYS; ++i)
        if (tok[i] >= 0) {
            const size_t kr = ((size_t)tok[i] * P.Hkv + g) * D;
            red_chunk<D>(P.dK_acc + kr, sub, dk[i], P.scale);
            red_chunk<D>(P.dV_acc + kr, sub, dv[i], 1.f);
        }
}

// Block = RB rows of the partition x all KV heads; unit (row, KV head g).  The rows of Q, dO and of the
// dQ staging (all heads of a row are contiguous) come in by bulk copies, so that the memory system sees
// the block's whole input at once instead of one 16-byte load per lane and head; the arithmetic then
// reads shared memory.  Between the passes of a row with more than two keys its dQ stays there.
// Bound by memory and by the latency of the dependent chain of a head (dot products, shuffles, exp2), so
// warps per SM count: shared memory allows one per 4 KB x 8 heads, which is why head_dim 128 has units
// of 16 lanes (8 lanes of twice the elements and 250 registers were 5 % slower).
// Shared memory: [RB][Hq * D] fp32 dQ rows, [2][RB][Hq * D] bf16 rows of Q and dO, [2][RB][Hq] fp32 row
// values.
constexpr int SINGLE_THREADS = 256;
template <int D>
__global__ void __launch_bounds__(SINGLE_THREADS, 1) bwd_finish_single(const SingleParams P)
{
    constexpr int LANES = D / 8;
    extern __shared__ __align__(128) uint8_t smem[];
    __shared__ __align__(8) uint64_t bar, bar_q; // the dQ staging; Q and dO
    __shared__ int abort_flag;
    pdl_wait();
    pdl_trigger();
    const int RB = P.rows_per_block;
    const int row_elems = P.Hq * D;
    float *sDQ = reinterpret_cast<float *>(smem);
    __nv_bfloat16 *sQ = reinterpret_cast<__nv_bfloat16 *>(sDQ + (size_t)RB * row_elems);
    __nv_bfloat16 *sdO = sQ + (size_t)RB * row_elems;
    float *snl2 = reinterpret_cast<float *>(sdO + (size_t)RB * row_elems);
    float *snd = snl2 + RB * P.Hq;
    // blocks walk the query tiles in the order K0 chose (tiles that share key rows together); RB
    // divides the tile height, so a block's rows lie in one tile
    const int qt = P.sperm[(blockIdx.x * RB) / BM];
    const int r0 = qt * BM + (blockIdx.x * RB) % BM;
    const int n_real = max(0, min(RB, (P.q_end - P.q_begin) - r0)); // rows of the partition
    if (n_real == 0)
        return;
    const uint32_t bar_a = smem_u32(&bar), bar_b = smem_u32(&bar_q);
    const uint32_t bytes = (uint32_t)(n_real * row_elems * 2);
    if (threadIdx.x == 0) {
        abort_flag = 0;
        mbar_init(bar_a, 1);
        mbar_init(bar_b, 1);
        fence_mbar_init();
        mbar_arrive_expect_tx(bar_a, 2 * bytes);
        bulk_load(smem_u32(sDQ), P.dq_acc + (size_t)r0 * row_elems, 2 * bytes, bar_a);
    }
    const int ns = P.scount[qt];
    if (ns > 0 && threadIdx.x == 0) {
        mbar_arrive_expect_tx(bar_b, 2 * bytes);
        const size_t off = (size_t)(P.q_begin + r0) * row_elems;
        bulk_load(smem_u32(sQ), P.Q + off, bytes, bar_b);
        bulk_load(smem_u32(sdO), P.dO + off, bytes, bar_b);
    }
    const int sub = threadIdx.x % LANES;
    const int ub = (threadIdx.x & 31) - sub; // first lane of the unit
    const unsigned um = (LANES == 8 ? 0xffu : 0xffffu) << ub;
    const int unit = threadIdx.x / LANES;
    const int rl = unit / P.Hkv, g = unit % P.Hkv;
    const int r = r0 + rl;
    const int G = P.Hq / P.Hkv;
    const bool real = rl < n_real;
    int t0 = -1, t1 = -1; // the row's keys, see next_keys
    if (ns > 0) {
        for (int i = threadIdx.x; i < n_real * P.Hq; i += blockDim.x) {
            const size_t ri = (size_t)(i % P.Hq) * P.q_pad + row_slot(r0 + i / P.Hq);
            snl2[i] = P.nl2[ri];
            snd[i] = P.nd[ri];
        }
        const uint8_t *cols = P.scs + (size_t)qt * MAX_SINGLE * BM + r % BM;
        const int *base = P.sbase + qt * MAX_SINGLE;
        if (real && sub < ns && cols[sub * BM] != NO_COL)
            t0 = base[sub] + cols[sub * BM];
        if (LANES == 8 && real && sub + 8 < ns && cols[(sub + 8) * BM] != NO_COL)
            t1 = base[sub + 8] + cols[(sub + 8) * BM];
        static_assert(MAX_SINGLE == 16, "one or two entries per lane of a unit");
    }
    __syncthreads(); // row values, barriers
    unsigned keys = (__ballot_sync(um, t0 >= 0) & um) >> ub;
    if (LANES == 8)
        keys |= ((__ballot_sync(um, t1 >= 0) & um) >> ub) << 8;
    const bool any = keys != 0;
    KeyRows cur;
    if (any)
        next_keys<D>(P, keys, t0, t1, sub, um, ub, g, cur);
    // every thread waits for the rows (bounded); the units past the partition's end then leave
    if (!mbar_wait(bar_a, 0, &abort_flag) || (ns > 0 && !mbar_wait(bar_b, 0, &abort_flag))) {
        if (threadIdx.x == 0)
            atomicCAS(P.status, 0, PEAGLE_ERR_TIMEOUT);
        return;
    }
    if (!real)
        return; // the lanes of a unit leave together
    const __nv_bfloat16 *sq = sQ + (size_t)rl * row_elems, *sdo = sdO + (size_t)rl * row_elems;
    float *sdq = sDQ + (size_t)rl * row_elems;
    const float *rnl2 = snl2 + rl * P.Hq, *rnd = snd + rl * P.Hq;
    if (!any) { // nothing to add: round what the tile kernel left
        for (int hh = 0; hh < G; ++hh) {
            const int h = g * G + hh;
            const float4 *acc = reinterpret_cast<const float4 *>(sdq + (size_t)h * D) + sub;
            store_dq<D>(P, r, h, sub, acc[0], acc[D / 8]);
        }
        return;
    }
    while (keys) {
        KeyRows nxt; // requested one pass ahead
        next_keys<D>(P, keys, t0, t1, sub, um, ub, g, nxt);
        single_pass<D, false>(P, cur, sub, um, r, g, G, sq, sdo, sdq, rnl2, rnd);
        cur = nxt;
    }
    single_pass<D, true>(P, cur, sub, um, r, g, G, sq, sdo, sdq, rnl2, rnd);
}

size_t single_row_bytes(int Hq, int D) { return (size_t)Hq * (8 * D + 8); }

int launch_finish_single(const Plan &p, const BwdArgs &a, cudaStream_t s)
{
    SingleParams P;
    P.scount = p.scount;
    P.scs = p.scs;
    P.sbase = p.sbase;
    P.sperm = p.sperm;
    P.Q = static_cast<const __nv_bfloat16 *>(a.Q);
    P.K = static_cast<const __nv_bfloat16 *>(a.K);
    P.V = static_cast<const __nv_bfloat16 *>(a.V);
    P.dO = static_cast<const __nv_bfloat16 *>(a.dO);
    P.nl2 = a.nl2;
    P.nd = a.nd;
    P.dq_acc = a.dq_acc;
    P.dQ = static_cast<__nv_bfloat16 *>(a.dQ);
    P.dK_acc = a.dK_acc;
    P.dV_acc = a.dV_acc;
    P.q_begin = p.q_begin;
    P.q_end = p.q_end;
    P.q_pad = p.n_qt * BM;
    P.Hq = a.Hq;
    P.Hkv = a.Hkv;
    P.scale = a.scale;
    P.scale_log2 = a.scale * 1.4426950408889634f;
    P.status = p.status;
    // rows per block: up to 128 threads within 48 KB of shared memory (the headline shape, 64 heads: one
    // row, 33 KB, 64 threads)
    const size_t row_bytes = single_row_bytes(a.Hq, a.D);
    const int row_threads = a.Hkv * (a.D / 8);
    int rb = 1; // a power of two, so that it divides the tile height
    while (2 * rb * row_threads <= 128 && 2 * rb * row_bytes <= 48 * 1024)
        rb *= 2;
    const size_t smem = rb * row_bytes;
    const int threads = rb * row_threads;
    if (threads > SINGLE_THREADS || smem > 200 * 1024)
        return PEAGLE_ERR_BAD_SHAPE;
    P.rows_per_block = rb;
    // per device, so set before every launch (host time only)
    void (*kern)(const SingleParams) = a.D == 64 ? bwd_finish_single<64> : bwd_finish_single<128>;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
        return PEAGLE_ERR_CUDA;
    launch_dependent(kern, (unsigned)((P.q_pad + rb - 1) / rb), threads, smem, s, P);
    return 1;
}

} // namespace peagle
