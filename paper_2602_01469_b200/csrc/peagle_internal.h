// Internal declarations shared by the translation units of libpeagle.
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <utility>

#include "../../include/peagle.h"

namespace peagle {

constexpr int BM = 128;          // query rows per tile
constexpr int BN = 128;          // keys per tile
constexpr int MAX_KRANGES = 32;  // visible key ranges per partition
#ifndef PEAGLE_BWD_CQ
#define PEAGLE_BWD_CQ 4 // 2 / 3 / 4: bwd64_kernel 3.03 / 3.00 / 3.01 ms at 4,096 positions, 22.1 / 21.8 / 21.6 at 11,008
#endif
constexpr int BWD_CQ = PEAGLE_BWD_CQ; // query tiles per backward work item (aligned chunk; at most 4)
static_assert(BWD_CQ >= 1 && BWD_CQ <= 4, "pack_item has four bits per field");
constexpr int32_t META_NONE_Q = -1;         // packed metadata of a row outside the partition (sees nothing)
constexpr int32_t META_NONE_K = 0x7fffffff; // packed metadata of a key outside the batch (seen by nobody)

// TILE_SINGLE is internal: a PARTIAL tile in which every query row allows at most one key (the
// chain tiles of the depth-major layout: one allowed pair per row).  Such tiles are taken out of
// the tensor-core lists and handled pair by pair.  The test hook reports them as PARTIAL.
enum TileClass : uint8_t { TILE_SKIP = 0, TILE_PARTIAL = 1, TILE_FULL = 2, TILE_SINGLE = 3 };
constexpr int MAX_SINGLE = 16;   // SINGLE entries kept per query tile; further ones stay PARTIAL
// device counters of a plan
constexpr int CNT_BWD_CURSOR = 2, CNT_FWD_CURSOR = 3, CNT_DONE = 4, CNT_ITEMS = 8, PLAN_COUNTERS = 16;
static_assert(CNT_ITEMS + BWD_CQ <= PLAN_COUNTERS, "a counter per item size");
constexpr int NO_COL = 255;      // "this row allows no key of the tile"

// Second word of a key list entry: bits 0-7 length, 8-15 keys in the first run of equal depth, 16-17 class; bit
// KLIST_RUN0 / KLIST_RUN1: the run's keys are depth-0 tokens; bit KLIST_EVEN: in each run the keys are all depth 0 or
// all deeper and their anchors follow one another.  (The bits above the class only where it is PARTIAL.)
constexpr int KLIST_RUN0 = 1 << 24, KLIST_RUN1 = 1 << 25, KLIST_EVEN = 1 << 26;
__device__ __forceinline__ int klist_len(int word) { return word & 0xff; }
__device__ __forceinline__ int klist_split(int word) { return word >> 8 & 0xff; }
__device__ __forceinline__ int klist_class(int word) { return word >> 16 & 3; }

// Visible key ranges of one call, passed to kernels by value.
struct RangeList {
    int n;
    int begin[MAX_KRANGES];
    int end[MAX_KRANGES];
};

// Everything the mask evaluator / tile classifier / scheduler (K0) produces for one call.
// All pointers are device memory inside the context's scratch buffer.
struct Plan {
    int T;                 // tokens in the batch
    int q_begin, q_end;    // query rows of the call
    int n_qt, n_kt;        // tile counts
    int32_t *meta;         // [T] packed (anchor << 8 | depth)
    int2 *ktile;           // [n_kt] (first token, length)
    int4 *qsum;            // [n_qt][2] (min anchor, max anchor, min depth, max depth) of the tile's first
                           // run of equal depth and of the rest; max anchor -1: no token
    int4 *ksum;            // [n_kt][2]
    int *ksplit;           // [n_kt] keys in the first run, flags of the runs
    uint8_t *cls;          // [n_qt][n_kt] tile classes
    int *counters;         // [PLAN_COUNTERS] device counters, zero before k0_plan: CNT_*
    int *cdone;            // [n_ch] query tiles of a chunk that are classified
    int2 *klist;           // [n_qt][n_kt] compact non-skip key tiles per query tile: (first token, KLIST_* word)
    int *kcount;           // [n_qt]
    int *qorder;           // [n_qt] query tiles, most key tiles first (no order among about equal ones)
    int2 *bitems;          // [BWD_CQ][n_ch * n_kt] backward work items by size (1 .. BWD_CQ query tiles):
                           // packed by pack_item; counters[CNT_ITEMS + size - 1] of each
    int allow_single;      // 1: the kernels of this shape take SINGLE tiles pair by pair
    int *scount;           // [n_qt] SINGLE entries per query tile (at most MAX_SINGLE): windows of 128 keys,
                           // ascending, in which every query row has at most one key
    int *sbase;            // [n_qt][MAX_SINGLE] first token of entry i's window
    uint8_t *scs;          // [n_qt][MAX_SINGLE][BM] key of row r in entry i's window, or NO_COL
    int *sperm;            // [n_qt] query tiles in the order the SINGLE-tile backward takes them:
                           // by the first key tile of their SINGLE entries, so that the query
                           // tiles that add to the same key rows run close together in time
    int *status;           // device status word
};

// A backward work item in two words: key tile; chunk of query tiles << 8 | which of them are FULL << 4 | which
// take part.  (A plan has BWD_CQ places per key tile and chunk for them, and grows with the square of the
// length.)  `mask`: bit b, query tile b of the chunk takes part; bit 8 + b, it is FULL.
__device__ __forceinline__ int2 pack_item(int key_tile, int chunk, unsigned mask)
{
    return make_int2(key_tile, (int)((unsigned)chunk << 8 | (mask >> 8 & 15u) << 4 | (mask & 15u)));
}
__device__ __forceinline__ int item_chunk(int2 item) { return (int)((unsigned)item.y >> 8); }
__device__ __forceinline__ unsigned item_mask(int2 item) { return ((unsigned)item.y & 15u) | ((unsigned)item.y >> 4 & 15u) << 8; }

struct FwdArgs {
    const void *Q, *K, *V;
    void *O;
    float *LSE;
    int Hq, Hkv, D;
    float scale;
    // optional hand-over to the backward of the same partition (all null when not wanted):
    // dO, the backward's per-row scratch, which the forward's epilogue then fills, and its dQ staging
    const void *dO = nullptr;
    float *nl2 = nullptr, *nd = nullptr;
    int32_t *mqp = nullptr;
    float *dq_acc = nullptr; // the backward's dQ staging, which the forward clears
};

struct BwdArgs {
    const void *Q, *K, *V, *O, *dO;
    const float *LSE;
    void *dQ;
    float *dK_acc, *dV_acc;
    // per-row scratch of the call, q_pad = query tiles * BM rows, rows past the partition padded;
    // row r's entry stands at row_slot(r).  Written, and dq_acc cleared, by the forward of the partition
    // in the driver, where dO is known, else beside the plan (PlanSide).
    float *nl2;     // [Hq][q_pad] -LSE * log2(e); -inf for a padded row or a row that saw no key
    float *nd;      // [Hq][q_pad] -Delta = -<dO, O>; 0 for a padded row
    int32_t *mqp;   // [q_pad] packed metadata of the partition's rows; META_NONE_Q when padded
    float *dq_acc;  // [q_len][Hq][D] scratch, fp32
    int Hq, Hkv, D;
    float scale;
};

typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *,
                                  const cuuint64_t *, const cuuint64_t *, const cuuint32_t *,
                                  const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// Where row r (of the padded partition) keeps its value in nl2, nd and mqp.  The compute warps of the
// backward hold their scores as tcgen05.ld.16x256b gives them: thread t of a warp has the query
// columns 8i + 2 (t % 4) and the next one.  With the 16 values of two such groups in the order of the
// threads that use them, a thread gets the four of a group pair with one 16-byte load.
__host__ __device__ inline int row_slot(int r)
{
    return (r & ~15) | (((r >> 1) & 3) << 2) | ((r >> 3 & 1) << 1) | (r & 1);
}

// Launches a kernel that begins with pdl_wait / pdl_trigger (sm100_ptx.cuh): its launch and set-up overlap
// the kernel before it.  A call of a few tokens is a chain of kernels of a few microseconds each, and the
// gaps between them were a fifth of its time (512 tokens, 4 heads: 56 -> 47 us a step).  Not for the
// projection products and the rotary prologue, where it measured nothing.
template <class... Params, class... Args>
inline cudaError_t launch_dependent(void (*kernel)(Params...), unsigned grid, unsigned threads, size_t smem,
                                    cudaStream_t s, Args &&...args)
{
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}

// What the plan kernel does on the side, in blocks of its own: it clears `zero_n` floats (a multiple of 4) at
// `zero` (16-byte aligned), and with O set it prepares the backward of the call's rows from O, dO and LSE (see
// BwdArgs).
struct PlanSide {
    float *zero = nullptr;
    size_t zero_n = 0;
    const void *O = nullptr, *dO = nullptr;
    const float *LSE = nullptr;
    float *nl2 = nullptr, *nd = nullptr;
    int32_t *mqp = nullptr;
    float *dq_acc = nullptr;
    int Hq = 0, D = 0;
};

// K0: mask evaluator, tile classifier, scheduler.  Returns the number of kernels launched.
int launch_plan(const Plan &p, const int32_t *anchor, const int32_t *depth, int K, int seq_begin,
                int seq_end, const RangeList &ranges, bool for_bwd, cudaStream_t s, const PlanSide &side = PlanSide());
int launch_mask_dense(const Plan &p, const RangeList &ranges, uint8_t *out, cudaStream_t s);
// One CTA whose bounded wait runs out after limit_ns: records PEAGLE_ERR_TIMEOUT in *status.
int launch_wait_expiry(int *status, unsigned long long limit_ns, int *reached_end, cudaStream_t s);

// K1 / K2.  Return the number of kernels launched, or a negative peagle_status.
// ev0/ev1 (may be null) are recorded on the stream right before / after the main kernel.
int launch_fwd(const Plan &p, const FwdArgs &a, EncodeTiledFn enc, int n_sm, cudaStream_t s,
               cudaEvent_t ev0, cudaEvent_t ev1);
int launch_bwd(const Plan &p, const BwdArgs &a, EncodeTiledFn enc, int n_sm, cudaStream_t s,
               cudaEvent_t ev0, cudaEvent_t ev1);
// The backward's last pass where SINGLE entries are enabled: their pairs, added to dK_acc / dV_acc and to
// the dQ staging that the tile kernel left, and dQ rounded to bf16.
int launch_finish_single(const Plan &p, const BwdArgs &a, cudaStream_t s);
// Shared memory that it takes per query row.
size_t single_row_bytes(int Hq, int D);
int launch_cast_grads(const float *dK_acc, const float *dV_acc, void *dK, void *dV, size_t n,
                      cudaStream_t s);
int launch_cast_one(const float *src, void *dst, size_t n, cudaStream_t s);

// Rotary prologue (backward = false: fused row -> Q, K, V) and its backward (dQ, dK, dV -> gradient
// of the fused row).  Returns the number of kernels launched.
int launch_rope(bool backward, const void *fused_in, void *fused_out, const void *q_in,
                const void *k_in, const void *v_in, void *q_out, void *k_out, void *v_out,
                const int32_t *anchor, const int32_t *depth, int T, int Hq, int Hkv, int D,
                float base, int n_sm, cudaStream_t s);

// C[m][n] (+)= sum_k A(m,k) B(n,k) in bf16 with fp32 accumulation (peagle_gemm.cu).  a_t / b_t: the
// operand is stored transposed ([k][m] / [k][n]); c_f32_add: C is fp32 and added to, else bf16 and
// stored.  Leading dimensions in elements.  Returns kernels launched or a negative status.
int launch_gemm(EncodeTiledFn enc, const void *A, long long lda, int a_t, const void *B, long long ldb,
                int b_t, void *C, long long ldc, int c_f32_add, int M, int N, int K, int *status,
                cudaStream_t s);

// Packed-metadata form of the attention predicate: m = anchor << 8 | depth.
// (depth_k == 0 and anchor_k <= anchor_q) or (anchor_k == anchor_q and depth_k <= depth_q)
__host__ __device__ inline bool allowed_packed(int32_t mq, int32_t mk)
{
    return (mk <= mq) && (((mk & 0xff) == 0) || ((mk ^ mq) < 256));
}
// The same as an interval: key mk is seen by the rows mk .. mk + allowed_span(mk), a subtraction and an
// unsigned comparison per pair.
__host__ __device__ inline uint32_t allowed_span(int32_t mk)
{
    return (mk & 0xff) == 0 ? (uint32_t)(0x7fffffff - mk) : (uint32_t)(255 - (mk & 0xff));
}

} // namespace peagle
