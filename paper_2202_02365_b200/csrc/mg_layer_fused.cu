// One GraphSage layer over DENSE as a single persistent kernel (Algorithm 3 with the mean
// aggregator, fused with the layer's linear maps):
//
//     H^l[r] = act([ self_r | mean_r ] . [W_self ; W_nbr] + b)
//
// The [self | mean] operand never goes to global memory.  Two CTAs work as a pair; producer warps of each gather the
// rows its tile of 128 output rows needs (64 in layers of few rows; layer 1: base representations straight from the
// partition buffer; later layers: rows of H^{l-1}), reduce each segment in entry order, round to the operand's
// precision (TF32, or fp16 over fp16 rows) and write 128-byte K slices directly into swizzled shared-memory stages.  One
// thread of the pair issues tcgen05.mma (cta_group::2) against weights that stay in tensor memory, or against weight
// slices that a TMA thread streams from L2 (no multicast); the fp32 accumulators of the tiles' halves live in tensor
// memory, so that the epilogue of one (bias, ReLU, store) overlaps the gather and MMAs of the next.  Tiles are handed
// out round-robin in packed row order, so all SMs work on the same mini-batch at a time and its rows stay in L2.
// The same gather feeds the kernel of the weights' gradients (k_sage_grad_weights).
// Every mbarrier wait is bounded; on a time-out the role records a code and stops.

#include <cuda_fp16.h>

#include <algorithm>
#include <cstdlib>

#include "mg_device.cuh"
#include "mg_internal.cuh"
#include "mg_tcgen05.cuh"

using namespace tc;

namespace {

constexpr int BM = 128;               // output rows per tile
constexpr int KC = 32;                // floats per K slice (one 128-byte swizzle row)
// Warp roles, laid out so that every role fills whole warpgroups (four consecutive warps):
//   warps 0..15   producers (gather + segment mean)         four warpgroups
//   warps 16..19  epilogue (tensor memory -> global)        one warpgroup
//   warp 20 TMA (weights), warp 21 MMA + tensor memory, warps 22..23 planners: one warpgroup
// Every thread has 80 registers (768 x 80 = 61,440 of the SM's 65,536).  A build option moves registers between the
// warpgroups with `setmaxnreg` (-DMG_FUSED_SETMAXNREG=1 -DMG_FUSED_MAXNREG=72 -DMG_REG_PROD=80 -DMG_REG_EPI=56
// -DMG_REG_CTL=56: the CTA then leaves room for a 256-thread block of the sampler beside it); it is off because every
// such configuration measured 15 % slower in the first layer than the plain one.
constexpr int kProducerWarps = 16;
constexpr int kFirstProducerWarp = 0;
constexpr int kFirstEpilogueWarp = 16;
constexpr int kTmaWarp = 20, kMmaWarp = 21;
constexpr int kPlannerWarps = 2;
constexpr int kFirstPlannerWarp = 22;
constexpr int kFusedThreads = (kFirstPlannerWarp + kPlannerWarps) * 32;  // 768
#ifndef MG_FUSED_MAXNREG
#define MG_FUSED_MAXNREG 80
#endif
#ifndef MG_FUSED_SETMAXNREG
#define MG_FUSED_SETMAXNREG 0
#endif
constexpr int kMaxStages = 8;
constexpr int kGroupCols = 128;                  // input columns whose (self, mean) slices the producers fill together (TF32 operands)
// With half-precision base representations the first layer can run its GEMM in kind::f16 (fp16 operands, fp32
// accumulate): a 128-byte slice row then holds 64 columns, a lane's 16 bytes are 8 columns, a group is 256 columns,
// and the same number of MMAs covers twice the K.  Everything else (slices per group, swizzle, stages, barriers) is
// the same, so the element-size dependent constants come from one place:
template <bool F16> struct Geo {
    static constexpr int kKC = F16 ? 64 : 32;        // columns per K slice (one 128-byte swizzle row)
    static constexpr int kLaneCols = F16 ? 8 : 4;    // columns of a group one lane owns (16 bytes of operand)
    static constexpr int kGroup = 32 * kLaneCols;    // columns per group
};
static_assert(Geo<false>::kKC == kPackCols32 && Geo<false>::kGroup == kPackGroup32 && Geo<true>::kKC == kPackCols16 && Geo<true>::kGroup == kPackGroup16,
              "the order the weights are packed in");
constexpr int kRowsInFlight = 2;                 // rows a producer warp builds at the same time
constexpr int kBlockRows = kProducerWarps * kRowsInFlight;   // 32: rows of a tile the producers build in one round
constexpr int kBlocksPerTile = BM / kBlockRows;              // 4
constexpr int kPlanSlots = kBlocksPerTile;                   // planned row blocks in shared memory (one tile's worth)
constexpr int HM = BM / 2;                                   // rows of a half tile: the unit the MMAs work on
constexpr int kAccBufs = 4;                                  // accumulator buffers in tensor memory (two tiles' halves)
constexpr int kSlicesPerGroup = 2 * kGroupCols / KC;         // 8 K slices: (self, mean) x four 32-column blocks
constexpr int kUnroll = 5;                       // neighbour rows per output row fetched before the first add
static_assert(kUnroll == 5, "the first-round table is read as four + one source rows");
// an A stage: a 128-byte slice row per row of the tile (16 or 8 KiB)
__host__ __device__ constexpr uint32_t stage_bytes(int halves) { return (uint32_t)(HM * halves) * 128; }
// Shared memory of a weight ring.  Two halves: shallow on purpose -- with 128 KB of A stages the CTA then fits the 196 KB
// carve-out, which leaves the gathers twice the L1 (measured: layer 1 of the bench 2.92 -> 2.75 ms).  One half: what the
// smaller A stages leave of the same carve-out.
constexpr int ring_bytes(int halves) { return (halves == 1 ? 96 : 32) * 1024; }
constexpr int fused_smem_limit(int halves) { return 8 * (int)stage_bytes(halves) + ring_bytes(halves) + 1024; }

struct FusedArgs {
    // DENSE (device arrays of the sample)
    int32_t B, k, layer;
    const int32_t* rowbase_out;  // [B+1] of layer l
    const int32_t* rowbase_in;   // [B+1] of layer l-1
    const int32_t* cum;          // [B][k+2]
    const int32_t* node_off;     // [k+1][B+1]
    const int32_t* nodes;
    const int32_t* ent_off;
    const int32_t* ent_nbrs;
    const int32_t* ent_repr;
    const int4* row_meta;        // [M] (self source row, first entry, entry count, first H^{l-1} row of the batch), or null: see row_of_sample
    // input rows
    const float* h_prev;         // layers >= 2: [rows of layer l-1, d_in]
    const char* src_base;        // layer 1: the feature buffer; later layers: h_prev
    uint32_t src_row_bytes;      // (32-bit: the row address is then one wide multiply-add)
    FeatGeom feat;               // layer 1: where a node's row lives in the partition buffer
    int32_t safe_src;            // a source row that is always valid to read (rows past the end load it)
    // shapes
    int32_t d_in, d_in_pad;      // d_in_pad = d_in rounded up to 32; K = 2 * d_in_pad
    int32_t N, BN;               // output width and its MMA tile width (multiple of 16, <= 256)
    int64_t row_lo;              // first packed output row this launch computes
    int64_t M;                   // one past its last packed output row
    int32_t sa, sb;              // A and B stages
    const void* w_rows;          // weights-in-tensor-memory form: the padded weight matrix [N][2 * d_in_pad] (fp32 or fp16), K order of the slices
    int32_t tmem_cols;
    int32_t relu;
    int32_t sum_aggr;            // neighbour term = sum of the sampled neighbours instead of their mean
    int32_t out_f16;             // the output rows are stored as fp16 (an intermediate layer of a model that keeps them so)
    const float* bias;
    float* out;                  // [M, N]
    float* out2;                 // the same rows once more, for the caller (the last layer with a device output), or null
    float* kept_agg;             // the rows' aggregates, [M, d_in] fp32 and not rounded (for the backward pass), or null
    uint32_t* positive;          // a bit per output value: above zero (kept layers of a ReLU, for the backward pass), or null
    uint32_t* error;
};

constexpr int kTsMaxEntriesPerRow = 8, kTsMaxEntriesNarrow = 16;   // layers with more entries per output row than this stream their weights (narrow: at most 128 output columns; between the two mg_layer_narrow_ts decides)
constexpr int kLaneEntries = 32;   // rows up to this long are translated by their own lane of the planner warp
constexpr int kKeyCap = 704;    // source-row indices of a row block's entries cached in shared memory (22 per row: what still fits the 196 KB carve-out)

// What a producer needs to build one output row: x = source row of the row's own representation; y = first
// entry and z = number of entries in the sample's entry arrays (z < 0: row past the end); w = first cached
// source-row index of the row when the block's entries fit the cache, else (layers >= 2) the first row of the
// mini-batch in H^{l-1}.
typedef int4 RowMeta;

// Source row of an entry.  Layer 1: the feature-buffer row of node `key` (its partition's slot);
// later layers: row of H^{l-1}.  The address is src_base + row * src_row_bytes.
template <bool FIRST>
__device__ __forceinline__ int32_t source_row(const FusedArgs& a, int32_t in_base, int32_t key) {
    if (FIRST) return (int32_t)feat_row(a.feat, key);
    return in_base + key;
}

// A lane's piece of a source row, as 16 bytes of registers: four fp32 values (fp16 sources widened exactly), or,
// for fp16 operands (F16), eight fp16 values as they are in memory.
template <bool HALF, bool F16>
__device__ __forceinline__ uint4 load_piece(const char* p) {
    if (F16) return __ldg(reinterpret_cast<const uint4*>(p));
    if (HALF) {
        const uint2 raw = __ldg(reinterpret_cast<const uint2*>(p));
        const float2 lo = __half22float2(*reinterpret_cast<const __half2*>(&raw.x));
        const float2 hi = __half22float2(*reinterpret_cast<const __half2*>(&raw.y));
        return make_uint4(__float_as_uint(lo.x), __float_as_uint(lo.y), __float_as_uint(hi.x), __float_as_uint(hi.y));
    }
    return __ldg(reinterpret_cast<const uint4*>(p));
}

// fp32 running sum of a lane's piece over a row's entries, and the operand forms of the result and of the self row
template <bool F16> struct PieceSum;
template <> struct PieceSum<false> {
    float a[4];
    __device__ __forceinline__ void zero() { a[0] = a[1] = a[2] = a[3] = 0.f; }
    __device__ __forceinline__ void add(const uint4& r) {
        a[0] += __uint_as_float(r.x); a[1] += __uint_as_float(r.y); a[2] += __uint_as_float(r.z); a[3] += __uint_as_float(r.w);
    }
    __device__ __forceinline__ uint4 operand(float scale) const {   // rounded to nearest TF32
        return make_uint4(__float_as_uint(to_tf32(a[0] * scale)), __float_as_uint(to_tf32(a[1] * scale)),
                          __float_as_uint(to_tf32(a[2] * scale)), __float_as_uint(to_tf32(a[3] * scale)));
    }
    static __device__ __forceinline__ uint4 self_operand(const uint4& r) {
        return make_uint4(__float_as_uint(to_tf32(__uint_as_float(r.x))), __float_as_uint(to_tf32(__uint_as_float(r.y))),
                          __float_as_uint(to_tf32(__uint_as_float(r.z))), __float_as_uint(to_tf32(__uint_as_float(r.w))));
    }
};
template <> struct PieceSum<true> {
    float a[8];
    __device__ __forceinline__ void zero() {
#pragma unroll
        for (int i = 0; i < 8; ++i) a[i] = 0.f;
    }
    __device__ __forceinline__ void add(const uint4& r) {
        const uint32_t w[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&w[i]));
            a[2 * i] += f.x; a[2 * i + 1] += f.y;
        }
    }
    __device__ __forceinline__ uint4 operand(float scale) const {   // rounded to nearest fp16 (the 10-bit mantissa TF32 keeps)
        uint32_t w[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const __half2 h = __floats2half2_rn(a[2 * i] * scale, a[2 * i + 1] * scale);
            w[i] = *reinterpret_cast<const uint32_t*>(&h);
        }
        return make_uint4(w[0], w[1], w[2], w[3]);
    }
    static __device__ __forceinline__ uint4 self_operand(const uint4& r) { return r; }   // fp16 rows are operands as they are
};

// Row metadata of a sample of one mini-batch, as the planners take it from the sample themselves: lane h knows hop h's first row and first
// node (there is no mini-batch to look up).  A row then takes the same round trip as from mg_layer_rows' table, and a call of few rows, which is a
// chain of launches, has one launch less (two layers on a graph of 10,000: the whole call 74.4 -> 71.5 us; three on 1M nodes: 155 us either way).
struct HopOfLane { int32_t row0, node0; };
__device__ __forceinline__ HopOfLane hop_of_lane(const FusedArgs& a) {
    const int lane = threadIdx.x & 31;
    const bool on = lane <= a.k - a.layer;
    return {on ? __ldg(a.cum + lane) : 0, on ? __ldg(a.node_off + 2 * lane) : 0};
}
template <bool FIRST>
__device__ __forceinline__ int4 row_of_sample(const FusedArgs& a, HopOfLane hops, int32_t r, bool on) {
    int32_t idx = 0;
    for (int h = 0; h <= a.k - a.layer; ++h) {
        const int32_t row0 = __shfl_sync(0xFFFFFFFFu, hops.row0, h), node0 = __shfl_sync(0xFFFFFFFFu, hops.node0, h);
        if (r >= row0) idx = node0 + (r - row0);
    }
    if (!on) return make_int4(a.safe_src, 0, -1, 0);
    const int32_t e0 = __ldg(a.ent_off + idx), e1 = __ldg(a.ent_off + idx + 1);
    return make_int4(FIRST ? (int32_t)feat_row(a.feat, __ldg(a.nodes + idx)) : r, e0, e1 - e0, 0);
}

// A planner warp's work on one row block, lane = row: the rows' metadata, their entries translated to source rows, each row's
// first kUnroll source rows, all in shared memory.
template <bool FIRST>
__device__ __forceinline__ void plan_block(const FusedArgs& a, const int32_t* keys, int4 rm, RowMeta* meta, int32_t* src_rows, int32_t (*first_rows)[8],
                                           int32_t* plan_total) {
    const int lane = threadIdx.x & 31;
    const int32_t end = (int32_t)warp_incl_scan((uint32_t)max(rm.z, 0));   // end of the row's cached entries
    const int32_t total = __shfl_sync(0xFFFFFFFFu, end, 31);
    const bool cached = total <= kKeyCap;
    const int32_t in_base = rm.w, koff = end - max(rm.z, 0);
    meta[lane] = make_int4(rm.x, rm.y, rm.z, cached ? koff : in_base);
    const int32_t zmax = (int32_t)__reduce_max_sync(0xFFFFFFFFu, (uint32_t)max(rm.z, 0));
    if (cached && zmax <= kLaneEntries) {
        // short rows (the usual case): every lane translates its own row's entries, kUnroll loads in flight
        // (the entries of consecutive rows are consecutive, so the lanes' loads share their cache lines)
        for (int32_t i0 = 0; i0 < zmax; i0 += kUnroll) {
            int32_t key[kUnroll];
#pragma unroll
            for (int u = 0; u < kUnroll; ++u) key[u] = i0 + u < rm.z ? __ldg(keys + rm.y + i0 + u) : 0;
#pragma unroll
            for (int u = 0; u < kUnroll; ++u)
                if (i0 + u < rm.z) src_rows[koff + i0 + u] = source_row<FIRST>(a, in_base, key[u]);
        }
    } else if (cached) {
        // entry j belongs to the first row whose end exceeds j
        for (int32_t j0 = 0; j0 < total; j0 += 32 * 4) {
            int32_t key[4], base[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int32_t j = j0 + u * 32 + lane;
                int lo = 0, hi = 31;
#pragma unroll
                for (int s = 0; s < 5; ++s) {
                    const int mid = (lo + hi) >> 1;
                    const int32_t e = __shfl_sync(0xFFFFFFFFu, end, mid);
                    if (lo < hi) { if (e > j) hi = mid; else lo = mid + 1; }
                }
                const int32_t e0 = __shfl_sync(0xFFFFFFFFu, rm.y, lo), k0 = __shfl_sync(0xFFFFFFFFu, koff, lo);
                base[u] = __shfl_sync(0xFFFFFFFFu, in_base, lo);
                key[u] = j < total ? __ldg(keys + e0 + (j - k0)) : 0;
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int32_t j = j0 + u * 32 + lane;
                if (j < total) src_rows[j] = source_row<FIRST>(a, base[u], key[u]);
            }
        }
    }
    if (lane == 0) *plan_total = cached ? total : -1;
    __syncwarp();
    if (cached) {
        // lane = row: its first kUnroll source rows, padded with its own source row
        int32_t fr[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) fr[j] = (j < kUnroll && j < rm.z) ? src_rows[koff + j] : rm.x;
        fr[5] = __float_as_int(rm.z > 0 ? (a.sum_aggr ? 1.f : 1.f / (float)rm.z) : 0.f);   // the mean's factor (1 for a sum)
        *reinterpret_cast<int4*>(&first_rows[lane][0]) = make_int4(fr[0], fr[1], fr[2], fr[3]);
        *reinterpret_cast<int4*>(&first_rows[lane][4]) = make_int4(fr[4], fr[5], fr[6], fr[7]);
        __syncwarp();
    }
}

// A gather warp's work on two planned rows: the lane's 16-byte operand pieces of each row's self part and aggregate.
// (RAW: fp32 values as they are, not rounded to the operand's precision.  KEEP: the aggregates go to `keep`, if it is given, as well:
// its rows are a.d_in floats apart.)
template <bool FIRST, bool HALF, bool F16, bool RAW = false, bool KEEP = false>
__device__ __forceinline__ void gather_rows(const FusedArgs& a, const char* src, bool on, bool cached, const RowMeta* meta, const int32_t (*first_rows)[8],
                                            const int32_t* rows_of, uint4* selfv, uint4* meanv, float* keep = nullptr) {
    RowMeta mq[kRowsInFlight];
    PieceSum<F16> acc[kRowsInFlight];
    int top = 0;
#pragma unroll
    for (int q2 = 0; q2 < kRowsInFlight; ++q2) {
        mq[q2] = meta[q2];
        selfv[q2] = make_uint4(0u, 0u, 0u, 0u);
        meanv[q2] = selfv[q2];
        acc[q2].zero();
        top = max(top, mq[q2].z);
    }
    if (on) {
#pragma unroll
        for (int q2 = 0; q2 < kRowsInFlight; ++q2)
            selfv[q2] = load_piece<HALF, F16>(src + (size_t)(uint32_t)mq[q2].x * (size_t)a.src_row_bytes);
        if (cached) {
            // Every load is issued unconditionally: a slot past the end of a row's entries re-reads
            // the row's own representation (a cache hit) and is not added.  Branch-free code is what
            // lets all loads of a round be in flight together.  First round: the planner has laid
            // out the kUnroll source rows per row, padding included.
            {
                uint4 v[kRowsInFlight][kUnroll];
#pragma unroll
                for (int q2 = 0; q2 < kRowsInFlight; ++q2) {
                    const int4 f4 = *reinterpret_cast<const int4*>(first_rows[q2]);
                    const int32_t f5 = first_rows[q2][4];
                    v[q2][0] = load_piece<HALF, F16>(src + (size_t)(uint32_t)f4.x * (size_t)a.src_row_bytes);
                    v[q2][1] = load_piece<HALF, F16>(src + (size_t)(uint32_t)f4.y * (size_t)a.src_row_bytes);
                    v[q2][2] = load_piece<HALF, F16>(src + (size_t)(uint32_t)f4.z * (size_t)a.src_row_bytes);
                    v[q2][3] = load_piece<HALF, F16>(src + (size_t)(uint32_t)f4.w * (size_t)a.src_row_bytes);
                    v[q2][4] = load_piece<HALF, F16>(src + (size_t)(uint32_t)f5 * (size_t)a.src_row_bytes);
                }
#pragma unroll
                for (int j = 0; j < kUnroll; ++j)   // entry order
#pragma unroll
                    for (int q2 = 0; q2 < kRowsInFlight; ++q2)
                        if (j < mq[q2].z) acc[q2].add(v[q2][j]);
            }
            for (int e = kUnroll; e < top; e += kUnroll) {
                uint4 v[kRowsInFlight][kUnroll];
#pragma unroll
                for (int j = 0; j < kUnroll; ++j)
#pragma unroll
                    for (int q2 = 0; q2 < kRowsInFlight; ++q2) {
                        const bool live = e + j < mq[q2].z;
                        const int32_t sr = rows_of[live ? mq[q2].w + e + j : 0];
                        v[q2][j] = load_piece<HALF, F16>(src + (size_t)(uint32_t)(live ? sr : mq[q2].x) * (size_t)a.src_row_bytes);
                    }
#pragma unroll
                for (int j = 0; j < kUnroll; ++j)   // entry order
#pragma unroll
                    for (int q2 = 0; q2 < kRowsInFlight; ++q2)
                        if (e + j < mq[q2].z) acc[q2].add(v[q2][j]);   // warp-uniform: predicated adds, not a branch around a load
            }
        } else {
            // a row block with more entries than the shared-memory cache holds: plain per-entry loop
            const int32_t* keys = FIRST ? a.ent_nbrs : a.ent_repr;
#pragma unroll
            for (int q2 = 0; q2 < kRowsInFlight; ++q2)
                for (int e = 0; e < mq[q2].z; ++e) {
                    const int32_t sr = source_row<FIRST>(a, mq[q2].w, __ldg(keys + mq[q2].y + e));
                    acc[q2].add(load_piece<HALF, F16>(src + (size_t)(uint32_t)sr * (size_t)a.src_row_bytes));
                }
        }
#pragma unroll
        for (int q2 = 0; q2 < kRowsInFlight; ++q2) {
            const float inv = cached ? __int_as_float(first_rows[q2][5])
                                     : (mq[q2].z > 0 ? (a.sum_aggr ? 1.f : 1.f / (float)mq[q2].z) : 0.f);
            if (RAW) {
                meanv[q2] = make_uint4(__float_as_uint(acc[q2].a[0] * inv), __float_as_uint(acc[q2].a[1] * inv), __float_as_uint(acc[q2].a[2] * inv),
                                       __float_as_uint(acc[q2].a[3] * inv));
                continue;
            }
            if (KEEP && keep && mq[q2].z >= 0)
                *reinterpret_cast<float4*>(keep + q2 * a.d_in) = make_float4(acc[q2].a[0] * inv, acc[q2].a[1] * inv, acc[q2].a[2] * inv, acc[q2].a[3] * inv);
            meanv[q2] = acc[q2].operand(inv);
            selfv[q2] = PieceSum<F16>::self_operand(selfv[q2]);
        }
    }
}

// TS: the weights stay in tensor memory for the whole kernel and are the MMAs' first operand (M = 256 output columns over
// the pair, a CTA's 128 in its 128 lanes, K <= 256 columns), the gathered rows the second (N = 128: a half tile of either
// CTA); the accumulator is the transposed output, [output column][row].  Nothing is streamed per half tile then -- with
// the weights in shared memory a half tile waits for eight 16 KB slices through a two-stage ring (4 us of latency).
//
// ROWS: 128 output rows per tile and CTA, or 64 (one half only) for layers of few rows.  Such a layer is one chain -- plan, gather, weight
// slices, epilogue -- whose links are halved, on twice the CTAs, with six weight slices in flight instead of two (the operand
// stages are half as large); layers of many rows want the second half, whose gather runs under the first half's MMAs.  32: a tile is
// one row block, for layers that all SMs together take in one round that way; the other half of a 64-row stage is then never
// written, and what the MMAs make of it never read (one mini-batch on 1M nodes, layers of 4,300 and 1,000 rows: 82 -> 62 us; two layers on
// a graph of 10,000: 24 -> 18 us).
//
// KEEP: what the backward pass wants is left on the way (its own instances, so that the others keep their registers).
template <bool FIRST, bool HALF, bool F16, bool TS, int ROWS, bool KEEP>
__global__ void __cluster_dims__(2, 1, 1) __maxnreg__(MG_FUSED_MAXNREG)
k_sage_layer_fused(const __grid_constant__ CUtensorMap map_w, const __grid_constant__ CUtensorMap map_out,
                   const __grid_constant__ CUtensorMap map_out2, FusedArgs a) {
    constexpr int KCE = Geo<F16>::kKC, GC = Geo<F16>::kGroup, LC = Geo<F16>::kLaneCols;
    constexpr int HALVES = ROWS > HM ? 2 : 1, TM = ROWS;     // rows of a tile
    constexpr int kBlocks = ROWS / kBlockRows, kHalfBlocks = kBlocks / HALVES;   // row blocks of a tile, of a half
    constexpr uint32_t kStage = stage_bytes(HALVES);
    extern __shared__ uint8_t smem_raw[];
    // a_ready and acc_empty are used in the leader CTA only (both CTAs arrive there); a_free, b_empty and acc_full
    // exist in both CTAs and are signalled in both by the leader's commits; b_full counts both halves' bytes in
    // the leader.
    __shared__ uint64_t a_ready[2], a_free[2], b_full[kMaxStages], b_empty[kMaxStages];   // a_*: one per half tile
    __shared__ uint64_t acc_full[kAccBufs], acc_empty[kAccBufs];
    __shared__ uint64_t w_ready;   // TS, leader only: both CTAs' weights are in tensor memory
    __shared__ uint32_t tmem_slot;
    __shared__ uint64_t plan_full[kPlanSlots], plan_empty[kPlanSlots];
    __shared__ RowMeta meta[kPlanSlots][kBlockRows];
    __shared__ int32_t src_rows[kPlanSlots][kKeyCap];
    __shared__ int32_t plan_total[kPlanSlots];   // entries of the block, or -1 when they do not fit the cache
    // source rows of each row's first kUnroll entries, padded with the row's own source row: the first round of
    // gathers then needs no selects
    __shared__ __align__(16) int32_t first_rows[kPlanSlots][kBlockRows][8];
    __shared__ __align__(1024) float out_stage[4][32 * 32];   // per epilogue warp: one 32 x 32 slice, 128-byte swizzled, for the TMA store

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = cluster_ctarank();      // 0: leader of the pair (issues the MMAs), 1: its peer
    const bool leader = rank == 0;
    const uint32_t pair = blockIdx.x >> 1, n_pairs = gridDim.x >> 1;
    const int half_n = a.BN / 2;                  // weight rows (output columns) this CTA stages
    const uint32_t b_bytes = (uint32_t)half_n * 128;   // one 128-byte slice row per staged output column
    uint8_t* a_base = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint8_t* b_base = a_base + (size_t)a.sa * kStage;
    const int n_chunks = 2 * a.d_in_pad / KCE;
    const int64_t n_tiles = (a.M - a.row_lo + TM - 1) / TM;
    const int64_t n_tile_pairs = (n_tiles + 1) / 2;
    // iteration `it` of this pair works on tile pair (pair + it * n_pairs): the leader on its even tile, the peer
    // on the odd one (which may lie past the end: then all its rows are padding)
    const uint32_t my_iters = pair < n_tile_pairs ? (uint32_t)((n_tile_pairs - pair + n_pairs - 1) / n_pairs) : 0u;
    auto tile_of = [&](uint32_t it) -> int64_t { return 2 * ((int64_t)pair + (int64_t)it * n_pairs) + rank; };

    if (threadIdx.x == 0) {
        for (int s = 0; s < 2; ++s) { mbar_init(&a_ready[s], 2 * kProducerWarps); mbar_init(&a_free[s], 1); }
        for (int s = 0; s < a.sb; ++s) { mbar_init(&b_full[s], 1); mbar_init(&b_empty[s], 1); }
        for (int s = 0; s < kAccBufs; ++s) { mbar_init(&acc_full[s], 1); mbar_init(&acc_empty[s], 2 * 4); }
        mbar_init(&w_ready, 2 * 4);   // the four loading warps of both CTAs
        for (int s = 0; s < kPlanSlots; ++s) { mbar_init(&plan_full[s], 1); mbar_init(&plan_empty[s], kProducerWarps); }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(&map_w) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(&map_out) : "memory");
    }
    if (warp == kMmaWarp) {
        // the same warp of both CTAs allocates the pair's tensor memory
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)), "r"((uint32_t)a.tmem_cols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    cluster_sync_all();       // barriers of both CTAs are initialised before anyone arrives on a remote one
    tc_fence_after();
    const uint32_t tmem_base = tmem_slot;
    const uint32_t acc_stride = (uint32_t)(a.tmem_cols / kAccBufs);  // columns per accumulator buffer (a multiple of 32)
    constexpr uint32_t kTsAcc0 = 256, kTsAccCols = 128;              // TS: weights in columns [0, 256), two accumulators behind them
    if constexpr (TS) {
        if (warp >= kFirstEpilogueWarp && warp < kTmaWarp) {   // (the warps that may touch lanes 32 q .. 32 q + 31)
            const int q = warp & 3;
            const int n = (int)rank * 128 + q * 32 + lane;     // this lane's output column = its row of the weights
            const int K = F16 ? a.d_in_pad : 2 * a.d_in_pad;   // 32-bit words per row of the weights (two fp16 values per word)
            const float4* wrow = reinterpret_cast<const float4*>(static_cast<const uint32_t*>(a.w_rows) + (size_t)min(n, a.N - 1) * K);
            for (int k0 = 0; k0 < K; k0 += 32) {
                uint32_t v[32];
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const float4 x = n < a.N ? __ldg(wrow + k0 / 4 + j) : make_float4(0.f, 0.f, 0.f, 0.f);
                    v[4 * j] = __float_as_uint(x.x); v[4 * j + 1] = __float_as_uint(x.y);
                    v[4 * j + 2] = __float_as_uint(x.z); v[4 * j + 3] = __float_as_uint(x.w);
                }
                tmem_st_32(tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)k0, v);
            }
            asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
            // only the leader's MMA thread waits for the weights: planners and gather warps start at once
            tc_fence_before();
            __syncwarp();
            if (lane == 0) {
                if (leader) mbar_arrive(&w_ready);
                else mbar_arrive_cluster(mapa_u32(smem_u32(&w_ready), 0));
            }
        }
    }
    const int n_groups = (a.d_in_pad + GC - 1) / GC;

    // (Build option) registers move from the epilogue's and the control warpgroup to the producers': each warpgroup
    // executes its one setmaxnreg at the head of its own branch, so that the compiler budgets the branch with it (the
    // decreases never wait, the increases wait for them; the static_assert keeps the sum within the launch allocation).
#define MG_STR2(x) #x
#define MG_STR(x) MG_STR2(x)
#if MG_FUSED_SETMAXNREG
#define MG_REG_SET(n) do { if ((n) < MG_FUSED_MAXNREG) asm volatile("setmaxnreg.dec.sync.aligned.u32 " MG_STR(n) ";" ::: "memory"); \
                           else if ((n) > MG_FUSED_MAXNREG) asm volatile("setmaxnreg.inc.sync.aligned.u32 " MG_STR(n) ";" ::: "memory"); } while (0)
#else
#define MG_REG_SET(n)
#endif
#ifndef MG_REG_PROD
#define MG_REG_PROD 80
#define MG_REG_EPI 56
#define MG_REG_CTL 56
#endif
    static_assert(MG_FUSED_SETMAXNREG == 0 || 16 * MG_REG_PROD + 4 * MG_REG_EPI + 4 * MG_REG_CTL <= 24 * MG_FUSED_MAXNREG,
                  "the warpgroups' registers must fit what the CTA was launched with");
    if (warp >= kTmaWarp) {
    MG_REG_SET(MG_REG_CTL);
    if (warp == kTmaWarp && !TS) {
        // ---------------- weight slices: each CTA stages its half of the output columns (TMA from L2) ----------------
        if (lane == 0) {
            uint32_t cnt = 0;
            bool ok = true;
            // the weight slices of a group are streamed once per half tile, in the order the MMAs consume them
            for (uint32_t it = 0; it < my_iters && ok; ++it)
                for (int grp = 0; grp < n_groups && ok; ++grp)
                    for (int h = 0; h < HALVES && ok; ++h) {
                        const int gch = min(kSlicesPerGroup, n_chunks - grp * kSlicesPerGroup);
                        for (int c = 0; c < gch; ++c, ++cnt) {
                            const int s = cnt % a.sb;
                            if (cnt >= (uint32_t)a.sb && !mbar_wait(&b_empty[s], ((cnt / a.sb) - 1) & 1)) { report(a.error, 11u); ok = false; break; }
                            if (leader) mbar_expect_tx(&b_full[s], 2 * b_bytes);   // both halves are counted on the leader's barrier
                            tma_load_2d_pair(b_base + (size_t)s * b_bytes, &map_w, mapa_u32(smem_u32(&b_full[s]), 0),
                                             (grp * kSlicesPerGroup + c) * KCE, (int)rank * half_n);
                        }
                    }
        }
        __syncwarp();
    } else if (warp == kMmaWarp) {
        // ---------------- MMA issue: one thread of the leader, for both CTAs ----------------
        if (TS && lane == 0 && leader) {
            // M = 256 output columns over the pair, N = 128 rows (a half tile of each CTA), fp32 accumulate, K-major
            const uint32_t idesc = (1u << 4) | ((F16 ? 0u : 2u) << 7) | ((F16 ? 0u : 2u) << 10) | ((uint32_t)(128 >> 3) << 17) | ((uint32_t)(256 >> 4) << 24);
            bool ok = mbar_wait(&w_ready, 0);
            if (!ok) report(a.error, 18u);
            tc_fence_after();
            for (uint32_t it = 0; it < my_iters && ok; ++it)
                for (int h = 0; h < HALVES && ok; ++h) {
                    const uint32_t hu = it * HALVES + h, buf = hu & 1;
                    if (hu >= 2 && !mbar_wait(&acc_empty[buf], ((hu >> 1) - 1) & 1)) { report(a.error, 12u); ok = false; break; }
                    tc_fence_after();
                    if (!mbar_wait(&a_ready[h], it & 1)) { report(a.error, 13u); ok = false; break; }
                    tc_fence_after();
                    const uint32_t d_tmem = tmem_base + kTsAcc0 + buf * kTsAccCols;
                    for (int c = 0; c < n_chunks; ++c) {
                        const uint64_t db = smem_desc_sw128(smem_u32(a_base + (size_t)c * kStage + (size_t)h * (HM * 128)));
#pragma unroll
                        for (int kk = 0; kk < 4; ++kk) {   // 32 bytes of every slice row = 8 columns of the weights per instruction
                            if (F16) mma_f16_pair_ts(d_tmem, tmem_base + (uint32_t)(c * 32 + kk * 8), db + (uint64_t)(kk * 2), idesc, (c | kk) ? 1u : 0u);
                            else mma_tf32_pair_ts(d_tmem, tmem_base + (uint32_t)(c * 32 + kk * 8), db + (uint64_t)(kk * 2), idesc, (c | kk) ? 1u : 0u);
                        }
                    }
                    mma_commit_pair(&a_free[h]);
                    mma_commit_pair(&acc_full[buf]);
                }
        }
        if (!TS && lane == 0 && leader) {
            // M = 128 over the pair: 64 rows (a half tile) of each CTA per instruction
            // fp32 accumulate; operands TF32 (format 2) or fp16 (format 0), both K-major
            const uint32_t idesc = (1u << 4) | ((F16 ? 0u : 2u) << 7) | ((F16 ? 0u : 2u) << 10) | ((uint32_t)(a.BN >> 3) << 17) |
                                   ((uint32_t)((2 * HM) >> 4) << 24);
            uint32_t cnt = 0;
            bool ok = true;
            for (uint32_t it = 0; it < my_iters && ok; ++it)
                for (int grp = 0; grp < n_groups && ok; ++grp)
                    for (int h = 0; h < HALVES && ok; ++h) {
                        const uint32_t hu = it * HALVES + h;                       // half tiles of this CTA, in order
                        const uint32_t buf = hu % kAccBufs;
                        const uint32_t s_h = it * (uint32_t)n_groups + grp;   // fills of half h's stage rows so far
                        if (grp == 0) {
                            if (hu >= (uint32_t)kAccBufs && !mbar_wait(&acc_empty[buf], ((hu / kAccBufs) - 1) & 1)) { report(a.error, 12u); ok = false; break; }
                            tc_fence_after();
                        }
                        // both CTAs' producers have filled the half's rows of this group's K slices
                        if (!mbar_wait(&a_ready[h], s_h & 1)) { report(a.error, 13u); ok = false; break; }
                        const uint32_t d_tmem = tmem_base + buf * acc_stride;
                        const int gch = min(kSlicesPerGroup, n_chunks - grp * kSlicesPerGroup);
                        for (int c = 0; c < gch; ++c, ++cnt) {
                            const int sb = cnt % a.sb;
                            if (!mbar_wait(&b_full[sb], (cnt / a.sb) & 1)) { report(a.error, 13u); ok = false; break; }
                            tc_fence_after();
                            const uint64_t da = smem_desc_sw128(smem_u32(a_base + (size_t)c * kStage + (size_t)h * (HM * 128)));
                            const uint64_t db = smem_desc_sw128(smem_u32(b_base + (size_t)sb * b_bytes));
#pragma unroll
                            for (int kk = 0; kk < 4; ++kk) {   // 32 bytes of every slice row per instruction: K = 8 (TF32) or 16 (fp16)
                                if (F16) mma_f16_pair(d_tmem, da + (uint64_t)(kk * 2), db + (uint64_t)(kk * 2), idesc, (grp | c | kk) ? 1u : 0u);
                                else mma_tf32_pair(d_tmem, da + (uint64_t)(kk * 2), db + (uint64_t)(kk * 2), idesc, (grp | c | kk) ? 1u : 0u);
                            }
                            mma_commit_pair(&b_empty[sb]);
                        }
                        if (!ok) break;
                        mma_commit_pair(&a_free[h]);    // one commit frees the half's rows of all the group's stages
                        if (grp == n_groups - 1) mma_commit_pair(&acc_full[buf]);
                    }
        }
        __syncwarp();
    } else {
        // ---------------- planners: row blocks of 32 rows, prepared ahead of the producers ----------------
        // A planner warp takes every kPlannerWarps-th row block: lane = row.  It reads the rows' metadata, scans the
        // entry counts, and translates the block's entries to source rows in shared memory, so that the producers'
        // gathers depend on nothing but shared memory.
        // (with the weights in tensor memory nothing is streamed and the weight warp is a third planner)
        constexpr int kPlanners = TS ? kPlannerWarps + 1 : kPlannerWarps;
        const int plw = warp == kTmaWarp ? kPlannerWarps : warp - kFirstPlannerWarp;
        const int32_t* keys = FIRST ? a.ent_nbrs : a.ent_repr;
        // The kernel may have started while the one before it (the row metadata, the layer below) still runs.  Barriers, tensor
        // memory and the weights -- which only kernels before the row metadata's write -- do not wait for it; the planners do,
        // and what the gather and epilogue warps touch comes behind the planners' barriers.  (The two instructions in every
        // warp cost the gather warps registers: the first layer of 128 mini-batches 1.81 -> 1.86 ms.)
        pdl_trigger();
        HopOfLane hops = {0, 0};
        if (ROWS < BM && !a.row_meta) hops = hop_of_lane(a);   // (the sample is older than the kernel before this one)
        pdl_wait();
        bool ok = true;
        for (uint32_t q = plw; ok; q += kPlanners) {
            if (q / kBlocks >= my_iters) break;
            const int64_t t = tile_of(q / kBlocks);   // past the end for the peer of an odd last tile: all padding
            const int slot = q % kPlanSlots;
            if (q >= (uint32_t)kPlanSlots && !mbar_wait(&plan_empty[slot], ((q / kPlanSlots) - 1) & 1)) {
                if (lane == 0) report(a.error, 17u);
                ok = false;
            }
            ok = __all_sync(0xFFFFFFFFu, ok);
            if (!ok) break;
            const int64_t r = a.row_lo + t * TM + (q % kBlocks) * kBlockRows + lane;
            int4 rm = make_int4(a.safe_src, 0, -1, 0);
            if (ROWS < BM && !a.row_meta) rm = row_of_sample<FIRST>(a, hops, (int32_t)r, r < a.M);
            else if (r < a.M) rm = __ldg(a.row_meta + r);   // (self source row, first entry, count, first H^{l-1} row of the batch)
            plan_block<FIRST>(a, keys, rm, meta[slot], src_rows[slot], first_rows[slot], &plan_total[slot]);
            if (lane == 0) mbar_arrive(&plan_full[slot]);
        }
    }
    } else if (warp >= kFirstEpilogueWarp) {
    MG_REG_SET(MG_REG_EPI);
    {
        // ---------------- epilogue: tensor memory -> bias, ReLU -> global ----------------
        // A half tile's accumulator: rows 0..63 of output columns [0, BN/2) in lanes 0..63, the same rows of columns
        // [BN/2, BN) in lanes 64..127.  Warp quadrant q reads lanes 32q..32q+31.
        const int lane_group = warp & 3;
        const int col_base = (lane_group >> 1) * half_n;
        const int n_cols = half_n;
        bool ok = true;
        if constexpr (TS) {
            // The accumulator of a half-tile pair: lane = output column (this CTA's 128), column j = row j of the
            // leader's half tile (j < 64) or row j - 64 of the peer's.  A warp turns 32 x 32 pieces round through its
            // staging tile (lane = column of the box, 128-byte swizzle) and stores them with TMA.
            const int n0 = (int)rank * 128 + lane_group * 32;
            const float bias_n = n0 + lane < a.N ? __ldg(a.bias + n0 + lane) : 0.f;
            uint8_t* stage = reinterpret_cast<uint8_t*>(out_stage[lane_group]);
            for (uint32_t hu = 0; hu < HALVES * my_iters && ok; ++hu) {
                const uint32_t buf = hu & 1;
                if (!mbar_wait(&acc_full[buf], (hu >> 1) & 1)) { if (lane == 0) report(a.error, 14u); ok = false; break; }
                tc_fence_after();
                for (int g = 0; g < 4; ++g) {
                    uint32_t v[32];
                    tmem_ld_32(tmem_base + kTsAcc0 + buf * kTsAccCols + ((uint32_t)(lane_group * 32) << 16) + (uint32_t)(g * 32), v);
                    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                    const int64_t t = 2 * ((int64_t)pair + (int64_t)(hu / HALVES) * n_pairs) + (g >> 1);   // the tile of CTA g / 2
                    const int64_t row0 = a.row_lo + t * TM + (hu % HALVES) * HM + (g & 1) * 32;
                    if (row0 >= a.M || n0 >= a.N || (ROWS < HM && (g & 1))) continue;
                    if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");   // the previous box has left the tile
                    __syncwarp();
#pragma unroll
                    for (int j = 0; j < 32; ++j) {
                        float o = __uint_as_float(v[j]) + bias_n;
                        if (a.relu) o = fmaxf(o, 0.f);
                        if (a.out_f16) *reinterpret_cast<__half*>(stage + j * 64 + lane * 2) = __float2half_rn(o);   // (boxes of 32 fp16 columns, not swizzled)
                        else *reinterpret_cast<float*>(stage + j * 128 + (((lane >> 2) ^ (j & 7)) << 4) + ((lane & 3) << 2)) = o;
                    }
                    if (KEEP && a.positive) {   // lane = column: a word for its 32 rows
                        uint32_t bits = 0;
#pragma unroll
                        for (int j = 0; j < 32; ++j) if (__uint_as_float(v[j]) + bias_n > 0.f) bits |= 1u << j;
                        if (n0 + lane < a.N) a.positive[(row0 >> 5) * a.N + n0 + lane] = bits;
                    }
                    fence_async_smem();
                    __syncwarp();
                    if (lane == 0) {
                        // rows past the end of the layer and columns past its width are clipped by the tensor map
                        tma_store_2d(&map_out, stage, n0, (int)row0);
                        if (a.out2) tma_store_2d(&map_out2, stage, n0, (int)row0);
                        asm volatile("cp.async.bulk.commit_group;" ::: "memory");
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) {
                    if (leader) mbar_arrive(&acc_empty[buf]);
                    else mbar_arrive_cluster(mapa_u32(smem_u32(&acc_empty[buf]), 0));
                }
            }
        }
        for (uint32_t hu = 0; !TS && hu < HALVES * my_iters && ok; ++hu) {
            const int64_t t = tile_of(hu / HALVES);
            const uint32_t buf = hu % kAccBufs;
            if (!mbar_wait(&acc_full[buf], (hu / kAccBufs) & 1)) { if (lane == 0) report(a.error, 14u); ok = false; break; }
            tc_fence_after();
            const int64_t row0 = a.row_lo + t * TM + (hu % HALVES) * HM + (lane_group & 1) * 32;
            uint8_t* stage = reinterpret_cast<uint8_t*>(out_stage[lane_group]);
            // 16 accumulator columns at a time (few registers); two such steps fill one 32-column fp32 box of the TMA
            // store, four a 64-column fp16 box
            for (int c0 = 0; c0 < n_cols; c0 += 16) {
                uint32_t v[16];
                tmem_ld_16(tmem_base + buf * acc_stride + ((uint32_t)(lane_group * 32) << 16) + (uint32_t)c0, v);
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                const int ncol0 = col_base + c0;   // first output column of this step
                if (row0 >= a.M || ncol0 >= a.N || (ROWS < HM && (lane_group & 1))) continue;
                if (KEEP && a.positive) {   // lane = row: 32 rows of a column are one vote, lane c keeps column c's
                    uint32_t bits = 0;
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        if (c0 + 4 * c >= n_cols || ncol0 + 4 * c >= a.N) break;
                        const float4 bb = __ldg(reinterpret_cast<const float4*>(a.bias + ncol0 + 4 * c));
                        const float b4[4] = {bb.x, bb.y, bb.z, bb.w};
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            const uint32_t w = __ballot_sync(0xFFFFFFFFu, __uint_as_float(v[4 * c + i]) + b4[i] > 0.f);
                            if (lane == 4 * c + i) bits = w;
                        }
                    }
                    if (lane < 16 && c0 + lane < n_cols && ncol0 + lane < a.N) a.positive[(row0 >> 5) * a.N + ncol0 + lane] = bits;
                }
                if (a.out_f16) {
                    // fp16 output (widths that are multiples of 128 only): 128 bytes per row and box, so a row of the next
                    // layer's input is again fetched in 512-byte requests
                    const int pbase = (c0 & 63) >> 3;    // first 16-byte piece (8 columns) of this step in the box's rows
                    if (pbase == 0) {
                        // the previous box's TMA store must have read the staging tile before it is rewritten
                        if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
                        __syncwarp();
                    }
#pragma unroll
                    for (int c = 0; c < 2; ++c) {
                        const int n = ncol0 + 8 * c;
                        const float4 b0 = __ldg(reinterpret_cast<const float4*>(a.bias + n)), b1 = __ldg(reinterpret_cast<const float4*>(a.bias + n + 4));
                        float o[8] = {__uint_as_float(v[8 * c]) + b0.x, __uint_as_float(v[8 * c + 1]) + b0.y, __uint_as_float(v[8 * c + 2]) + b0.z,
                                      __uint_as_float(v[8 * c + 3]) + b0.w, __uint_as_float(v[8 * c + 4]) + b1.x, __uint_as_float(v[8 * c + 5]) + b1.y,
                                      __uint_as_float(v[8 * c + 6]) + b1.z, __uint_as_float(v[8 * c + 7]) + b1.w};
                        uint32_t w[4];
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            const __half2 h = a.relu ? __floats2half2_rn(fmaxf(o[2 * i], 0.f), fmaxf(o[2 * i + 1], 0.f)) : __floats2half2_rn(o[2 * i], o[2 * i + 1]);
                            w[i] = *reinterpret_cast<const uint32_t*>(&h);
                        }
                        *reinterpret_cast<uint4*>(stage + lane * 128 + (((pbase + c) ^ (lane & 7)) << 4)) = make_uint4(w[0], w[1], w[2], w[3]);
                    }
                    if (pbase == 6) {
                        fence_async_smem();
                        __syncwarp();
                        if (lane == 0) {
                            tma_store_2d(&map_out, stage, ncol0 - 48, (int)row0);
                            asm volatile("cp.async.bulk.commit_group;" ::: "memory");
                        }
                    }
                } else if ((c0 & ~31) + 32 <= n_cols) {
                    const int pbase = (c0 & 31) >> 2;    // 0 or 4: first 16-byte piece (4 columns) of this step
                    if (pbase == 0) {
                        if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
                        __syncwarp();
                    }
                    // lane = row of the box; 16-byte piece c of the row goes to piece c ^ (row % 8) (128-byte swizzle)
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        const int n = ncol0 + 4 * c;
                        float4 o = make_float4(__uint_as_float(v[4 * c]), __uint_as_float(v[4 * c + 1]),
                                               __uint_as_float(v[4 * c + 2]), __uint_as_float(v[4 * c + 3]));
                        if (n < a.N) {
                            const float4 bb = __ldg(reinterpret_cast<const float4*>(a.bias + n));
                            o.x += bb.x; o.y += bb.y; o.z += bb.z; o.w += bb.w;
                        }
                        if (a.relu) { o.x = fmaxf(o.x, 0.f); o.y = fmaxf(o.y, 0.f); o.z = fmaxf(o.z, 0.f); o.w = fmaxf(o.w, 0.f); }
                        *reinterpret_cast<float4*>(stage + lane * 128 + (((pbase + c) ^ (lane & 7)) << 4)) = o;
                    }
                    if (pbase == 4) {
                        fence_async_smem();
                        __syncwarp();
                        if (lane == 0) {
                            // rows past the end of the layer and columns past its width are clipped by the tensor map
                            tma_store_2d(&map_out, stage, ncol0 - 16, (int)row0);
                            if (a.out2) tma_store_2d(&map_out2, stage, ncol0 - 16, (int)row0);
                            asm volatile("cp.async.bulk.commit_group;" ::: "memory");
                        }
                    }
                } else {
                    // the ragged end of the half (BN / 2 is not a multiple of 32): lane = row, plain stores
                    const int64_t row = row0 + lane;
                    if (row < a.M) {
#pragma unroll
                        for (int c = 0; c < 4; ++c) {
                            const int n = ncol0 + 4 * c;
                            if (c0 + 4 * c < n_cols && n < a.N) {
                                const float4 bb = __ldg(reinterpret_cast<const float4*>(a.bias + n));
                                float4 o = make_float4(__uint_as_float(v[4 * c]) + bb.x, __uint_as_float(v[4 * c + 1]) + bb.y,
                                                       __uint_as_float(v[4 * c + 2]) + bb.z, __uint_as_float(v[4 * c + 3]) + bb.w);
                                if (a.relu) { o.x = fmaxf(o.x, 0.f); o.y = fmaxf(o.y, 0.f); o.z = fmaxf(o.z, 0.f); o.w = fmaxf(o.w, 0.f); }
                                *reinterpret_cast<float4*>(a.out + row * a.N + n) = o;
                                if (a.out2) *reinterpret_cast<float4*>(a.out2 + row * a.N + n) = o;
                            }
                        }
                    }
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) {   // this accumulator buffer of this CTA is drained: tell the leader's MMA thread
                if (leader) mbar_arrive(&acc_empty[buf]);
                else mbar_arrive_cluster(mapa_u32(smem_u32(&acc_empty[buf]), 0));
            }
        }
    }
    } else {
    MG_REG_SET(MG_REG_PROD);
    {
        // ---------------- producers: gather + segment mean -> swizzled A slices ----------------
        // K slices come in groups of eight: (self, mean) pairs for four consecutive 32-column blocks, i.e. 128
        // columns of the input rows.  A tile is built in rounds of 32 rows (a row block, planned ahead by the
        // planner warps): a warp builds two rows per round from whole 512-byte row segments (lane L owns columns
        // 4L..4L+3 of the group) and keeps 2 x (1 + kUnroll) loads in flight per lane -- memory-level parallelism
        // comes from registers.  Each lane scatters its 16-byte pieces into the group's stages: slice pair L / 8,
        // slot L % 8.  Producer warps only meet at the mbarriers, never at a block-wide barrier.
        const int pw = warp - kFirstProducerWarp;     // 0 .. kProducerWarps-1
        const int gl = lane & 7;                      // 16-byte slot inside a 128-byte slice row
        bool ok = true;
        for (uint32_t it = 0; it < my_iters; ++it) {
            for (int grp = 0; grp < n_groups; ++grp) {
                const uint32_t s_h = it * (uint32_t)n_groups + (uint32_t)grp;   // fills of each half's stage rows so far
                const int pairs = min(GC / KCE, (a.d_in_pad - grp * GC) / KCE);   // slice pairs in this group
                const int col = grp * GC + lane * LC;
                const bool lane_on = (lane >> 3) < pairs;
                const bool col_ok = lane_on && col < a.d_in;
                const char* src = a.src_base + (size_t)col * (HALF ? 2 : 4);
                for (int blk = 0; blk < kBlocks; ++blk) {
                    const int h = blk / kHalfBlocks;               // the half tile this block belongs to
                    const uint32_t q = it * kBlocks + blk;     // row block counter of this CTA
                    const int slot = q % kPlanSlots;
                    if (grp == 0 && ok && !mbar_wait(&plan_full[slot], (q / kPlanSlots) & 1)) {
                        if (lane == 0) report(a.error, 16u);
                        ok = false;
                    }
                    ok = __all_sync(0xFFFFFFFFu, ok);
                    const bool cached = plan_total[slot] >= 0;
                    const int32_t* rows_of = src_rows[slot];
                    const int brow = pw * kRowsInFlight;              // this warp's first row inside the block
                    uint4 selfv[kRowsInFlight], meanv[kRowsInFlight];   // the two operand pieces of each row
                    constexpr bool kKeepAgg = KEEP && !FIRST;
                    float* keep = kKeepAgg && a.kept_agg ? a.kept_agg + (a.row_lo + tile_of(it) * TM + blk * kBlockRows + brow) * a.d_in + col : nullptr;
                    gather_rows<FIRST, HALF, F16, false, kKeepAgg>(a, src, col_ok && ok, cached, &meta[slot][brow], &first_rows[slot][brow], rows_of, selfv, meanv, keep);
                    if (grp == n_groups - 1) {
                        // the block's plan has been read for the last time: its slot may be planned again
                        __syncwarp();
                        if (lane == 0) mbar_arrive(&plan_empty[slot]);
                    }
                    if (blk % kHalfBlocks == 0) {
                        // the half's rows of the stages must have been read by the MMAs of their previous fill (one
                        // commit frees them all); those MMAs ran while the other half was gathered, and the loads
                        // above are already in flight while this waits
                        if (ok && s_h >= 1 && !mbar_wait(&a_free[h], (s_h - 1) & 1)) {
                            if (lane == 0) report(a.error, 15u);
                            ok = false;
                        }
                        ok = __all_sync(0xFFFFFFFFu, ok);
                    }
                    if (ok && lane_on) {
                        // K-major, 128-byte swizzle: 16-byte slot gl of row r lands in slot gl ^ (r % 8)
                        const uint32_t s_self = 2 * (lane >> 3), s_mean = 2 * (lane >> 3) + 1;   // the group's slice = its stage
                        uint8_t* stage_self = a_base + (size_t)s_self * kStage;
                        uint8_t* stage_mean = a_base + (size_t)s_mean * kStage;
#pragma unroll
                        for (int q2 = 0; q2 < kRowsInFlight; ++q2) {
                            const int row = blk * kBlockRows + brow + q2;
                            const size_t off = (size_t)(row >> 3) * 1024 + (size_t)(row & 7) * 128 + (size_t)((gl ^ (row & 7)) << 4);
                            *reinterpret_cast<uint4*>(stage_self + off) = selfv[q2];
                            *reinterpret_cast<uint4*>(stage_mean + off) = meanv[q2];
                        }
                    }
                    if (blk % kHalfBlocks == kHalfBlocks - 1) {
                        // this warp's rows of the half are in place: tell the leader's MMA thread
                        fence_async_smem();
                        __syncwarp();
                        if (ok && lane == 0) {
                            if (leader) mbar_arrive(&a_ready[h]);
                            else mbar_arrive_cluster(mapa_u32(smem_u32(&a_ready[h]), 0));
                        }
                    }
                }
            }
        }
    }
    }
    if (warp >= kFirstEpilogueWarp && warp < kTmaWarp && lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
    tc_fence_before();
    cluster_sync_all();   // neither CTA leaves (or frees tensor memory) while the other may still signal or read it
    if (warp == kMmaWarp) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"((uint32_t)a.tmem_cols) : "memory");
    }
}

// ---- weight gradients: dW += [self | aggregate]^T dPre --------------------------------------------------------------------
// The layer's operand is brought together block by block of 32 rows in shared memory, and contracted over the rows with the gradient
// rows that TMA brings: self rows are gathered, aggregates are gathered or, where the forward pass has left them (KEPT), come by TMA.
// (Before: an aggregation kernel wrote all of it, 1 to 2 KB per row, and a product over split chunks read it back.)  Bound by the gather like the forward layer.  A CTA owns 128 input columns -- their
// self and aggregate halves are the two M = 128 tiles of its accumulators, all 512 columns of tensor memory with 256 output
// columns -- and every n_slices-th block of rows; at the end it adds its 256 x 256 sums to dW with 16-byte reductions.  24 mini-batches of
// 1,000 targets on 2M nodes: 540k rows of 2 x 128 in 252 us (257 + 190 before), 91k + 24k rows of 2 x 256 in 188 us (178 + 100).
// Both operands lie with the contraction across rows ("MN-major"): boxes of 32 rows x 32 floats, swizzled in 32-byte units.
//   warps 0..15  gather, two rows each per block     warps 16..19  planners     warp 20  TMA     warp 21  MMA, tensor memory
constexpr int kGradPlanners = 4, kGradFirstPlanner = 16, kGradTmaWarp = 20, kGradMmaWarp = 21;
constexpr int kGradThreads = (kGradMmaWarp + 1) * 32;   // 704
// (two stages leave the gathers 92 KB of L1: the MMAs of a block take a fifth of its gather; kept aggregates come by TMA, three deep)
__host__ __device__ constexpr int grad_stages(bool kept) { return kept ? 3 : 2; }
constexpr uint32_t kGradBox = kBlockRows * 128, kGradStageX = 8 * kGradBox;

struct GradWArgs {
    FusedArgs f;          // rows, entries, sources of the layer; N, d_in, M
    int32_t n_slices, col_groups, n_cols;   // n_cols: output columns of a CTA, a multiple of 32, at most 256
    float* dw;            // [2 d_in, N]
};

// KEPT: the forward pass has left the aggregates (FusedArgs::kept_agg).  They lie as they are wanted, so TMA brings them like the gradient
// rows, and the gather warps read the rows themselves only (92k + 24k rows of 2 x 256: 183 -> 110 us, 34k + 8k: 98 -> 62).
template <bool FIRST, bool HALF, bool KEPT>
__global__ void __launch_bounds__(kGradThreads, 1) k_sage_grad_weights(const __grid_constant__ CUtensorMap map_g, const __grid_constant__ CUtensorMap map_x,
                                                                       GradWArgs p) {
    constexpr int kGradStages = grad_stages(KEPT);
    extern __shared__ uint8_t smem_raw[];
    __shared__ uint64_t x_ready[kGradStages], g_full[kGradStages], stage_free[kGradStages], acc_full;
    __shared__ uint64_t plan_full[kPlanSlots], plan_empty[kPlanSlots];
    __shared__ uint32_t tmem_slot;
    __shared__ RowMeta meta[kPlanSlots][kBlockRows];
    __shared__ int32_t src_rows[kPlanSlots][kKeyCap];
    __shared__ int32_t plan_total[kPlanSlots];
    __shared__ __align__(16) int32_t first_rows[kPlanSlots][kBlockRows][8];
    const FusedArgs& a = p.f;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int col0 = (int)(blockIdx.y % p.col_groups) * kGroupCols, n0 = (int)(blockIdx.y / p.col_groups) * 256;
    const int bn = min(p.n_cols, (a.N - n0 + 31) / 32 * 32);
    uint8_t* x_base = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint8_t* g_base = x_base + kGradStages * kGradStageX;
    const uint32_t g_bytes = (uint32_t)(p.n_cols / 32) * kGradBox;   // a stage of gradient rows
    const int64_t blocks = (a.M + kBlockRows - 1) / kBlockRows;
    const uint32_t my = (int64_t)blockIdx.x < blocks ? (uint32_t)((blocks - blockIdx.x + p.n_slices - 1) / p.n_slices) : 0u;
    auto first_row = [&](uint32_t it) -> int64_t { return ((int64_t)blockIdx.x + (int64_t)it * p.n_slices) * kBlockRows; };

    if (threadIdx.x == 0) {
        for (int s = 0; s < kGradStages; ++s) { mbar_init(&x_ready[s], kProducerWarps); mbar_init(&g_full[s], 1); mbar_init(&stage_free[s], 1); }
        mbar_init(&acc_full, 1);
        for (int s = 0; s < kPlanSlots; ++s) { mbar_init(&plan_full[s], 1); mbar_init(&plan_empty[s], kProducerWarps); }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(&map_g) : "memory");
    }
    if (warp == kGradMmaWarp) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)), "r"((uint32_t)a.tmem_cols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = tmem_slot;
    const uint32_t acc_cols = (uint32_t)a.tmem_cols / 2;   // the aggregate half's accumulator starts here

    if (warp < kProducerWarps) {
        const int col = col0 + lane * 4;
        const bool col_ok = col < a.d_in;
        const char* src = a.src_base + (size_t)col * (HALF ? 2 : 4);
        const int brow = warp * kRowsInFlight;
        bool ok = true;
        for (uint32_t it = 0; it < my; ++it) {
            const int slot = it % kPlanSlots, s = it % kGradStages;
            if (ok && !mbar_wait(&plan_full[slot], (it / kPlanSlots) & 1)) { if (lane == 0) report(a.error, 41u); ok = false; }
            ok = __all_sync(0xFFFFFFFFu, ok);
            if (!ok) break;
            uint4 selfv[kRowsInFlight], meanv[kRowsInFlight];
            if (KEPT) {
#pragma unroll
                for (int q = 0; q < kRowsInFlight; ++q)
                    selfv[q] = col_ok ? load_piece<HALF, false>(src + (size_t)(uint32_t)meta[slot][brow + q].x * (size_t)a.src_row_bytes) : make_uint4(0u, 0u, 0u, 0u);
            } else {
                gather_rows<FIRST, HALF, false, true>(a, src, col_ok, plan_total[slot] >= 0, &meta[slot][brow], &first_rows[slot][brow], src_rows[slot], selfv, meanv);
            }
#pragma unroll
            for (int q = 0; q < kRowsInFlight; ++q)   // a row past the end meets a gradient row of zeros: it only has to be finite
                if (meta[slot][brow + q].z < 0) selfv[q] = make_uint4(0u, 0u, 0u, 0u);
            __syncwarp();
            if (lane == 0) mbar_arrive(&plan_empty[slot]);
            if (it >= (uint32_t)kGradStages && !mbar_wait(&stage_free[s], ((it / kGradStages) - 1) & 1)) { if (lane == 0) report(a.error, 42u); ok = false; }
            ok = __all_sync(0xFFFFFFFFu, ok);
            if (!ok) break;
            if (col_ok) {
                // box lane / 8 of the half; the 32-byte pieces of a row are exchanged by the row number mod 4
                uint8_t* xs = x_base + (size_t)s * kGradStageX + (size_t)(lane >> 3) * kGradBox;
#pragma unroll
                for (int q = 0; q < kRowsInFlight; ++q) {
                    const int row = brow + q;
                    const size_t off = (size_t)row * 128 + (size_t)((((lane & 7) >> 1) ^ (row & 3)) << 5) + (size_t)((lane & 1) << 4);
                    *reinterpret_cast<uint4*>(xs + off) = selfv[q];
                    if (!KEPT) *reinterpret_cast<uint4*>(xs + 4 * kGradBox + off) = meanv[q];
                }
            }
            fence_async_smem();
            __syncwarp();
            if (lane == 0) mbar_arrive(&x_ready[s]);
        }
        // the CTA's sums: warp = a quarter of the accumulators' lanes (input columns) x every fourth 32 output columns
        if (my > 0 && ok) {
            ok = mbar_wait(&acc_full, 0);
            if (!ok && lane == 0) report(a.error, 43u);
            ok = __all_sync(0xFFFFFFFFu, ok);
            tc_fence_after();
            const int quarter = warp & 3, c = col0 + quarter * 32 + lane;
            for (int part = 0; part < 2 && ok; ++part)
                for (int j0 = (warp >> 2) * 32; j0 < bn; j0 += 128) {
                    uint32_t v[32];
                    tmem_ld_32(tmem_base + part * acc_cols + ((uint32_t)(quarter * 32) << 16) + (uint32_t)j0, v);
                    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                    if (c >= a.d_in) continue;
                    float4* dst = reinterpret_cast<float4*>(p.dw + (int64_t)(part * a.d_in + c) * a.N + n0 + j0);
#pragma unroll
                    for (int j = 0; j < 8; ++j)
                        if (n0 + j0 + 4 * j < a.N)
                            atomicAdd(dst + j, make_float4(__uint_as_float(v[4 * j]), __uint_as_float(v[4 * j + 1]), __uint_as_float(v[4 * j + 2]),
                                                           __uint_as_float(v[4 * j + 3])));
                }
        }
    } else if (warp < kGradTmaWarp) {
        const int32_t* keys = FIRST ? a.ent_nbrs : a.ent_repr;
        bool ok = true;
        for (uint32_t it = warp - kGradFirstPlanner; it < my; it += kGradPlanners) {
            const int slot = it % kPlanSlots;
            if (it >= (uint32_t)kPlanSlots && !mbar_wait(&plan_empty[slot], ((it / kPlanSlots) - 1) & 1)) { if (lane == 0) report(a.error, 44u); ok = false; }
            ok = __all_sync(0xFFFFFFFFu, ok);
            if (!ok) break;
            const int64_t r = first_row(it) + lane;
            int4 rm = make_int4(a.safe_src, 0, -1, 0);
            if (r < a.M) rm = __ldg(a.row_meta + r);
            if (KEPT) {
                meta[slot][lane] = rm;
                __syncwarp();
            } else {
                plan_block<FIRST>(a, keys, rm, meta[slot], src_rows[slot], first_rows[slot], &plan_total[slot]);
            }
            if (lane == 0) mbar_arrive(&plan_full[slot]);
        }
    } else if (warp == kGradTmaWarp) {
        if (lane == 0) {
            const int n_agg = KEPT ? min(4, (a.d_in - col0 + 31) / 32) : 0;   // boxes of this CTA's input columns
            uint32_t it = 0;
            for (; it < my; ++it) {
                const int s = it % kGradStages;
                if (it >= (uint32_t)kGradStages && !mbar_wait(&stage_free[s], ((it / kGradStages) - 1) & 1)) { report(a.error, 45u); break; }
                mbar_expect_tx(&g_full[s], (uint32_t)(bn / 32 + n_agg) * kGradBox);
                for (int j = 0; j < bn / 32; ++j)   // (rows past the end and columns past the width come as zeros)
                    tma_load_2d(g_base + (size_t)s * g_bytes + (size_t)j * kGradBox, &map_g, &g_full[s], n0 + 32 * j, (int)first_row(it));
                for (int j = 0; j < n_agg; ++j)
                    tma_load_2d(x_base + (size_t)s * kGradStageX + (size_t)(4 + j) * kGradBox, &map_x, &g_full[s], col0 + 32 * j, (int)first_row(it));
            }
            // nothing of this CTA's may be in flight when it ends
            for (uint32_t i = it >= (uint32_t)kGradStages ? it - kGradStages : 0; i < it; ++i)
                if (!mbar_wait(&g_full[i % kGradStages], (i / kGradStages) & 1)) report(a.error, 46u);
        }
        __syncwarp();
    } else {
        if (lane == 0 && my > 0) {
            // fp32 accumulate, TF32 x TF32, the contiguous dimension of both operands is M (N): bits 15 and 16
            const uint32_t idesc = (1u << 4) | (2u << 7) | (2u << 10) | (1u << 15) | (1u << 16) | ((uint32_t)(bn >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
            bool ok = true;
            for (uint32_t it = 0; it < my && ok; ++it) {
                const int s = it % kGradStages;
                if (!mbar_wait(&g_full[s], (it / kGradStages) & 1) || !mbar_wait(&x_ready[s], (it / kGradStages) & 1)) { report(a.error, 47u); ok = false; break; }
                tc_fence_after();
                const uint64_t db = smem_desc_sw128_mn(smem_u32(g_base + (size_t)s * g_bytes), kGradBox);
                for (int part = 0; part < 2; ++part) {
                    const uint64_t da = smem_desc_sw128_mn(smem_u32(x_base + (size_t)s * kGradStageX + (size_t)part * 4 * kGradBox), kGradBox);
#pragma unroll
                    for (int kk = 0; kk < kBlockRows / 8; ++kk)   // 8 rows of every box = 1024 bytes further on
                        mma_tf32(tmem_base + part * acc_cols, da + (uint64_t)(kk * 64), db + (uint64_t)(kk * 64), idesc, (it | kk) ? 1u : 0u);
                }
                mma_commit(&stage_free[s]);
            }
            if (ok) mma_commit(&acc_full);
        }
        __syncwarp();
    }
    tc_fence_before();
    __syncthreads();
    if (warp == kGradMmaWarp) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"((uint32_t)a.tmem_cols) : "memory");
    }
}

// Pre-pass: for every output row of every layer, where its own representation lives and which entries it aggregates.  One
// thread per row, full occupancy; the fused kernels then need a single coalesced load per row instead of a chain of dependent
// look-ups.  One launch for all layers (one mini-batch, three layers: three launches of 2 us and their gaps before).
struct RowsArgs {
    int32_t B, k;
    const int32_t* rowbase;      // [(k + 1)][B + 1]
    const int32_t* cum;          // [B][k + 2]
    const int32_t* node_off;     // [(k + 1)][B + 1]
    const int32_t* nodes;
    const int32_t* ent_off;
    FeatGeom feat;
    int64_t start[MG_MAX_HOPS + 2];   // layer l's rows go to meta[start[l] .. start[l + 1])
};
__global__ void __launch_bounds__(256) k_layer_rows(RowsArgs a, int4* __restrict__ meta) {
    pdl_trigger();
    const int64_t total = a.start[a.k + 1];
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
        int layer = 1;
        while (i >= a.start[layer + 1]) ++layer;
        const int32_t* rb = a.rowbase + (int64_t)layer * (a.B + 1);
        const int32_t r = (int32_t)(i - a.start[layer]);
        const int b = upper_segment(rb, a.B + 1, r);
        const int32_t l = r - rb[b];
        const int32_t* cum = a.cum + b * (a.k + 2);
        int h = 0;
        while (h < a.k - layer && l >= cum[h + 1]) ++h;
        const int32_t idx = a.node_off[h * (a.B + 1) + b] + (l - cum[h]);
        const int32_t e0 = a.ent_off[idx];
        const int32_t in_base = rb[b - (a.B + 1)];
        meta[i] = make_int4(layer == 1 ? (int32_t)feat_row(a.feat, a.nodes[idx]) : in_base + l, e0, a.ent_off[idx + 1] - e0, in_base);
    }
}

// row-major [rows, K] fp16 matrix in boxes of 32 halves x 32 rows, not swizzled (the transposed epilogue's fp16 stores)
static bool make_map_f16_box32(CUtensorMap* map, const void* base, int64_t rows, int K) {
    EncodeTiledFn enc = get_encode();
    if (!enc) return false;
    const cuuint64_t dims[2] = {(cuuint64_t)K, (cuuint64_t)rows};
    const cuuint64_t strides[1] = {(cuuint64_t)K * 2};
    const cuuint32_t box[2] = {32u, 32u};
    const cuuint32_t estr[2] = {1, 1};
    return enc(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}
// the same in boxes of 64 halves x box_rows, 128-byte swizzle, zero fill
static bool make_map_f16(CUtensorMap* map, const void* base, int64_t rows, int K, int box_rows) {
    EncodeTiledFn enc = get_encode();
    if (!enc) return false;
    const cuuint64_t dims[2] = {(cuuint64_t)K, (cuuint64_t)rows};
    const cuuint64_t strides[1] = {(cuuint64_t)K * 2};
    const cuuint32_t box[2] = {64u, (cuuint32_t)box_rows};
    const cuuint32_t estr[2] = {1, 1};
    return enc(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace

bool mg_layer_fused_supported(int d_in, int d_out) { return d_out <= 256 && d_out % 4 == 0 && d_in % 4 == 0; }

// Rows of a layer's tiles.  Halves per tile: the CTA pair with the most rows sets the time, and a row of a one-half tile costs about a seventh
// more where its pair has several of them.  (The three layers of one mini-batch on 1M nodes, 23,400, 4,300 and 1,000 rows: 93 us in
// 128-row tiles, the whole call 214 -> 195 us; 128 mini-batches keep them: 4.0 ms either way.)
static int mg_layer_tile(const mg_ctx* ctx, int64_t rows) {
    const int64_t pairs = ctx->n_sms / 2;
    const int64_t rounds1 = (rows + 2 * HM * pairs - 1) / (2 * HM * pairs), rounds2 = (rows + 4 * HM * pairs - 1) / (4 * HM * pairs);
    return rows <= 2 * kBlockRows * pairs ? kBlockRows : rounds1 * 8 < rounds2 * 14 ? HM : BM;
}

// Whether a layer of 9 to 16 entries per row and at most 128 output columns keeps its weights in tensor memory, by what it gains there (time with
// them there over time with them streamed; 9 and 16 entries, 600 to 130,000 rows, 16 to 256 input columns, fp32 and fp16 rows).  For it: no slice is
// waited for, and half the epilogue of a wider layer.  Against it: all weights have to be there before a tile's first product.  That shows in the
// one tile that a CTA has of a small first layer (a later layer's weights come in beside the layer before), and where there are no more slices than the
// ring holds (n_chunks = 2), which arrive in time anyway.
//   32-row tiles                      0.80 - 1.04; first layers of fp32 rows wider than 64 into more than 112 columns 0.98 - 1.06
//   first layers, one tile per CTA    more than four slices and up to 112 columns 0.90 - 1.04, else 0.95 - 1.10
//   ... several                       two slices 0.93 - 1.01 (65 to 112 columns) and 0.98 - 1.05 (others), more 0.88 - 1.03
//   later layers                      two slices and one tile per CTA 0.96 - 1.05, else 0.80 - 1.03; that leave aggregates for the backward pass: up to
//                                     four slices in 128-row tiles 1.02 - 1.08, else 0.81 - 1.01
static bool mg_layer_narrow_ts(bool first, bool keep, bool f16, int n_chunks, int d_out, int tile_rows, bool one_tile) {
    const bool two = n_chunks <= 2, wide = d_out > 112;
    if (tile_rows == kBlockRows) return !first || !wide || f16 || n_chunks <= 4;
    if (!first) return n_chunks > 4 || (keep ? tile_rows == HM : !two || !one_tile);
    return one_tile ? n_chunks > 4 && !wide : !two || (d_out > 64 && !wide);
}

bool mg_layer_rows_inline(const mg_ctx* ctx, const mg_dense* d) {
    if (d->n_batches != 1) return false;
    for (int l = 1; l <= d->k; ++l)
        if (mg_layer_tile(ctx, d->h_hdr.rows_total[l]) == BM) return false;
    return true;
}

static void fill_args(mg_ctx* ctx, const mg_dense* d, int layer, int d_in, int d_out, FusedArgs* pa) {
    FusedArgs& a = *pa;
    const int B = d->n_batches;
    a.B = B; a.k = d->k; a.layer = layer;
    a.rowbase_out = d->rowbase + (size_t)layer * (B + 1);
    a.rowbase_in = d->rowbase + (size_t)(layer - 1) * (B + 1);
    a.cum = d->cum; a.node_off = d->node_off; a.nodes = d->nodes;
    a.ent_off = d->ent_off; a.ent_nbrs = d->ent_nbrs; a.ent_repr = d->ent_repr;
    a.feat = mg_feat_geom(ctx);
    a.d_in = d_in;
    a.d_in_pad = (d_in + KC - 1) / KC * KC;
    a.N = d_out;
    a.BN = (d_out + 15) / 16 * 16;
    a.row_lo = 0;
    a.M = d->h_hdr.rows_total[layer];
    a.error = ctx->d_flags;
}

// Pre-pass of a forward pass: meta[start[l] + r] for every packed output row r of every layer l = 1 .. k.
int mg_layer_rows(mg_ctx* ctx, const mg_dense* d, int4* meta, const int64_t* start) {
    RowsArgs a;
    a.B = d->n_batches; a.k = d->k;
    a.rowbase = d->rowbase; a.cum = d->cum; a.node_off = d->node_off; a.nodes = d->nodes; a.ent_off = d->ent_off;
    a.feat = mg_feat_geom(ctx);
    for (int l = 1; l <= d->k + 1; ++l) a.start[l] = start[l];
    const int64_t total = start[d->k + 1];
    if (total <= 0) return MG_OK;
    k_layer_rows<<<(int)std::min<int64_t>(mg_grid(ctx, 8), (total + 255) / 256), 256, 0, ctx->stream>>>(a, meta);
    ctx->launches++;
    return MG_OK;
}

// Runs layer `layer` (1-based) for the packed output rows [row_lo, row_hi).  h_prev and h_out are indexed by
// GLOBAL packed row (callers that keep only a window of a layer pass pointers shifted accordingly).  h_out2 (nullable, 16-byte
// aligned): receives the same rows.  positive (nullable): mg_positive_words of the layer; kept_agg (nullable, layers >= 2):
// [rows of the layer, d_in].  row_meta: the layer's part of mg_layer_rows' result, or null where mg_layer_rows_inline says so.  The kernel is
// launched as a programmatic dependent of the one queued before it where that is mg_layer_rows' or another layer's: all layers but a
// first one without row_meta, whose weights the kernel before it may have written.
int mg_layer_fused(mg_ctx* ctx, const mg_dense* d, int layer, int d_in, int d_out, const float* w_pad_t, const float* bias,
                   const float* h_prev, float* h_out, float* h_out2, int flags, const int4* row_meta, int64_t row_lo, int64_t row_hi,
                   int64_t safe_src_row, const void* w_pad_h, int in_f16, int out_f16, uint32_t* positive, float* kept_agg) {
    if (row_hi <= row_lo) return MG_OK;
    FusedArgs a;
    memset(&a, 0, sizeof(a));
    fill_args(ctx, d, layer, d_in, d_out, &a);
    a.row_lo = row_lo;
    a.M = row_hi;
    a.row_meta = row_meta;
    a.safe_src = (int32_t)safe_src_row;
    a.h_prev = h_prev;
    a.src_base = layer == 1 ? ctx->slots : reinterpret_cast<const char*>(h_prev);
    a.src_row_bytes = layer == 1 ? (uint32_t)ctx->row_bytes : (uint32_t)d_in * (in_f16 ? 2u : 4u);
    a.out_f16 = out_f16;
    a.relu = flags & 1;
    a.sum_aggr = (flags >> 1) & 1;
    a.bias = bias; a.out = h_out; a.out2 = h_out2; a.positive = positive; a.kept_agg = kept_agg;
    // fp16 operands: first layer over fp16 base representations, mean aggregator (a sum of fp16 values may leave the
    // fp16 range), weights given in fp16 form (the caller withholds them when they do not suit fp16)
    // (later layers: in_f16 says that H^{l-1} was stored as fp16; the caller only does that with fp16 weights at hand)
    const bool f16 = (layer == 1 ? ctx->feat_dtype == MG_DTYPE_F16 : in_f16 != 0) && w_pad_h && !a.sum_aggr;
    if (layer > 1 && in_f16 && !f16) return mg_fail(ctx, MG_ERR_STATE, "fp16 layer input without fp16 operands");
    if (out_f16 && d_out % 128 != 0) return mg_fail(ctx, MG_ERR_STATE, "fp16 layer outputs need widths that are multiples of 128");
    const int kce = f16 ? 64 : KC;
    a.d_in_pad = (d_in + kce - 1) / kce * kce;
    int stride = 32;
    while (stride < a.BN / 2) stride <<= 1;
    a.tmem_cols = kAccBufs * stride;   // accumulator buffers of half tiles: BN / 2 columns each, a power of two >= 32
    const int b_bytes = (a.BN / 2) * 128;       // each CTA of a pair stages half of the output columns
    const int n_chunks = 2 * a.d_in_pad / kce;
    a.sa = std::min(8, n_chunks);   // one group of (self, mean) slice pairs: 128 input columns
    const int64_t rows = row_hi - row_lo, pairs = ctx->n_sms / 2;
    const int tile_rows = mg_layer_tile(ctx, rows), halves = tile_rows > HM ? 2 : 1;
    a.sb = std::max(2, std::min({kMaxStages, n_chunks, ring_bytes(halves) / b_bytes}));
    // weights in tensor memory: TF32 operands, fp32 output, all of K in 256 columns, at most 256 output columns
    // ... and rows with few entries: a half tile of long rows is gathered for longer than its weight slices take to
    // arrive, so the stream costs nothing there, while the transposed epilogue does (measured: 5.3 entries per row,
    // 2.03 -> 1.92 ms with the weights in tensor memory; 20 per row, 0.83 -> 0.90 ms).  Up to 128 output columns: mg_layer_narrow_ts
    // (71,000 rows of 11 entries, 100 -> 100 columns, 92 -> 87 us)
    const bool first = layer == 1, half = first && ctx->feat_dtype == MG_DTYPE_F16, keep = positive || kept_agg;
    const int64_t n_tiles = (rows + tile_rows - 1) / tile_rows;
    const int64_t layer_entries = d->h_hdr.ent_base[d->k - layer + 1], layer_rows = d->h_hdr.rows_total[layer];
    const bool few = layer_entries <= kTsMaxEntriesPerRow * layer_rows || (d_out <= 128 && layer_entries <= kTsMaxEntriesNarrow * layer_rows &&
                                                                          mg_layer_narrow_ts(first, keep, f16, n_chunks, d_out, tile_rows, n_tiles <= 2 * pairs));
    const bool ts = n_chunks <= 8 && d_out <= 256 && few && !getenv("MG_FUSED_NO_TS");
    if (ts) { a.tmem_cols = 512; a.sb = 0; a.w_rows = f16 ? (const void*)w_pad_h : (const void*)w_pad_t; }
    const size_t smem = (size_t)a.sa * stage_bytes(halves) + (size_t)a.sb * b_bytes + 1024;
    CUtensorMap mw;
    if (!(f16 ? make_map_f16(&mw, w_pad_h, d_out, 2 * a.d_in_pad, a.BN / 2) : make_map_f32(&mw, w_pad_t, d_out, 2 * a.d_in_pad, a.BN / 2)))
        return mg_fail(ctx, MG_ERR_CUDA, "cuTensorMapEncodeTiled failed for the layer weights");
    // output [row_hi rows, d_out] fp32, 32 x 32 boxes, 128-byte swizzle; rows are global packed rows, so a window's
    // shifted base pointer works unchanged (rows below row_lo are never stored)
    CUtensorMap mo;
    if (!(out_f16 ? (ts ? make_map_f16_box32(&mo, h_out, row_hi, d_out) : make_map_f16(&mo, h_out, row_hi, d_out, 32))
                  : make_map_f32(&mo, h_out, row_hi, d_out, 32)))
        return mg_fail(ctx, MG_ERR_CUDA, "cuTensorMapEncodeTiled failed for the layer output");
    CUtensorMap mo2 = mo;
    if (h_out2 && (out_f16 || !make_map_f32(&mo2, h_out2, row_hi, d_out, 32)))
        return mg_fail(ctx, MG_ERR_CUDA, "cuTensorMapEncodeTiled failed for the layer output");
    typedef void (*Kernel)(CUtensorMap, CUtensorMap, CUtensorMap, FusedArgs);
    // (kept outputs are fp32: fp16 rows as a later layer's input have no instance that keeps)
#define MG_FUSED_KERNELS(TS, ROWS, KEEP) \
    k_sage_layer_fused<true, false, false, TS, ROWS, KEEP>, k_sage_layer_fused<true, true, false, TS, ROWS, KEEP>, \
    k_sage_layer_fused<true, true, true, TS, ROWS, KEEP>, k_sage_layer_fused<false, false, false, TS, ROWS, KEEP>
#define MG_FUSED_FORMS(TS, ROWS) {MG_FUSED_KERNELS(TS, ROWS, false), k_sage_layer_fused<false, true, true, TS, ROWS, false>, MG_FUSED_KERNELS(TS, ROWS, true)}
    static const Kernel kernels[3][2][9] = {{MG_FUSED_FORMS(false, kBlockRows), MG_FUSED_FORMS(true, kBlockRows)}, {MG_FUSED_FORMS(false, HM), MG_FUSED_FORMS(true, HM)},
                                            {MG_FUSED_FORMS(false, BM), MG_FUSED_FORMS(true, BM)}};
#undef MG_FUSED_FORMS
#undef MG_FUSED_KERNELS
    if (keep && (in_f16 || out_f16)) return mg_fail(ctx, MG_ERR_STATE, "fp16 layer outputs are not kept");
    const int which = (first ? (f16 ? 2 : half ? 1 : 0) : (f16 ? 4 : 3)) + (keep ? 5 : 0);
    const Kernel kern = kernels[tile_rows == BM ? 2 : tile_rows == HM ? 1 : 0][ts][which];
    MG_CUDA(ctx, mg_smem_limit(ctx, (const void*)kern, fused_smem_limit(halves)));
    const int grid = 2 * (int)std::min<int64_t>((n_tiles + 1) / 2, pairs);   // CTA pairs
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid); cfg.blockDim = dim3(kFusedThreads); cfg.dynamicSmemBytes = smem; cfg.stream = ctx->stream;
    cudaLaunchAttribute pdl;
    pdl.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    pdl.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &pdl; cfg.numAttrs = layer > 1 || row_meta ? 1 : 0;
    MG_CUDA(ctx, cudaLaunchKernelEx(&cfg, kern, mw, mo, mo2, a));
    ctx->launches++;
    MG_CUDA(ctx, cudaGetLastError());
    return MG_OK;
}

// dw [2 d_in, d_out] += X^T dpre over the packed rows of layer `layer`, X = [self | aggregate]; row_meta: the layer's part of
// mg_layer_rows' result.  dpre: DEVICE [rows, d_out], 16-byte aligned.  kept_agg (nullable, layers >= 2): what mg_layer_fused left.
int mg_layer_grad_weights(mg_ctx* ctx, const mg_dense* d, int layer, int d_in, int d_out, const float* h_prev, const float* dpre, const int4* row_meta,
                          int sum_aggr, const float* kept_agg, float* dw) {
    GradWArgs p;
    memset(&p, 0, sizeof(p));
    FusedArgs& a = p.f;
    fill_args(ctx, d, layer, d_in, d_out, &a);
    if (a.M <= 0) return MG_OK;
    a.row_meta = row_meta;
    a.src_base = layer == 1 ? ctx->slots : reinterpret_cast<const char*>(h_prev);
    a.src_row_bytes = layer == 1 ? (uint32_t)ctx->row_bytes : (uint32_t)d_in * 4u;
    a.sum_aggr = sum_aggr;
    p.n_cols = std::min(256, (d_out + 31) / 32 * 32);
    int cols = 32;
    while (cols < p.n_cols) cols <<= 1;
    a.tmem_cols = 2 * cols;
    p.col_groups = (d_in + kGroupCols - 1) / kGroupCols;
    const int groups = p.col_groups * ((d_out + 255) / 256);
    // a CTA per SM; below eight blocks of rows each, the sums' way into dW would cost more than the rows
    const int64_t blocks = (a.M + kBlockRows - 1) / kBlockRows;
    p.n_slices = (int)std::max<int64_t>(1, std::min<int64_t>(ctx->n_sms / groups, (blocks + 7) / 8));
    p.dw = dw;
    CUtensorMap mg;
    if (!make_map_f32(&mg, dpre, a.M, d_out, kBlockRows, true)) return mg_fail(ctx, MG_ERR_CUDA, "cuTensorMapEncodeTiled failed for the gradient rows");
    CUtensorMap mx = mg;
    if (kept_agg && !make_map_f32(&mx, kept_agg, a.M, d_in, kBlockRows, true)) return mg_fail(ctx, MG_ERR_CUDA, "cuTensorMapEncodeTiled failed for the aggregates");
    const int stages = grad_stages(kept_agg != nullptr);
    const size_t smem = stages * (kGradStageX + (size_t)(p.n_cols / 32) * kGradBox) + 1024;
    typedef void (*Kernel)(CUtensorMap, CUtensorMap, GradWArgs);
    static const Kernel kernels[4] = {k_sage_grad_weights<true, false, false>, k_sage_grad_weights<true, true, false>, k_sage_grad_weights<false, false, false>,
                                      k_sage_grad_weights<false, false, true>};
    const int which = kept_agg ? 3 : layer > 1 ? 2 : ctx->feat_dtype == MG_DTYPE_F16 ? 1 : 0;
    MG_CUDA(ctx, mg_smem_limit(ctx, (const void*)kernels[which], (int)(stages * (kGradStageX + 8 * kGradBox) + 1024)));
    kernels[which]<<<dim3((unsigned)p.n_slices, (unsigned)groups), kGradThreads, smem, ctx->stream>>>(mg, mx, p);
    ctx->launches++;
    MG_CUDA(ctx, cudaGetLastError());
    return MG_OK;
}
