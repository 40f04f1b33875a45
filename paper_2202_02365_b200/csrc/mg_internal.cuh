// Internal declarations shared by the translation units of libmgdense.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>
#include <stdio.h>
#include <string.h>

#include <string>
#include <vector>

#include "mgdense.h"
#include "mg_device.cuh"

// ---------------------------------------------------------------------------------------
// status word written by kernels (never a trap): bit flags, read by the host after a call
// ---------------------------------------------------------------------------------------
enum : uint32_t {
    ST_RANGE = 1u,         // target id outside [0, n_nodes)
    ST_NONRESIDENT = 2u,   // target in a non-resident partition
    ST_DUPLICATE = 4u,     // same target twice in a batch
    ST_CAP_ENTRIES = 8u,   // neighbour arena too small
    ST_CAP_NODES = 16u,    // node arena too small
    ST_CAP_TABLE = 32u,    // per-batch id table full (max_nodes_per_batch too small)
    ST_INTERNAL = 64u,     // an invariant did not hold (bug guard; access skipped)
};

// what a kernel leaves in mg_ctx::d_flags besides the roles of the tensor-core kernels
constexpr uint32_t MG_ROLE_REV_SCAN = 31u;   // the scan of the backward pass's turned-round entries

// Device-side header of a sample: counters every kernel sizes itself from.
struct DenseHeader {
    uint32_t status;
    uint32_t epoch;                       // number of the sample into this handle: tags the states of k_hop's tiles
    uint64_t targets;                     // device address the targets are read from
    uint32_t ticket[MG_MAX_HOPS];         // k_hop: the next tile of the hop
    int32_t hop_base[MG_MAX_HOPS + 2];    // node arena: hop h occupies [hop_base[h], hop_base[h+1])
    int32_t ent_base[MG_MAX_HOPS + 1];    // entry arena: hop h occupies [ent_base[h], ent_base[h+1])
    int32_t rows_total[MG_MAX_HOPS + 1];  // rows of H^l summed over batches, l = 0..k
};

struct ProfPhase {
    const char* name;
    double ms;
    int64_t launches;
};

enum {
    PH_SAMPLE_INIT = 0,
    PH_SAMPLE_PICK,
    PH_SAMPLE_SORT,
    PH_SAMPLE_PLACE,
    PH_SAMPLE_RELABEL,
    PH_AGG_L1,
    PH_AGG_REST,
    PH_GEMM,
    PH_DISTMULT,
    PH_OTHER,
    PH_COUNT
};

// Reads of memory of the library's that callers have queued on streams of their own; one event stands for all of them.
struct QueuedReads {
    cudaEvent_t done = nullptr;
    bool queued = false;
};

struct mg_ctx {
    int device = 0;
    cudaStream_t stream = nullptr;
    cudaStream_t side = nullptr;  // partition swaps, asynchronous output copies
    cudaStream_t sample_stream = nullptr;  // all sampling kernels
    cudaEvent_t ev_user = nullptr;
    std::string err;
    int64_t launches = 0;
    int n_sms = 148;
    std::vector<const void*> smem_raised;   // kernels whose shared-memory limit this context has raised (mg_smem_limit)
    // word the tensor-core kernels report a barrier time-out in: mapped host memory (a copy of a device word cost a forward pass
    // 17 us behind its last kernel), read by the host once the stream has drained; d_flags is its device address
    uint32_t* h_flags = nullptr;
    uint32_t* d_flags = nullptr;

    // graph store (device)
    int64_t n_nodes = 0, n_edges = 0;
    int64_t* row_off = nullptr;  // [n_nodes + 1]
    int32_t* nbrs = nullptr;     // [n_edges]
    // in-buffer view (device); equal to the store when everything is resident
    int64_t* view_off = nullptr;
    int32_t* view_nbrs = nullptr;
    int64_t view_edges = 0;
    bool view_owned = false;
    char* view_ws = nullptr; size_t view_ws_bytes = 0;   // scratch of the view rebuild (keep bits, prefixes, tile bases)
    // second edge list (rows by source) and its in-buffer view; sample_inout = draw from both lists
    int64_t n_edges_out = 0;
    int64_t* row_off_out = nullptr;
    int32_t* nbrs_out = nullptr;
    int64_t* view_off_out = nullptr;
    int32_t* view_nbrs_out = nullptr;
    int64_t view_edges_out = 0;
    bool view_out_owned = false;
    bool sample_inout = false;

    // partitioning and buffer
    int32_t n_parts = 1;
    int64_t part_size = 0;
    int32_t capacity = 1;
    std::vector<int32_t> slot_of_part;  // committed; -1 = not resident
    std::vector<int32_t> pending_slot;  // after set_resident, before commit
    uint64_t resident_serial = 0;       // bumped whenever the committed slot map or the slots themselves change
    bool has_pending = false;
    std::vector<cudaEvent_t> pending_events;
    std::vector<char> dirty_part;       // host backing: the partition's slot was updated (mg_apply_embedding_sgd) and not written back yet
    // partition-id array (mg_set_partitioning with part_of_node): null for contiguous equal ranges
    uint8_t* d_part_of_node = nullptr;    // [n_nodes]
    int32_t* d_local_of_node = nullptr;   // [n_nodes] rank of the node inside its partition (ascending id)
    int32_t* d_nodes_by_part = nullptr;   // [n_nodes] node ids partition after partition, ascending inside a partition
    std::vector<int64_t> part_count, part_start;   // population of each partition; first row of its block in a partition-major table
    int32_t* d_slot_of_part = nullptr;   // [MG_MAX_PARTS]
    int64_t* d_res_prefix = nullptr;     // [MG_MAX_PARTS + 1] resident-node prefix counts
    int64_t* d_part_start = nullptr;     // [MG_MAX_PARTS + 1] first row of each partition's block (prefix of the populations)
    int64_t n_resident_nodes = 0;

    // features
    int feat_dtype = MG_DTYPE_F32;
    int32_t feat_dim = 0;
    int backing = MG_BACKING_HBM;
    const char* host_table = nullptr;  // MG_BACKING_HOST (may be null: then every partition needs a source of its own)
    std::vector<const char*> part_source;  // MG_BACKING_HOST: host block of a partition when it is not at its place in host_table
    char* slots = nullptr;             // device: slot s at slots + s * slot_bytes
    bool slots_owned = false;
    int32_t n_slots = 0;
    int64_t slot_bytes = 0;
    int64_t row_bytes = 0;

    // forward workspaces (grown on demand)
    float* ws_x = nullptr; size_t ws_x_bytes = 0;
    float* ws_h[2] = {nullptr, nullptr}; size_t ws_h_bytes[2] = {0, 0};
    int4* ws_meta = nullptr; size_t ws_meta_elems = 0;   // row metadata of the fused layers (mg_layer_rows) ...
    bool meta_left = false;                              // ... of the last forward pass, where that did not look it up on the way
    // what a forward pass that keeps its layers leaves to save the backward pass work: a bit per value of the outputs (above zero), then
    // aggregates of the rows.  The backward pass does without where there is no memory for it (mg_malloc).
    uint32_t* ws_saved = nullptr; size_t ws_saved_elems = 0;

    // forward schedule
    int32_t layer_window_batches = 0;  // mini-batches per window of the layer schedule; 0 = whole layers
    bool keep_layers = false;          // keep H^1..H^{k-1} for mg_layer_output (whole-layer schedule)
    bool layers_kept = false;          // what the last forward did
    int64_t agg_at[MG_MAX_HOPS + 1] = {0};        // where layer l's aggregates start in ws_saved (32-bit words); below zero: it left none
    bool agg_sum = false;                         // ... by the model's aggregator at the time
    int64_t positive_at[MG_MAX_HOPS + 1] = {0};   // where layer l's bits start in ws_saved; below zero: it left none

    // asynchronous output copy of mg_forward_host_async
    cudaEvent_t ev_fwd_done = nullptr, ev_out_done = nullptr;
    cudaEvent_t ev_backward = nullptr;   // the end of the last mg_backward_begin
    bool out_check_gemm = false;
    // H^k goes to one of two buffers in turn, so that a forward pass need not wait for the copy of the previous
    // pass's output to the host
    float* hk_buf[2] = {nullptr, nullptr};
    size_t hk_elems[2] = {0, 0};
    cudaEvent_t ev_hk_done[2] = {nullptr, nullptr};
    bool hk_pending[2] = {false, false};
    int hk_cur = 0;
    const float* last_hk = nullptr;

    QueuedReads array_reads;   // copies of mini-batches' arrays that mg_dense_arrays_copy queued on a caller's stream

    // link-prediction batches: scratch of mg_lp_prepare (grows, never shrinks)
    char* lp_ws = nullptr; size_t lp_ws_bytes = 0;
    // blocks of freed link-prediction batches, for the next ones: two, so that a batch can be prepared while the scores of the one
    // before it are still being computed; `idle` is recorded on the context's stream when the batch is freed, `reads` stands for the
    // reads that callers queued on streams of their own
    struct LpSpare { char* block = nullptr; size_t bytes = 0; cudaEvent_t idle = nullptr; QueuedReads reads; };
    LpSpare lp_spare[2];
    cudaStream_t prep_stream = nullptr;   // mg_lp_prepare's copies and kernels
    int32_t* lp_words = nullptr;       // mapped pinned host words {status, n_targets} that mg_lp_prepare's last kernel writes (behind h_flags)
    int32_t* lp_words_dev = nullptr;   // their device address
    float* gat_x = nullptr; float* gat_z = nullptr; float* gat_s = nullptr; float* gat_h[2] = {nullptr, nullptr};   // mg_gat_forward scratch
    size_t gat_x_elems = 0, gat_z_elems = 0, gat_s_elems = 0, gat_h_elems[2] = {0, 0};
    const struct mg_model* last_fwd_model = nullptr; const struct mg_dense* last_fwd_dense = nullptr;   // what mg_backward may follow
    float* bw_g = nullptr; float* bw_x = nullptr; float* bw_dx = nullptr;   // mg_backward scratch
    size_t bw_g_elems = 0, bw_x_elems = 0, bw_dx_elems = 0;
    uint32_t* bw_lists = nullptr; size_t bw_lists_elems = 0;   // mg_backward: the turned-round entries of all layers whose dX is handed down
    char* dm_images = nullptr; size_t dm_images_bytes = 0;   // TF32 operand images of the negatives (mg_distmult_score)
    // profiling
    bool prof_on = false;
    bool sample_graphs = true;   // replay the sampler's launches from a CUDA graph
    ProfPhase prof[PH_COUNT];
    std::vector<std::pair<int, std::pair<cudaEvent_t, cudaEvent_t>>> prof_pending;
};

// everything the sampler's captured device work depends on
struct SampleSignature {
    int32_t B, k, table_size, fanouts[MG_MAX_HOPS];
    int64_t T_bound, cap_batch, cap_nodes, cap_entries, n_nodes, part_size, inout;
    const void* ptrs[32];
};

struct mg_dense {
    mg_ctx* ctx = nullptr;
    int device = 0;
    int32_t k = 0, n_batches = 0;
    int32_t fanouts[MG_MAX_HOPS] = {0};
    int64_t cap_nodes = 0, cap_entries = 0;
    int32_t table_size = 0;  // slots per batch, power of two
    int64_t n_targets_total = 0;
    int64_t n_nodes = 0;     // of the graph that was sampled: ids lie below it (the context may have loaded another one since)

    // device arrays
    DenseHeader* hdr = nullptr;
    int32_t* nodes = nullptr;       // [cap_nodes] hop-major, batch-major inside a hop
    int32_t* node_batch = nullptr;  // [cap_nodes]
    int32_t* ent_off = nullptr;     // [cap_nodes + 1] start of each sampled node's entries
    uint64_t* tile_state = nullptr; // k_hop: running entry counts of the tiles, tagged with (epoch, hop)
    uint32_t epoch = 0;
    int2* pairs = nullptr;          // last hop, shared-memory deduplication: (id, entry) grouped by (batch, share, bucket)
    int32_t* share_off = nullptr;   // its group bounds
    int64_t cap_pairs = 0, cap_share = 0;
    int32_t* ent_nbrs = nullptr;    // [cap_entries] neighbour ids
    int32_t* ent_repr = nullptr;    // [cap_entries] neighbour's local row in its batch
    int32_t* node_off = nullptr;    // [(k+1) * (B+1)] arena index where batch b's hop-h nodes start
    int32_t* cum = nullptr;         // [B * (k+2)] local row of the first node of hop h; [k+1] = V
    int32_t* rowbase = nullptr;     // [(k+1) * (B+1)] first packed row of batch b in H^l
    int32_t* hkeys = nullptr;       // [B * table_size]
    int32_t* hvals = nullptr;       // [B * table_size]
    int32_t* new_ids = nullptr;     // [cap_entries] a hop's new ids by rank, a mini-batch's from the place of its first entry on
    uint64_t* newlist[2] = {nullptr, nullptr};  // [cap_nodes] keys of an export
    uint64_t* d_seeds = nullptr;    // [B]
    int32_t* scan_tmp = nullptr;    // block sums
    uint32_t* sort_hist = nullptr;  // radix histograms; bins of an export
    size_t scan_tmp_elems = 0, sort_hist_elems = 0;
    void* seg_tiles = nullptr;      // export: the (mini-batch, delta) segments and their tiles
    int64_t cap_sort_tiles = 0;     // tiles the sort scratch (histograms, block sums, segment and tile tables) is sized for
    int64_t alloc_batches = 0, alloc_table = 0;

    // export buffer for mg_dense_view
    int32_t* exp_buf = nullptr; size_t exp_elems = 0;

    // host mirror
    DenseHeader h_hdr;
    std::vector<int32_t> h_cum;      // [B * (k+2)]
    std::vector<int32_t> h_node_off; // [(k+1) * (B+1)]
    std::vector<int32_t> h_rowbase;  // [(k+1) * (B+1)]
    std::vector<int32_t> h_ent_hop;  // [k * (B+1)] arena entry index where batch b's hop-h entries start
    int32_t* d_ent_hop = nullptr;    // device copy of the same
    bool valid = false;
    // the slot map the sample was drawn under: its feature rows are addressed through it, so a later call may only
    // use the sample while every partition resident then still sits in the same slot
    uint64_t resident_serial = 0;
    std::vector<int32_t> slot_of_part_at_sample;
    // export of all mini-batches at once (mg_dense_export_many): one buffer, laid out by export_layout()
    int32_t* expm_buf = nullptr; size_t expm_elems = 0;
    cudaEvent_t ev_exported = nullptr;
    QueuedReads expm_reads;              // copies out of the export buffer that were queued on a caller's stream (mg_dense_export_copy)
    bool export_valid = false, export_pending = false;
    int32_t* perm_buf = nullptr; size_t perm_elems = 0;   // perm | inv of mini-batch perm_batch (mg_dense_batch_perm)
    int perm_batch = -1;
    uint32_t* batch_cnt = nullptr;   // [k][B] new nodes per hop and mini-batch
    // asynchronous sampling: the summary lands in pinned memory, ev_sampled marks its arrival
    // one mapped pinned block: header, offsets, seeds and a few targets of the call being queued, then the summary
    int32_t* h_stage = nullptr; size_t h_stage_ints = 0, h_summary_at = 0;
    int32_t* h_stage_dev = nullptr;                        // the same memory as the device sees it
    cudaGraphExec_t graph_exec = nullptr;                 // the sampler's device work for graph_sig
    SampleSignature graph_sig;
    int64_t graph_launches = 0;
    cudaEvent_t ev_sampled = nullptr;
    cudaEvent_t ev_read_done = nullptr;  // recorded after the last kernel that read this sample
    bool pending = false;
};

struct mg_model {
    mg_ctx* ctx = nullptr;
    int device = 0;
    int32_t k = 0;
    int32_t dims[MG_MAX_HOPS + 1] = {0};
    int precision = MG_GEMM_TF32;
    bool sum_aggr = false;   // neighbour term: sum instead of mean (Algorithm 3 as printed)
    float* w_cat[MG_MAX_HOPS] = {nullptr};  // device [2*d_in, d_out]: rows 0..d_in-1 self, then neighbour
    float* w_cat_t[MG_MAX_HOPS] = {nullptr}; // device [d_out, 2*d_in] (K-major copy for the tensor-core path)
    float* w_pad_t[MG_MAX_HOPS] = {nullptr}; // device [d_out, 2*roundup32(d_in)], zero padded, for the fused layer kernel
    // device fp16 [dims[l+1], 2*roundup64(dims[l])]: a layer's weights for fp16 operands (layer 1 over fp16 base
    // representations, later layers over fp16 intermediate outputs); null when the weights do not suit fp16
    void* w_pad_h[MG_MAX_HOPS] = {nullptr};
    bool f16_intermediates = false;   // store H^1 .. H^{k-1} as fp16 (mg_model_set_intermediates)
    float* bias[MG_MAX_HOPS] = {nullptr};
    // mg_backward: gradients of w_cat and bias (allocated by the first backward pass), a zero vector
    // (one block: layer after layer its weights' gradients, then its bias's)
    float* g_block = nullptr;
    size_t g_elems = 0;
    float* g_w_cat[MG_MAX_HOPS] = {nullptr};
    float* g_bias[MG_MAX_HOPS] = {nullptr};
    QueuedReads g_reads;                       // copies of the block that mg_backward_begin queued on a caller's stream
    float* s_block = nullptr;                  // Adagrad: accumulated squared gradients, laid out like them
    float* zeros = nullptr;
};

struct mg_lp_batch {
    mg_ctx* ctx = nullptr;
    int device = 0;
    int64_t n_edges = 0;
    int32_t n_chunks = 0, negs = 0, n_targets = 0;
    int32_t* targets = nullptr;  // device
    int32_t* src_idx = nullptr;
    int32_t* dst_idx = nullptr;
    int32_t* rel = nullptr;
    int32_t* neg_ids = nullptr;
    int32_t* neg_idx = nullptr;
    char* block = nullptr;       // the one device allocation the six arrays above live in
    size_t block_bytes = 0;
    mutable QueuedReads reads;       // of the block
};

// ---------------------------------------------------------------------------------------
// host helpers
// ---------------------------------------------------------------------------------------
int mg_fail(mg_ctx* ctx, int code, const char* fmt, ...);
// MG_OK when the partitions that were resident while `d` was sampled are still resident in the same slots (the
// sample's feature rows are then where its ids say); MG_ERR_STATE otherwise.  Host-side check, no device work.
int mg_check_sample_residency(mg_ctx* ctx, const mg_dense* d);
int mg_cuda_fail(mg_ctx* ctx, cudaError_t e, const char* what);

#define MG_CUDA(ctx, call)                                      \
    do {                                                        \
        cudaError_t e__ = (call);                               \
        if (e__ != cudaSuccess) return mg_cuda_fail(ctx, e__, #call); \
    } while (0)

// Device memory.  What the context holds only to save work is given back before an allocation fails.
static inline cudaError_t mg_malloc(mg_ctx* ctx, void** ptr, size_t bytes) {
    cudaError_t e = cudaMalloc(ptr, bytes);
    if (e != cudaErrorMemoryAllocation || !ctx->ws_saved) return e;
    cudaGetLastError();
    cudaFree(ctx->ws_saved);   // (waits for kernels that use it)
    ctx->ws_saved = nullptr; ctx->ws_saved_elems = 0;
    for (int l = 0; l <= MG_MAX_HOPS; ++l) ctx->agg_at[l] = ctx->positive_at[l] = -1;
    return cudaMalloc(ptr, bytes);
}

// grow-only device buffer
template <typename T>
static inline int mg_ensure(mg_ctx* ctx, T** ptr, size_t* have_elems, size_t need_elems) {
    if (*ptr && *have_elems >= need_elems) return MG_OK;
    if (*ptr) cudaFree(*ptr);
    *ptr = nullptr;
    *have_elems = 0;
    if (need_elems == 0) need_elems = 1;
    cudaError_t e = mg_malloc(ctx, (void**)ptr, need_elems * sizeof(T));
    if (e != cudaSuccess) {
        cudaGetLastError();
        return mg_fail(ctx, MG_ERR_OOM, "device allocation of %zu bytes failed", need_elems * sizeof(T));
    }
    *have_elems = need_elems;
    return MG_OK;
}

void mg_prof_begin(mg_ctx* ctx, int phase);
void mg_prof_end(mg_ctx* ctx, int phase, int64_t n_launches);

struct ProfScope {   // the kernels launched while it lives belong to the phase
    mg_ctx* c; int ph; int64_t before;
    ProfScope(mg_ctx* ctx, int phase) : c(ctx), ph(phase), before(ctx->launches) { mg_prof_begin(c, ph); }
    ~ProfScope() { mg_prof_end(c, ph, c->launches - before); }
};

// dynamic shared-memory limit of a kernel, raised once per context (a context has one device, and belongs to one thread)
static inline cudaError_t mg_smem_limit(mg_ctx* ctx, const void* kernel, int bytes) {
    for (const void* k : ctx->smem_raised) if (k == kernel) return cudaSuccess;
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e == cudaSuccess) ctx->smem_raised.push_back(kernel);
    return e;
}

// `stream` has just been given a read: `r` stands for it too
static inline cudaError_t mg_reads_add(QueuedReads* r, cudaStream_t stream) {
    cudaError_t e = cudaSuccess;
    if (!r->done) e = cudaEventCreateWithFlags(&r->done, cudaEventDisableTiming);
    if (e == cudaSuccess && r->queued) e = cudaStreamWaitEvent(stream, r->done);   // (from another stream)
    if (e == cudaSuccess) e = cudaEventRecord(r->done, stream);
    if (e == cudaSuccess) r->queued = true;
    return e;
}
// what `stream` is given from here on comes behind the reads
static inline cudaError_t mg_reads_wait(QueuedReads* r, cudaStream_t stream) { return r->queued ? cudaStreamWaitEvent(stream, r->done) : cudaSuccess; }
static inline void mg_reads_free(QueuedReads* r) {
    if (r->done) cudaEventDestroy(r->done);
    r->done = nullptr; r->queued = false;
}

// Host memory that a call was handed.  Pageable memory is what the host's own program order says it is, and may be read at once.
// Pinned memory may be the destination of a copy that is still queued: it is read in stream order, by a copy or, where the whole range
// is mapped, through `*mapped` by a kernel.
enum HostMemory { HOST_PAGEABLE, HOST_PINNED, HOST_MAPPED };
static inline HostMemory mg_host_memory(const void* p, size_t bytes, const void** mapped) {
    cudaPointerAttributes first, last;
    if (cudaPointerGetAttributes(&first, p) != cudaSuccess) { cudaGetLastError(); return HOST_PINNED; }
    if (first.type == cudaMemoryTypeUnregistered) return HOST_PAGEABLE;
    const char* end = static_cast<const char*>(p) + (bytes ? bytes - 1 : 0);
    if (first.type != cudaMemoryTypeHost || !first.devicePointer || cudaPointerGetAttributes(&last, end) != cudaSuccess || last.type != cudaMemoryTypeHost ||
        static_cast<const char*>(last.devicePointer) - static_cast<const char*>(first.devicePointer) != end - static_cast<const char*>(p)) {
        cudaGetLastError();
        return HOST_PINNED;
    }
    *mapped = first.devicePointer;
    return HOST_MAPPED;
}

// 32-bit words of a layer among mg_ctx::ws_saved: bit r % 32 of word (r / 32) * width + c stands for row r, column c
static inline int64_t mg_positive_words(int64_t rows, int width) { return (rows + 31) / 32 * width; }

static inline int mg_grid(const mg_ctx* ctx, int ctas_per_sm) { return ctx->n_sms * ctas_per_sm; }

// how kernels find a node's partition and its row in the feature buffer
static inline FeatGeom mg_feat_geom(const mg_ctx* ctx) {
    FeatGeom g;
    g.slot_of_part = ctx->d_slot_of_part;
    g.part_of_node = ctx->d_part_of_node;
    g.local_of_node = ctx->d_local_of_node;
    g.part_size = (uint32_t)ctx->part_size;
    g.identity = ctx->backing == MG_BACKING_HBM ? 1 : 0;   // the whole table in device memory, in node order
    return g;
}

// K order of the fused layer kernel's weights (fused_k_place): columns per block and per group, TF32 and fp16 operands
constexpr int kPackCols32 = 32, kPackGroup32 = 128, kPackCols16 = 64, kPackGroup16 = 256;

// ---- generic device-sized scan and sort (mg_sample.cu) -------------------------------------
struct SortParams {   // device-resident
    int32_t zero;
    int32_t n;        // keys
    int32_t ntiles;   // ceil(n / 4096)
    int32_t hist_len; // bins * ntiles
};
size_t mg_sort_hist_elems(int64_t max_keys);
void mg_sort_params_host(SortParams* sp, int64_t n);
// The device keeps every delta in discovery order; exports go through a permutation of the mini-batch's local rows
// (perm[c] = local row of canonical row c: deltas in the paper's order, ids ascending inside a delta, targets in the
// caller's order; inv = its inverse).  Device arrays owned by d; on ctx->stream, synchronous, off the hot path.
int mg_dense_batch_perm(mg_ctx* ctx, mg_dense* d, int b, const int32_t** perm, const int32_t** inv);
void mg_sort_u64(mg_ctx* ctx, uint64_t* const buf[2], const SortParams* sp, int lo_bit, int bits, uint32_t* hist,
                 uint32_t* scan_tmp, int* res_buf);

