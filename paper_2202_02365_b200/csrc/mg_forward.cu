// GraphSage forward over DENSE (Section 4.2): per layer a segment-mean over the sampled
// neighbours (Algorithm 3 with mean instead of sum) and the self / neighbour linear maps.
//
// Rows are kept in sampling order (targets first), so layer l's output rows of a batch are the
// prefix [0, N_l) of its local rows and the "update" of Algorithm 2 is only a smaller row count.
// All batches are packed: H^l holds rowbase[l][b] .. rowbase[l][b+1] for batch b.
// Layer 1 reads base representations straight from the partition buffer (H^0 is never stored).

#include <cuda_fp16.h>

#include <algorithm>
#include <cmath>
#include <cstdlib>

#include "mg_device.cuh"

#include "mg_internal.cuh"

int mg_gemm_tf32(mg_ctx* ctx, const float* x, const float* w_t, const float* bias, float* out, int64_t M, int N, int K,
                 bool relu);  // mg_gemm_tcgen05.cu
int mg_gemm_tf32_status(mg_ctx* ctx);
// mg_layer_fused.cu
bool mg_layer_fused_supported(int d_in, int d_out);
int mg_layer_rows(mg_ctx* ctx, const mg_dense* d, int4* meta, const int64_t* start /* [k + 2], layer l at start[l] */);
bool mg_layer_rows_inline(const mg_ctx* ctx, const mg_dense* d);   // the layers' kernels do without it
int mg_layer_fused(mg_ctx* ctx, const mg_dense* d, int layer, int d_in, int d_out, const float* w_pad_t, const float* bias,
                   const float* h_prev, float* h_out, float* h_out2 /* nullable: the rows once more */, int flags /* 1 = ReLU, 2 = sum instead of mean */, const int4* row_meta,
                   int64_t row_lo, int64_t row_hi, int64_t safe_src_row, const void* w_pad_h /* the layer's fp16 weights, nullable */,
                   int in_f16 /* layers >= 2: h_prev holds fp16 rows */, int out_f16 /* h_out receives fp16 rows */,
                   uint32_t* positive /* nullable: a bit per value of h_out, above zero */, float* kept_agg /* nullable: the rows' aggregates */);

int mg_layer_grad_weights(mg_ctx* ctx, const mg_dense* d, int layer, int d_in, int d_out, const float* h_prev, const float* dpre, const int4* row_meta,
                          int sum_aggr, const float* kept_agg /* nullable: what mg_layer_fused left */, float* dw);

namespace {

constexpr int kThreads = 256;

struct AggArgs {
    int32_t B, k, layer;     // layer l = 1..k
    int32_t d_in;
    int32_t row_lo, row_hi;  // packed output rows handled by this launch
    const int32_t* rowbase_out;  // [B+1] of layer l
    const int32_t* rowbase_in;   // [B+1] of layer l-1
    const int32_t* cum;          // [B][k+2]
    const int32_t* node_off;     // [k+1][B+1]
    const int32_t* nodes;
    const int32_t* ent_off;
    const int32_t* ent_nbrs;
    const int32_t* ent_repr;
    const float* h_prev;         // layers >= 2
    // layer 1: the partition buffer
    const char* slots;
    FeatGeom feat;
    int64_t row_bytes;
    float* x;                    // [rows, 2 * d_in], row r of this launch at x + (r - row_lo) * 2 * d_in
    int round_tf32;
    int sum_aggr;                // neighbour term = sum of the sampled neighbours instead of their mean
};

__device__ __forceinline__ float to_tf32(float v) {
    uint32_t u;
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(u) : "f"(v));
    return __uint_as_float(u);
}

__device__ __forceinline__ const char* feature_row(const AggArgs& a, int32_t node) {
    return a.slots + feat_row(a.feat, node) * a.row_bytes;
}

// one 16-byte chunk -> 4 (fp32) or 8 (fp16) floats
template <bool HALF>
struct Chunk {
    static constexpr int kVals = HALF ? 8 : 4;
    float v[kVals];
    __device__ __forceinline__ void zero() {
#pragma unroll
        for (int i = 0; i < kVals; ++i) v[i] = 0.f;
    }
    __device__ __forceinline__ void load(const char* row, int chunk) {
        const uint4 raw = __ldg(reinterpret_cast<const uint4*>(row) + chunk);
        if (HALF) {
            const __half2* h = reinterpret_cast<const __half2*>(&raw);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float2 f = __half22float2(h[i]);
                v[2 * i] = f.x;
                v[2 * i + 1] = f.y;
            }
        } else {
            v[0] = __uint_as_float(raw.x); v[1] = __uint_as_float(raw.y);
            v[2] = __uint_as_float(raw.z); v[3] = __uint_as_float(raw.w);
        }
    }
    __device__ __forceinline__ void add(const Chunk& o) {
#pragma unroll
        for (int i = 0; i < kVals; ++i) v[i] += o.v[i];
    }
    __device__ __forceinline__ void store(float* dst, float scale, bool round) const {
#pragma unroll
        for (int i = 0; i < kVals; i += 4) {
            float4 o = make_float4(v[i] * scale, v[i + 1] * scale, v[i + 2] * scale, v[i + 3] * scale);
            if (round) { o.x = to_tf32(o.x); o.y = to_tf32(o.y); o.z = to_tf32(o.z); o.w = to_tf32(o.w); }
            *reinterpret_cast<float4*>(dst + i) = o;
        }
    }
};

// G lanes per output row; each lane owns NCH 16-byte chunks of the row (chunk = gl + j * G).
template <int G, int NCH, bool FIRST, bool HALF>
__global__ void __launch_bounds__(kThreads) k_aggregate(AggArgs a) {
    using C = Chunk<HALF>;
    constexpr int kRowsPerBlock = kThreads / G;
    const int gl = threadIdx.x % G;
    const int n_chunks = a.d_in / C::kVals;
    const int kk = a.k;
    for (int32_t r = a.row_lo + blockIdx.x * kRowsPerBlock + threadIdx.x / G; r < a.row_hi; r += gridDim.x * kRowsPerBlock) {
        const int b = upper_segment(a.rowbase_out, a.B + 1, r);
        const int32_t l = r - a.rowbase_out[b];
        const int32_t* cum = a.cum + b * (kk + 2);
        int h = 0;
        while (h < kk - a.layer && l >= cum[h + 1]) ++h;
        const int32_t idx = a.node_off[h * (a.B + 1) + b] + (l - cum[h]);
        const int32_t e0 = a.ent_off[idx], e1 = a.ent_off[idx + 1];
        const int64_t in_base = FIRST ? 0 : (int64_t)a.rowbase_in[b];
        float* xrow = a.x + (int64_t)(r - a.row_lo) * 2 * a.d_in;

        // self row
        const char* self_row = FIRST ? feature_row(a, a.nodes[idx])
                                     : reinterpret_cast<const char*>(a.h_prev + (in_base + l) * a.d_in);
        C acc[NCH];
#pragma unroll
        for (int j = 0; j < NCH; ++j) {
            const int c = gl + j * G;
            if (c < n_chunks) {
                C s;
                s.load(self_row, c);
                s.store(xrow + c * C::kVals, 1.f, a.round_tf32);
            }
            acc[j].zero();
        }
        // neighbours, in entry order, two rows in flight
        int32_t e = e0;
        for (; e + 1 < e1; e += 2) {
            const char* r0 = FIRST ? feature_row(a, a.ent_nbrs[e])
                                   : reinterpret_cast<const char*>(a.h_prev + (in_base + a.ent_repr[e]) * a.d_in);
            const char* r1 = FIRST ? feature_row(a, a.ent_nbrs[e + 1])
                                   : reinterpret_cast<const char*>(a.h_prev + (in_base + a.ent_repr[e + 1]) * a.d_in);
            C t0[NCH], t1[NCH];
#pragma unroll
            for (int j = 0; j < NCH; ++j) {
                const int c = gl + j * G;
                if (c < n_chunks) { t0[j].load(r0, c); t1[j].load(r1, c); }
            }
#pragma unroll
            for (int j = 0; j < NCH; ++j) {
                const int c = gl + j * G;
                if (c < n_chunks) { acc[j].add(t0[j]); acc[j].add(t1[j]); }
            }
        }
        if (e < e1) {
            const char* r0 = FIRST ? feature_row(a, a.ent_nbrs[e])
                                   : reinterpret_cast<const char*>(a.h_prev + (in_base + a.ent_repr[e]) * a.d_in);
#pragma unroll
            for (int j = 0; j < NCH; ++j) {
                const int c = gl + j * G;
                if (c < n_chunks) { C t; t.load(r0, c); acc[j].add(t); }
            }
        }
        const float inv = e1 > e0 ? (a.sum_aggr ? 1.f : 1.f / (float)(e1 - e0)) : 0.f;
#pragma unroll
        for (int j = 0; j < NCH; ++j) {
            const int c = gl + j * G;
            if (c < n_chunks) acc[j].store(xrow + a.d_in + c * C::kVals, inv, a.round_tf32);
        }
    }
}

// ---- CUDA-core fp32 GEMM with bias / ReLU epilogue (MG_GEMM_FP32) ---------------------------
// out[M, N] = act(x[M, K] . w[K, N] + bias)
template <bool RELU>
__global__ void __launch_bounds__(256) k_gemm_fp32(const float* __restrict__ x, const float* __restrict__ w,
                                                   const float* __restrict__ bias, float* __restrict__ out, int64_t M,
                                                   int N, int K) {
    constexpr int BM = 64, BN = 64, BK = 16;
    __shared__ float As[BK][BM + 4];
    __shared__ float Bs[BK][BN + 4];
    const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
    const int64_t m0 = (int64_t)blockIdx.x * BM;
    const int n0 = blockIdx.y * BN;
    float acc[4][4] = {};
    for (int k0 = 0; k0 < K; k0 += BK) {
        for (int i = threadIdx.x; i < BM * BK; i += 256) {
            const int mm = i / BK, kk = i % BK;
            As[kk][mm] = (m0 + mm < M && k0 + kk < K) ? x[(m0 + mm) * K + k0 + kk] : 0.f;
        }
        for (int i = threadIdx.x; i < BK * BN; i += 256) {
            const int kk = i / BN, nn = i % BN;
            Bs[kk][nn] = (k0 + kk < K && n0 + nn < N) ? w[(int64_t)(k0 + kk) * N + n0 + nn] : 0.f;
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < BK; ++kk) {
            float av[4], bv[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) { av[i] = As[kk][ty * 4 + i]; bv[i] = Bs[kk][tx * 4 + i]; }
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(av[i], bv[j], acc[i][j]);
        }
        __syncthreads();
    }
    for (int i = 0; i < 4; ++i) {
        const int64_t m = m0 + ty * 4 + i;
        if (m >= M) continue;
        for (int j = 0; j < 4; ++j) {
            const int n = n0 + tx * 4 + j;
            if (n >= N) continue;
            float v = acc[i][j] + bias[n];
            if (RELU) v = fmaxf(v, 0.f);
            out[m * N + n] = v;
        }
    }
}

// ---- canonical-order exports ---------------------------------------------------------------
struct RowExportArgs {
    int32_t k, n_rows, first_delta;  // rows of Delta_{first_delta} .. Delta_k in the paper's order
    int32_t nio[MG_MAX_HOPS + 2];    // canonical offsets of the deltas of this batch
    int32_t cum[MG_MAX_HOPS + 2];
    int32_t dim;
    const int32_t* perm;             // local row of every canonical row of the mini-batch (mg_dense_batch_perm)
};

// out[c, :] = src[local(c), :] where c runs over the paper's row order
__global__ void __launch_bounds__(kThreads) k_export_rows(RowExportArgs a, const float* __restrict__ src, float* __restrict__ out) {
    const int vec = a.dim / 4;
    const int64_t total = (int64_t)a.n_rows * vec;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
        const int32_t c = (int32_t)(i / vec) + a.nio[a.first_delta];
        const int q = (int)(i % vec);
        const int32_t l = a.perm[c];
        reinterpret_cast<float4*>(out)[i] = reinterpret_cast<const float4*>(src + (int64_t)l * a.dim)[q];
    }
}

struct H0Args {
    RowExportArgs r;
    int32_t node_off[MG_MAX_HOPS + 1];
    const int32_t* nodes;
    const char* slots;
    FeatGeom feat;
    int64_t row_bytes;
};

template <bool HALF>
__global__ void __launch_bounds__(kThreads) k_gather_h0(H0Args a, float* __restrict__ out) {
    using C = Chunk<HALF>;
    const int n_chunks = a.r.dim / C::kVals;
    const int64_t total = (int64_t)a.r.n_rows * n_chunks;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
        const int32_t c = (int32_t)(i / n_chunks);
        const int q = (int)(i % n_chunks);
        const int32_t l = a.r.perm[c];
        int h = 0;
        while (h < a.r.k && l >= a.r.cum[h + 1]) ++h;
        const int32_t node = a.nodes[a.node_off[h] + (l - a.r.cum[h])];
        const char* row = a.slots + feat_row(a.feat, node) * a.row_bytes;
        C v;
        v.load(row, q);
        v.store(out + (int64_t)c * a.r.dim + q * C::kVals, 1.f, false);
    }
}

// ---- weights: the optimisers' steps and the copies that the kernels read ------------------------------------------------
// One launch for all layers: a block takes 32 rows x 32 columns of a layer's [W_self; W_nbr], applies the step, and writes the
// tile into every copy -- the plain transpose, and the padded K orders of the fused layer kernel -- along the copies' rows.
// (Five launches per layer before: 15 of 2 to 4 us and the gaps between them for three layers.)
enum { W_COPY = 0, W_SGD = 1, W_ADAGRAD = 2 };
struct WeightArgs {
    int32_t k;
    int32_t tile_at[MG_MAX_HOPS + 1];   // first tile of the layer; a block per layer for the biases behind the tiles
    int32_t d_in[MG_MAX_HOPS], d_out[MG_MAX_HOPS];
    float* w[MG_MAX_HOPS];
    float* w_t[MG_MAX_HOPS];
    float* w_pad[MG_MAX_HOPS];
    __half* w_pad_h[MG_MAX_HOPS];       // null: none
    float* bias[MG_MAX_HOPS];
    int64_t g_at[MG_MAX_HOPS];          // the layer's place in the gradient block and the optimiser's state
    const float* g;
    float* state;
    float lr, eps;
    int32_t round_tf32;                 // w_t holds TF32 values
};

// SGD: w -= lr * g; Adagrad: state += g^2, w -= lr * g / (sqrt(state) + eps)
template <int MODE>
__device__ __forceinline__ float weight_step(const WeightArgs& a, float w, int64_t at) {
    if (MODE == W_COPY) return w;
    const float g = a.g[at];
    if (MODE == W_SGD) return w - a.lr * g;
    const float s = a.state[at] + g * g;
    a.state[at] = s;
    return w - a.lr * g / (sqrtf(s) + a.eps);
}

template <int MODE>
__global__ void __launch_bounds__(kThreads) k_weights(WeightArgs a) {
    __shared__ float tile[32][33];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int t = (int)blockIdx.x;
    if (t >= a.tile_at[a.k]) {
        const int l = t - a.tile_at[a.k];
        const int64_t g0 = a.g_at[l] + 2 * (int64_t)a.d_in[l] * a.d_out[l];
        for (int n = threadIdx.x; n < a.d_out[l]; n += kThreads) a.bias[l][n] = weight_step<MODE>(a, a.bias[l][n], g0 + n);
        return;
    }
    int l = 0;
    while (t >= a.tile_at[l + 1]) ++l;
    const int di = a.d_in[l], dn = a.d_out[l];
    const int col_blocks = (di + 31) / 32, n_blocks = (dn + 31) / 32;
    int q = t - a.tile_at[l];
    const int n0 = q % n_blocks * 32;
    q /= n_blocks;
    const int c0 = q % col_blocks * 32, part = q / col_blocks;   // 32 input columns of the self (0) or the neighbour (1) weights
    for (int r = warp; r < 32; r += kThreads / 32) {
        const int c = c0 + r, n = n0 + lane;
        float w = 0.f;
        if (c < di && n < dn) {
            const int64_t i = (int64_t)(part * di + c) * dn + n;
            w = weight_step<MODE>(a, a.w[l][i], a.g_at[l] + i);
            if (MODE != W_COPY) a.w[l][i] = w;
        }
        tile[r][lane] = w;
    }
    __syncthreads();
    const int pad32 = (di + kPackCols32 - 1) / kPackCols32 * kPackCols32, pad16 = (di + kPackCols16 - 1) / kPackCols16 * kPackCols16;
    for (int r = warp; r < 32; r += kThreads / 32) {
        const int c = c0 + lane, n = n0 + r;
        if (c >= di || n >= dn) continue;
        const float w = tile[lane][r], w32 = to_tf32(w);
        a.w_t[l][(int64_t)n * 2 * di + part * di + c] = a.round_tf32 ? w32 : w;
        a.w_pad[l][(int64_t)n * 2 * pad32 + fused_k_place(part, c, kPackCols32, kPackGroup32)] = w32;
        if (a.w_pad_h[l]) a.w_pad_h[l][(int64_t)n * 2 * pad16 + fused_k_place(part, c, kPackCols16, kPackGroup16)] = __float2half_rn(w);
    }
}

template <bool FIRST, bool HALF>
void launch_aggregate(const AggArgs& a, int grid, cudaStream_t st) {
    const int vals = HALF ? 8 : 4;
    const int n_chunks = a.d_in / vals;
    int G = 4;
    while (G < 32 && G < n_chunks) G <<= 1;
    const int nch = (n_chunks + G - 1) / G;
#define MG_AGG(GG, NN) k_aggregate<GG, NN, FIRST, HALF><<<grid, kThreads, 0, st>>>(a)
    if (G == 4) MG_AGG(4, 1);
    else if (G == 8) MG_AGG(8, 1);
    else if (G == 16) MG_AGG(16, 1);
    else if (nch == 1) MG_AGG(32, 1);
    else if (nch == 2) MG_AGG(32, 2);
    else if (nch == 3) MG_AGG(32, 3);
    else if (nch == 4) MG_AGG(32, 4);
    else if (nch <= 6) MG_AGG(32, 6);
    else MG_AGG(32, 8);
#undef MG_AGG
}

void fill_row_export(const mg_dense* d, int batch, int first_delta, int dim, RowExportArgs* r) {
    const int k = d->k;
    memset(r, 0, sizeof(*r));
    r->k = k;
    r->dim = dim;
    r->first_delta = first_delta;
    for (int h = 0; h <= k + 1; ++h) r->cum[h] = d->h_cum[(size_t)batch * (k + 2) + h];
    r->nio[0] = 0;
    for (int j = 0; j <= k; ++j) r->nio[j + 1] = r->nio[j] + (r->cum[k - j + 1] - r->cum[k - j]);
    r->n_rows = r->nio[k + 1] - r->nio[first_delta];
}

}  // namespace

// A model's weights: MODE's step, then every copy, on ctx's stream
template <int MODE>
static void launch_weights(mg_ctx* ctx, mg_model* m, float lr, float eps) {
    WeightArgs a;
    memset(&a, 0, sizeof(a));
    a.k = m->k;
    int64_t at = 0;
    for (int l = 0; l < m->k; ++l) {
        const int di = m->dims[l], dn = m->dims[l + 1];
        a.tile_at[l + 1] = a.tile_at[l] + 2 * ((di + 31) / 32) * ((dn + 31) / 32);
        a.d_in[l] = di; a.d_out[l] = dn;
        a.w[l] = m->w_cat[l]; a.w_t[l] = m->w_cat_t[l]; a.w_pad[l] = m->w_pad_t[l]; a.w_pad_h[l] = static_cast<__half*>(m->w_pad_h[l]); a.bias[l] = m->bias[l];
        a.g_at[l] = at;
        at += 2 * (int64_t)di * dn + dn;
    }
    a.g = m->g_block; a.state = m->s_block; a.lr = lr; a.eps = eps; a.round_tf32 = m->precision == MG_GEMM_TF32;
    k_weights<MODE><<<a.tile_at[m->k] + m->k, kThreads, 0, ctx->stream>>>(a);
    ctx->launches++;
}

// ---------------------------------------------------------------------------------------
extern "C" int mg_model_create(mg_ctx* ctx, int32_t k, const int32_t* dims, const float* const* w_self,
                               const float* const* w_nbr, const float* const* bias, int gemm_precision, mg_model** out) {
    if (!ctx) return MG_ERR_ARG;
    if (!out || !dims || !w_self || !w_nbr || !bias) return mg_fail(ctx, MG_ERR_ARG, "null argument");
    if (k <= 0 || k > MG_MAX_HOPS) return mg_fail(ctx, MG_ERR_ARG, "k must be in [1, %d]", MG_MAX_HOPS);
    if (gemm_precision != MG_GEMM_TF32 && gemm_precision != MG_GEMM_FP32) return mg_fail(ctx, MG_ERR_ARG, "unknown gemm precision");
    for (int l = 0; l <= k; ++l)
        if (dims[l] <= 0 || dims[l] % 4 != 0 || dims[l] > 1024) return mg_fail(ctx, MG_ERR_ARG, "layer widths must be multiples of 4 in [4, 1024]");
    for (int l = 0; l < k; ++l)
        if (!w_self[l] || !w_nbr[l] || !bias[l]) return mg_fail(ctx, MG_ERR_ARG, "null weight pointer");
    MG_CUDA(ctx, cudaSetDevice(ctx->device));
    mg_model* m = new mg_model();
    m->ctx = ctx;
    m->device = ctx->device;
    m->k = k;
    m->precision = gemm_precision;
    for (int l = 0; l <= k; ++l) m->dims[l] = dims[l];
    for (int l = 0; l < k; ++l) {
        const size_t di = dims[l], dn = dims[l + 1];
        if (mg_malloc(ctx, (void**)&m->w_cat[l], sizeof(float) * 2 * di * dn) != cudaSuccess ||
            mg_malloc(ctx, (void**)&m->w_cat_t[l], sizeof(float) * 2 * di * dn) != cudaSuccess ||
            mg_malloc(ctx, (void**)&m->w_pad_t[l], sizeof(float) * 2 * ((di + 31) / 32 * 32) * dn) != cudaSuccess ||
            mg_malloc(ctx, (void**)&m->bias[l], sizeof(float) * dn) != cudaSuccess) {
            cudaGetLastError();
            mg_model_free(m);
            return mg_fail(ctx, MG_ERR_OOM, "weight allocation failed");
        }
        cudaMemcpyAsync(m->w_cat[l], w_self[l], sizeof(float) * di * dn, cudaMemcpyHostToDevice, ctx->stream);
        cudaMemcpyAsync(m->w_cat[l] + di * dn, w_nbr[l], sizeof(float) * di * dn, cudaMemcpyHostToDevice, ctx->stream);
        cudaMemcpyAsync(m->bias[l], bias[l], sizeof(float) * dn, cudaMemcpyHostToDevice, ctx->stream);
        cudaMemsetAsync(m->w_pad_t[l], 0, sizeof(float) * 2 * ((di + 31) / 32 * 32) * dn, ctx->stream);   // (the padding stays zero)
    }
    // Every layer's weights in fp16 form too, for layers whose input rows are fp16 (layer 1 over fp16 base
    // representations; later layers when the model stores its intermediate outputs as fp16).  fp16 keeps the 10-bit
    // mantissa TF32 keeps but has a 5-bit exponent: the copy is made only when the weights sit well inside its range
    // (largest magnitude below 2^15, root mean square above 2^-10); otherwise that layer stays on TF32 operands.
    for (int l = 0; l < k && gemm_precision == MG_GEMM_TF32; ++l) {
        const size_t di = dims[l], dn = dims[l + 1];
        if (di % 8 != 0) continue;
        double sq = 0.0, mx = 0.0;
        for (size_t i = 0; i < di * dn; ++i) {
            const double a = std::fabs((double)w_self[l][i]), b = std::fabs((double)w_nbr[l][i]);
            sq += a * a + b * b;
            mx = std::max(mx, std::max(a, b));
        }
        const double rms = std::sqrt(sq / (double)(2 * di * dn));
        if (!(mx < 32768.0 && rms > 1.0 / 1024.0)) continue;
        if (mg_malloc(ctx, (void**)&m->w_pad_h[l], sizeof(uint16_t) * 2 * ((di + 63) / 64 * 64) * dn) != cudaSuccess) {
            cudaGetLastError();
            mg_model_free(m);
            return mg_fail(ctx, MG_ERR_OOM, "weight allocation failed");
        }
        cudaMemsetAsync(m->w_pad_h[l], 0, sizeof(uint16_t) * 2 * ((di + 63) / 64 * 64) * dn, ctx->stream);
    }
    // K-major copies [d_out, 2 d_in], rounded to nearest TF32 once, for the tensor-core path
    launch_weights<W_COPY>(ctx, m, 0.f, 0.f);
    cudaError_t e = cudaStreamSynchronize(ctx->stream);
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e != cudaSuccess) { mg_model_free(m); return mg_cuda_fail(ctx, e, "weight upload"); }
    *out = m;
    return MG_OK;
}

extern "C" int mg_model_set_aggregator(mg_model* m, int aggregator) {
    if (!m) return MG_ERR_ARG;
    if (aggregator != MG_AGGR_MEAN && aggregator != MG_AGGR_SUM) return mg_fail(m->ctx, MG_ERR_ARG, "unknown aggregator");
    m->sum_aggr = aggregator == MG_AGGR_SUM;
    return MG_OK;
}

extern "C" int mg_model_set_intermediates(mg_model* m, int dtype) {
    if (!m) return MG_ERR_ARG;
    if (dtype != MG_DTYPE_F32 && dtype != MG_DTYPE_F16) return mg_fail(m->ctx, MG_ERR_ARG, "unknown dtype");
    m->f16_intermediates = dtype == MG_DTYPE_F16;
    return MG_OK;
}

extern "C" int mg_model_free(mg_model* m) {
    if (!m) return MG_OK;
    cudaSetDevice(m->device);
    for (int l = 0; l < MG_MAX_HOPS; ++l) {
        cudaFree(m->w_cat[l]); cudaFree(m->w_cat_t[l]); cudaFree(m->w_pad_t[l]); cudaFree(m->bias[l]);
    }
    cudaFree(m->zeros); cudaFree(m->g_block); cudaFree(m->s_block);
    mg_reads_free(&m->g_reads);
    for (int l = 0; l < MG_MAX_HOPS; ++l) cudaFree(m->w_pad_h[l]);
    if (m->ctx && m->ctx->last_fwd_model == m) m->ctx->last_fwd_model = nullptr;
    delete m;
    return MG_OK;
}

static int forward_checks(mg_ctx* ctx, const mg_model* m, const mg_dense* d) {
    if (!m || !d) return mg_fail(ctx, MG_ERR_ARG, "null argument");
    if (d->pending) return mg_fail(ctx, MG_ERR_STATE, "a sample is in flight on this mg_dense: call mg_sample_many_end first");
    if (!d->valid) return mg_fail(ctx, MG_ERR_STATE, "mg_dense holds no completed sample");
    if (d->ctx != ctx || m->ctx != ctx) return mg_fail(ctx, MG_ERR_ARG, "handle belongs to another context");
    if (!ctx->slots || ctx->feat_dim <= 0) return mg_fail(ctx, MG_ERR_STATE, "no feature table loaded");
    if (m->k != d->k) return mg_fail(ctx, MG_ERR_STATE, "model has %d layers, sample has %d hops", m->k, d->k);
    if (m->dims[0] != ctx->feat_dim) return mg_fail(ctx, MG_ERR_STATE, "model input width %d != feature dim %d", m->dims[0], ctx->feat_dim);
    return mg_check_sample_residency(ctx, d);
}

// rows of a layer are processed in chunks small enough for the [self | mean] staging matrix to
// stay in L2 between the aggregation kernel that writes it and the GEMM that reads it
static int64_t chunk_rows_for(int d_in) {
    const int64_t bytes_per_row = (int64_t)2 * d_in * 4;
    int64_t rows = (48ll << 20) / bytes_per_row;
    rows = std::max<int64_t>(rows / 128 * 128, 128);
    return rows;
}

constexpr int64_t kKeepEntriesPerRow = 3;   // layers with more entries per row leave their aggregates for the backward pass

enum { OUT_DEVICE = 0, OUT_HOST = 1, OUT_HOST_ASYNC = 2 };

// hands H^k (device, packed) to the caller: device or host copy, blocking or on the side stream
// (out_written: the last layer's kernel has stored the rows there itself)
static int finish_forward(mg_ctx* ctx, const mg_model* m, mg_dense* d, float* out, int out_mode, const float* hk, bool out_written) {
    cudaStream_t st = ctx->stream;
    if (!d->ev_read_done) MG_CUDA(ctx, cudaEventCreateWithFlags(&d->ev_read_done, cudaEventDisableTiming));
    MG_CUDA(ctx, cudaEventRecord(d->ev_read_done, st));   // the next sample into d waits for this
    const int k = d->k;
    const size_t out_bytes = (size_t)d->h_hdr.rows_total[k] * m->dims[k] * sizeof(float);
    if (out_mode == OUT_HOST_ASYNC) {
        // the copy to the host runs on the side stream behind the last layer kernel; the caller's next
        // calls (sampling the next group) overlap it
        MG_CUDA(ctx, cudaEventRecord(ctx->ev_fwd_done, st));
        MG_CUDA(ctx, cudaStreamWaitEvent(ctx->side, ctx->ev_fwd_done, 0));
        MG_CUDA(ctx, cudaMemcpyAsync(out, hk, out_bytes, cudaMemcpyDeviceToHost, ctx->side));
        MG_CUDA(ctx, cudaEventRecord(ctx->ev_out_done, ctx->side));
        MG_CUDA(ctx, cudaEventRecord(ctx->ev_hk_done[ctx->hk_cur], ctx->side));   // this H^k buffer is free again after the copy
        ctx->hk_pending[ctx->hk_cur] = true;
        ctx->out_check_gemm = m->precision == MG_GEMM_TF32;
        return MG_OK;
    }
    if (!out_written) MG_CUDA(ctx, cudaMemcpyAsync(out, hk, out_bytes, out_mode == OUT_DEVICE ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost, st));
    MG_CUDA(ctx, cudaStreamSynchronize(st));
    if (m->precision == MG_GEMM_TF32) return mg_gemm_tf32_status(ctx);
    return MG_OK;
}

// mg_layer_rows of all layers into ws_meta, layer l's at meta_at[l]
static int row_metadata(mg_ctx* ctx, const mg_dense* d, int64_t* meta_at) {
    for (int l = 1; l <= d->k; ++l) meta_at[l + 1] = meta_at[l] + (int64_t)d->h_hdr.rows_total[l];
    const size_t need = (size_t)meta_at[d->k + 1];
    if (ctx->ws_meta_elems < need)
        if (int rc = mg_ensure(ctx, &ctx->ws_meta, &ctx->ws_meta_elems, need + need / 4 + 4)) return rc;
    ProfScope ps(ctx, PH_OTHER);
    return mg_layer_rows(ctx, d, ctx->ws_meta, meta_at);
}

static int forward_pass(mg_ctx* ctx, const mg_model* m, mg_dense* d, float* out, int out_mode) {
    int rc;
    const int k = d->k, B = d->n_batches;
    cudaStream_t st = ctx->stream;
    // H^k of this pass goes to the buffer the pass before last used; an output copy of that pass to the host (side
    // stream) may still read it.  The copy of the previous pass reads the other buffer and is not waited for.
    float* hk = nullptr;
    {
        const int hi = ctx->hk_cur ^= 1;
        if (!ctx->ev_hk_done[hi]) MG_CUDA(ctx, cudaEventCreateWithFlags(&ctx->ev_hk_done[hi], cudaEventDisableTiming));
        if (ctx->hk_pending[hi]) {
            MG_CUDA(ctx, cudaStreamWaitEvent(st, ctx->ev_hk_done[hi], 0));
            ctx->hk_pending[hi] = false;
        }
        const size_t need = (size_t)d->h_hdr.rows_total[k] * m->dims[k];
        if (ctx->hk_elems[hi] < need && (rc = mg_ensure(ctx, &ctx->hk_buf[hi], &ctx->hk_elems[hi], need + need / 4 + 4))) return rc;
        hk = ctx->hk_buf[hi];
        ctx->last_hk = hk;
    }

    // Windowed schedule: when every layer runs in the fused kernel and the intermediate layer outputs need not
    // be kept, the layers are run over sub-groups of a few mini-batches at a time through small reused
    // buffers.  H^l of a sub-group is then still in L2 when layer l+1 reads it, and is overwritten in L2 by the
    // next sub-group before most of it is written back to DRAM.
    bool all_fused = m->precision == MG_GEMM_TF32;
    for (int l = 1; l <= k; ++l) all_fused = all_fused && mg_layer_fused_supported(m->dims[l - 1], m->dims[l]);
    // row metadata of the layers the fused kernel runs, all in one launch
    const bool any_fused = m->precision == MG_GEMM_TF32;
    // (few rows of one mini-batch: the layers' kernels look it up themselves, unless the profile is to have its phase)
    int64_t meta_at[MG_MAX_HOPS + 2] = {0};
    const bool rows_inline = all_fused && !ctx->keep_layers && !ctx->prof_on && ctx->layer_window_batches == 0 && mg_layer_rows_inline(ctx, d);
    ctx->meta_left = any_fused && !rows_inline;
    if (ctx->meta_left && (rc = row_metadata(ctx, d, meta_at))) return rc;
    // H^k stays in the library's buffer (mg_layer_output, mg_backward) and goes to the caller's: the last layer's kernel
    // stores its tiles to both when it can (the copy behind it read and wrote the rows once more: 41 us for 128,000 rows of
    // 1 KB, and a launch).  Not into the feature table, which other tiles still read.
    const uintptr_t out_at = reinterpret_cast<uintptr_t>(out), table_at = reinterpret_cast<uintptr_t>(ctx->slots);
    const size_t out_bytes = (size_t)d->h_hdr.rows_total[k] * m->dims[k] * sizeof(float);
    const size_t table_bytes = ctx->backing == MG_BACKING_HBM ? (size_t)ctx->n_nodes * ctx->row_bytes : (size_t)ctx->n_slots * ctx->slot_bytes;
    const bool in_table = out_at < table_at + table_bytes && table_at < out_at + out_bytes;
    float* out2 = out_mode == OUT_DEVICE && any_fused && mg_layer_fused_supported(m->dims[k - 1], m->dims[k]) && out_at % 16 == 0 && !in_table ? out : nullptr;
    const int sub = ctx->layer_window_batches;
    ctx->layers_kept = !(all_fused && sub > 0 && !ctx->keep_layers && k > 1);
    if (!ctx->layers_kept) {
        const int32_t* rb = d->h_rowbase.data();      // [(k+1)][B+1]
        size_t ring_off[MG_MAX_HOPS + 1] = {0}, ring_total = 0;
        for (int l = 1; l <= k; ++l) {
            ring_off[l] = ring_total;
            if (l == k) break;
            int64_t widest = 0;
            for (int b0 = 0; b0 < B; b0 += sub) {
                const int b1 = std::min(B, b0 + sub);
                widest = std::max<int64_t>(widest, rb[(size_t)l * (B + 1) + b1] - rb[(size_t)l * (B + 1) + b0]);
            }
            ring_total += (size_t)widest * m->dims[l];
        }
        {
            size_t have = ctx->ws_h_bytes[0] / sizeof(float);
            if (have < ring_total && (rc = mg_ensure(ctx, &ctx->ws_h[0], &have, ring_total + ring_total / 4))) return rc;
            ctx->ws_h_bytes[0] = have * sizeof(float);
        }
        float* base = ctx->ws_h[0];
        for (int b0 = 0; b0 < B; b0 += sub) {
            const int b1 = std::min(B, b0 + sub);
            for (int l = 1; l <= k; ++l) {
                const int64_t lo = rb[(size_t)l * (B + 1) + b0], hi = rb[(size_t)l * (B + 1) + b1];
                const int64_t lo_in = rb[(size_t)(l - 1) * (B + 1) + b0];
                // pointers shifted so that the kernel's global packed row indices land inside the windows
                const float* h_prev = l > 1 ? base + ring_off[l - 1] - lo_in * m->dims[l - 1] : nullptr;
                float* h_out = l == k ? hk : base + ring_off[l] - lo * m->dims[l];
                ProfScope ps(ctx, l == 1 ? PH_AGG_L1 : PH_AGG_REST);
                rc = mg_layer_fused(ctx, d, l, m->dims[l - 1], m->dims[l], m->w_pad_t[l - 1], m->bias[l - 1], h_prev, h_out, l == k ? out2 : nullptr,
                                    (l < k ? 1 : 0) | (m->sum_aggr ? 2 : 0), ctx->ws_meta + meta_at[l], lo, hi, l > 1 ? lo_in : 0, l == 1 ? m->w_pad_h[0] : nullptr, 0, 0, nullptr, nullptr);
                if (rc) return rc;
            }
        }
        MG_CUDA(ctx, cudaGetLastError());
        return finish_forward(ctx, m, d, out, out_mode, hk, out2 != nullptr);
    }

    // per-layer outputs H^1..H^k live in one workspace (kept for mg_layer_output).  A model may ask for fp16
    // intermediates (mg_model_set_intermediates): used when every layer runs in the fused kernel with fp16 weights
    // at hand, the widths allow 64-column output boxes, and nobody needs the fp32 layer outputs afterwards.
    bool f16_inter = m->f16_intermediates && all_fused && !ctx->keep_layers && !m->sum_aggr && k > 1;
    for (int l = 1; l < k && f16_inter; ++l) f16_inter = m->dims[l] % 128 == 0 && m->w_pad_h[l] != nullptr;
    ctx->layers_kept = !f16_inter;
    size_t total = 0;           // bytes
    size_t off[MG_MAX_HOPS + 1];
    for (int l = 1; l < k; ++l) {
        off[l] = total;
        total += (size_t)d->h_hdr.rows_total[l] * m->dims[l] * (f16_inter ? 2 : 4);   // (widths are multiples of 4: 16-byte aligned starts)
    }
    off[k] = 0;   // H^k has buffers of its own
    {
        size_t have = ctx->ws_h_bytes[0] / sizeof(float);
        // a quarter of headroom: the row counts of consecutive calls differ slightly, and growing means a
        // device-wide synchronising free + malloc
        const size_t need = (total + 3) / 4;
        if (have < need && (rc = mg_ensure(ctx, &ctx->ws_h[0], &have, need + need / 4))) return rc;
        ctx->ws_h_bytes[0] = have * sizeof(float);
    }
    char* ws_bytes = reinterpret_cast<char*>(ctx->ws_h[0]);
    int64_t max_x = 0;
    for (int l = 1; l <= k; ++l) {
        if (m->precision == MG_GEMM_TF32 && mg_layer_fused_supported(m->dims[l - 1], m->dims[l])) continue;
        const int64_t rows = std::min<int64_t>(chunk_rows_for(m->dims[l - 1]), d->h_hdr.rows_total[l]);
        max_x = std::max<int64_t>(max_x, rows * 2 * m->dims[l - 1]);
    }
    {
        size_t have = ctx->ws_x_bytes / sizeof(float);
        if (max_x > 0 && (rc = mg_ensure(ctx, &ctx->ws_x, &have, (size_t)max_x))) return rc;
        ctx->ws_x_bytes = have * sizeof(float);
    }

    // What is left for the backward pass beside the kept outputs, in one block.  A bit for each of them: it takes them through a ReLU once more and
    // only has to know which were above zero, a thirty-second of what reading the rows again takes.  And the rows' aggregates, which the weights'
    // gradients want again, where a row has several entries of a layer's outputs: a row to write and to read in place of a row for each
    // entry.  (Layer 1's rows have few entries and come from the table, where the other mini-batches' copies are as many: it gathers again.)
    // Without room for the aggregates, or for either, the backward pass reads the rows.
    {
        int64_t words = 0, bits = 0;
        const auto fused = [&](int l) { return ctx->keep_layers && m->precision == MG_GEMM_TF32 && mg_layer_fused_supported(m->dims[l - 1], m->dims[l]); };
        for (int l = 1; l <= k; ++l) {
            ctx->positive_at[l] = l < k && fused(l) ? words : -1;
            if (ctx->positive_at[l] >= 0) words += mg_positive_words(d->h_hdr.rows_total[l], m->dims[l]);
        }
        bits = words;
        for (int l = 1; l <= k; ++l) {
            ctx->agg_at[l] = l > 1 && fused(l) && (int64_t)d->h_hdr.ent_base[k - l + 1] > kKeepEntriesPerRow * d->h_hdr.rows_total[l] ? words : -1;
            if (ctx->agg_at[l] >= 0) words += (int64_t)d->h_hdr.rows_total[l] * m->dims[l - 1];   // (widths are multiples of 4: 16-byte aligned starts)
        }
        ctx->agg_sum = m->sum_aggr;
        if (ctx->ws_saved_elems < (size_t)words) {
            cudaFree(ctx->ws_saved);
            ctx->ws_saved = nullptr; ctx->ws_saved_elems = 0;
            for (const int64_t want : {words, bits}) {
                if (want < words) for (int l = 1; l <= k; ++l) ctx->agg_at[l] = -1;
                const size_t room = (size_t)(want + want / 4);
                if (want == 0 || cudaMalloc((void**)&ctx->ws_saved, room * sizeof(uint32_t)) == cudaSuccess) { ctx->ws_saved_elems = want ? room : 0; break; }
                cudaGetLastError();
                ctx->ws_saved = nullptr;
            }
            if (!ctx->ws_saved) for (int l = 1; l <= k; ++l) ctx->agg_at[l] = ctx->positive_at[l] = -1;
        }
    }

    const bool half = ctx->feat_dtype == MG_DTYPE_F16;
    for (int l = 1; l <= k; ++l) {
        const int d_in = m->dims[l - 1], d_out = m->dims[l];
        const int64_t M = d->h_hdr.rows_total[l];
        float* h_out = l == k ? hk : reinterpret_cast<float*>(ws_bytes + off[l]);
        const float* h_prev = l > 1 ? reinterpret_cast<const float*>(ws_bytes + off[l - 1]) : nullptr;
        if (m->precision == MG_GEMM_TF32 && mg_layer_fused_supported(d_in, d_out)) {
            // gather + segment mean + both linear maps in one persistent tensor-core kernel
            {
                ProfScope ps(ctx, l == 1 ? PH_AGG_L1 : PH_AGG_REST);
                rc = mg_layer_fused(ctx, d, l, d_in, d_out, m->w_pad_t[l - 1], m->bias[l - 1], h_prev, h_out, l == k ? out2 : nullptr,
                                    (l < k ? 1 : 0) | (m->sum_aggr ? 2 : 0), rows_inline ? nullptr : ctx->ws_meta + meta_at[l], 0, M, 0,
                                    (l == 1 || f16_inter) ? m->w_pad_h[l - 1] : nullptr, f16_inter && l > 1, f16_inter && l < k,
                                    ctx->positive_at[l] >= 0 ? ctx->ws_saved + ctx->positive_at[l] : nullptr,
                                    ctx->agg_at[l] >= 0 ? reinterpret_cast<float*>(ctx->ws_saved + ctx->agg_at[l]) : nullptr);
            }
            if (rc) return rc;
            continue;
        }
        const int64_t chunk = chunk_rows_for(d_in);
        for (int64_t r0 = 0; r0 < M; r0 += chunk) {
            const int64_t r1 = std::min(M, r0 + chunk);
            AggArgs a;
            a.B = B; a.k = k; a.layer = l; a.d_in = d_in;
            a.row_lo = (int32_t)r0; a.row_hi = (int32_t)r1;
            a.rowbase_out = d->rowbase + (size_t)l * (B + 1);
            a.rowbase_in = d->rowbase + (size_t)(l - 1) * (B + 1);
            a.cum = d->cum; a.node_off = d->node_off; a.nodes = d->nodes;
            a.ent_off = d->ent_off; a.ent_nbrs = d->ent_nbrs; a.ent_repr = d->ent_repr;
            a.h_prev = h_prev;
            a.slots = ctx->slots; a.feat = mg_feat_geom(ctx); a.row_bytes = ctx->row_bytes;
            a.x = ctx->ws_x;
            a.round_tf32 = m->precision == MG_GEMM_TF32;
            a.sum_aggr = m->sum_aggr ? 1 : 0;
            {
                ProfScope ps(ctx, l == 1 ? PH_AGG_L1 : PH_AGG_REST);
                const int grid = mg_grid(ctx, 8);
                if (l == 1) { if (half) launch_aggregate<true, true>(a, grid, st); else launch_aggregate<true, false>(a, grid, st); }
                else launch_aggregate<false, false>(a, grid, st);
                ctx->launches++;
            }
            {
                ProfScope ps(ctx, PH_GEMM);
                const int64_t rows = r1 - r0;
                const bool relu = l < k;
                if (m->precision == MG_GEMM_FP32) {
                    dim3 grid((unsigned)((rows + 63) / 64), (unsigned)((d_out + 63) / 64));
                    if (relu) k_gemm_fp32<true><<<grid, 256, 0, st>>>(ctx->ws_x, m->w_cat[l - 1], m->bias[l - 1], h_out + r0 * d_out, rows, d_out, 2 * d_in);
                    else k_gemm_fp32<false><<<grid, 256, 0, st>>>(ctx->ws_x, m->w_cat[l - 1], m->bias[l - 1], h_out + r0 * d_out, rows, d_out, 2 * d_in);
                    ctx->launches++;
                } else {
                    rc = mg_gemm_tf32(ctx, ctx->ws_x, m->w_cat_t[l - 1], m->bias[l - 1], h_out + r0 * d_out, rows, d_out, 2 * d_in, relu);
                    if (rc) return rc;
                }
            }
        }
    }
    MG_CUDA(ctx, cudaGetLastError());
    return finish_forward(ctx, m, d, out, out_mode, hk, out2 != nullptr);
}

static int forward_impl(mg_ctx* ctx, const mg_model* m, mg_dense* d, float* out, int out_mode) {
    if (!ctx) return MG_ERR_ARG;
    if (int rc = forward_checks(ctx, m, d)) return rc;
    if (!out) return mg_fail(ctx, MG_ERR_ARG, "null output");
    MG_CUDA(ctx, cudaSetDevice(ctx->device));
    // a pass that ends in an error leaves neither layer outputs nor anything that mg_backward may follow
    ctx->last_fwd_model = nullptr; ctx->last_fwd_dense = nullptr; ctx->last_hk = nullptr;
    const int rc = forward_pass(ctx, m, d, out, out_mode);
    if (rc) { ctx->last_hk = nullptr; return rc; }
    ctx->last_fwd_model = m; ctx->last_fwd_dense = d;
    return MG_OK;
}

extern "C" int mg_forward(mg_ctx* ctx, const mg_model* m, mg_dense* d, float* out, int out_on_device) {
    return forward_impl(ctx, m, d, out, out_on_device ? OUT_DEVICE : OUT_HOST);
}

extern "C" int mg_forward_host_async(mg_ctx* ctx, const mg_model* m, mg_dense* d, float* out_host) {
    return forward_impl(ctx, m, d, out_host, OUT_HOST_ASYNC);
}

extern "C" int mg_wait_output(mg_ctx* ctx) {
    if (!ctx) return MG_ERR_ARG;
    MG_CUDA(ctx, cudaSetDevice(ctx->device));
    MG_CUDA(ctx, cudaEventSynchronize(ctx->ev_out_done));   // completes at once when nothing was recorded
    if (ctx->out_check_gemm) { ctx->out_check_gemm = false; return mg_gemm_tf32_status(ctx); }
    return MG_OK;
}

extern "C" int mg_gather_h0(mg_ctx* ctx, mg_dense* d, int32_t batch, float* out_dev) {
    if (!ctx) return MG_ERR_ARG;
    if (!d || !out_dev) return mg_fail(ctx, MG_ERR_ARG, "null argument");
    if (!d->valid) return mg_fail(ctx, MG_ERR_STATE, "mg_dense holds no completed sample");
    if (!ctx->slots || ctx->feat_dim <= 0) return mg_fail(ctx, MG_ERR_STATE, "no feature table loaded");
    if (batch < 0 || batch >= d->n_batches) return mg_fail(ctx, MG_ERR_ARG, "batch out of range");
    if (int rs = mg_check_sample_residency(ctx, d)) return rs;
    MG_CUDA(ctx, cudaSetDevice(ctx->device));
    H0Args a;
    fill_row_export(d, batch, 0, ctx->feat_dim, &a.r);
    {
        const int32_t* inv_unused;
        const int rc0 = mg_dense_batch_perm(ctx, d, batch, &a.r.perm, &inv_unused);   // rows come in the paper's order
        if (rc0) return rc0;
    }
    for (int h = 0; h <= d->k; ++h) a.node_off[h] = d->h_node_off[(size_t)h * (d->n_batches + 1) + batch];
    a.nodes = d->nodes; a.slots = ctx->slots; a.feat = mg_feat_geom(ctx); a.row_bytes = ctx->row_bytes;
    if (a.r.n_rows > 0) {
        if (ctx->feat_dtype == MG_DTYPE_F16) k_gather_h0<true><<<mg_grid(ctx, 4), kThreads, 0, ctx->stream>>>(a, out_dev);
        else k_gather_h0<false><<<mg_grid(ctx, 4), kThreads, 0, ctx->stream>>>(a, out_dev);
        ctx->launches++;
    }
    MG_CUDA(ctx, cudaGetLastError());
    MG_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
    return MG_OK;
}

extern "C" int mg_layer_output(mg_ctx* ctx, const mg_model* m, mg_dense* d, int32_t layer, int32_t batch, float* out_dev) {
    if (!ctx) return MG_ERR_ARG;
    int rc = forward_checks(ctx, m, d);
    if (rc) return rc;
    if (!out_dev) return mg_fail(ctx, MG_ERR_ARG, "null output");
    if (layer < 1 || layer > d->k) return mg_fail(ctx, MG_ERR_ARG, "layer must be in [1, k]");
    if (batch < 0 || batch >= d->n_batches) return mg_fail(ctx, MG_ERR_ARG, "batch out of range");
    if (!ctx->last_hk) return mg_fail(ctx, MG_ERR_STATE, "mg_forward has not run");
    if (!ctx->layers_kept) return mg_fail(ctx, MG_ERR_STATE, "the last forward did not keep its intermediate layers: call mg_keep_layer_outputs(ctx, 1) first");
    MG_CUDA(ctx, cudaSetDevice(ctx->device));
    size_t off = 0;   // bytes; the layers were kept as fp32 (layers_kept)
    for (int l = 1; l < layer; ++l) off += (size_t)d->h_hdr.rows_total[l] * m->dims[l] * 4;
    const int B = d->n_batches;
    const float* layer_base = layer == d->k ? ctx->last_hk : reinterpret_cast<const float*>(reinterpret_cast<const char*>(ctx->ws_h[0]) + off);
    if (!layer_base) return mg_fail(ctx, MG_ERR_STATE, "mg_forward has not run");
    const float* src = layer_base + (size_t)d->h_rowbase[(size_t)layer * (B + 1) + batch] * m->dims[layer];
    RowExportArgs r;
    fill_row_export(d, batch, layer, m->dims[layer], &r);
    {
        const int32_t* inv_unused;
        if ((rc = mg_dense_batch_perm(ctx, d, batch, &r.perm, &inv_unused))) return rc;
    }
    if (r.n_rows > 0) {
        k_export_rows<<<mg_grid(ctx, 4), kThreads, 0, ctx->stream>>>(r, src, out_dev);
        ctx->launches++;
    }
    MG_CUDA(ctx, cudaGetLastError());
    MG_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
    return MG_OK;
}

// ---------------------------------------------------------------------------------------
// Backward pass through the GraphSage layers (Section 3: the gradients of a mini-batch update the model and the
// base representations).  Chain rule through Algorithm 3 and Algorithm 2, layer k down to layer 1, whole layers at a time:
//   dPre = dH^l (masked by H^l > 0 below the last layer),
//   dW += X^T dPre with X = [self | aggregate] from H^{l-1} (kept by the forward pass): the self rows gathered again, the aggregates
//   too unless the forward pass has left them, dbias += column sums of dPre, dX = dPre W^T,
//   dH^{l-1}[row] = its self part of dX + the neighbour parts of every entry that names it, times 1 / count (1 for a sum).
// A model with TF32 products takes dW and dX on the tensor cores (X, dPre and W as they lie in memory, of which the tensor cores
// read ten bits of the mantissa; fp32 accumulate), one with fp32 products on CUDA cores, there with X in chunks of rows.  All
// other sums are fp32.  Sums over rows meet by atomic adds, so low-order bits vary from run to run.
// ---------------------------------------------------------------------------------------
namespace {

struct RowGeom {
    int32_t B, k;
    const int32_t* rowbase;   // [(k + 1)][B + 1]
    const int32_t* cum;       // [B][k + 2]
    const int32_t* node_off;  // [(k + 1)][B + 1]
};

// packed row of layer `layer` -> its mini-batch, its local row, its place in the hop-major node list
__device__ __forceinline__ void locate_row(const RowGeom& g, int layer, int64_t row, int32_t* b_out, int32_t* local_out, int32_t* node_out) {
    const int32_t* rb = g.rowbase + (int64_t)layer * (g.B + 1);
    int lo = 0, hi = g.B;   // rb[lo] <= row < rb[hi]
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if ((int64_t)rb[mid] <= row) lo = mid; else hi = mid;
    }
    const int32_t local = (int32_t)(row - rb[lo]);
    const int32_t* cum = g.cum + (int64_t)lo * (g.k + 2);
    int j = 0;
    while (j + 1 <= g.k && cum[j + 1] <= local) ++j;
    *b_out = lo; *local_out = local;
    *node_out = g.node_off[(int64_t)j * (g.B + 1) + lo] + (local - cum[j]);
}

// The gradient of the last layer's bias: db += column sums of g (below it, k_grad_gather sums the bias on its way).  A thread keeps
// four columns and walks down the rows (16-byte accesses, two rows in flight, a block covers whole rows); column sums meet in shared
// memory, one atomic add per column and block.
__global__ void __launch_bounds__(kThreads) k_grad_bias(const float* __restrict__ g, float* db, int64_t rows, int N) {
    __shared__ float sums[1024];
    const int n4 = N / 4;                       // (widths are multiples of 4, at most 1024)
    const int rows_per_pass = kThreads / n4;    // >= 1
    for (int c = threadIdx.x; c < N; c += kThreads) sums[c] = 0.f;
    __syncthreads();
    const int c4 = threadIdx.x % n4, rr = threadIdx.x / n4;
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
    if (rr < rows_per_pass) {
        const float4* g4 = reinterpret_cast<const float4*>(g);
        const int64_t step = (int64_t)gridDim.x * rows_per_pass;
        for (int64_t r = (int64_t)blockIdx.x * rows_per_pass + rr; r < rows; r += 2 * step) {
            const float4 v0 = g4[r * n4 + c4], v1 = r + step < rows ? g4[(r + step) * n4 + c4] : make_float4(0.f, 0.f, 0.f, 0.f);
            s.x += v0.x + v1.x; s.y += v0.y + v1.y; s.z += v0.z + v1.z; s.w += v0.w + v1.w;
        }
        atomicAdd(&sums[4 * c4], s.x); atomicAdd(&sums[4 * c4 + 1], s.y); atomicAdd(&sums[4 * c4 + 2], s.z); atomicAdd(&sums[4 * c4 + 3], s.w);
    }
    __syncthreads();
    for (int c = threadIdx.x; c < N; c += kThreads) atomicAdd(&db[c], sums[c]);
}

// dW[Kx, N] += X[rows, Kx]^T dPre[rows, N]; a block owns a 64 x 64 tile of dW and a slice of the rows
constexpr int kGradRowsPerBlock = 1024;
__global__ void __launch_bounds__(256) k_grad_weights(const float* __restrict__ x, const float* __restrict__ dpre, float* dw,
                                                      int64_t rows, int Kx, int N) {
    constexpr int T = 64, BR = 16;
    __shared__ float xs[BR][T + 4];
    __shared__ float gs[BR][T + 4];
    const int k0 = blockIdx.x * T, n0 = blockIdx.y * T;
    const int64_t r_lo = (int64_t)blockIdx.z * kGradRowsPerBlock, r_hi = min(rows, r_lo + kGradRowsPerBlock);
    const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
    float acc[4][4] = {};
    for (int64_t r0 = r_lo; r0 < r_hi; r0 += BR) {
        for (int i = threadIdx.x; i < BR * T; i += 256) {
            const int rr = i / T, c = i % T;
            const bool on = r0 + rr < r_hi;
            xs[rr][c] = (on && k0 + c < Kx) ? x[(r0 + rr) * Kx + k0 + c] : 0.f;
            gs[rr][c] = (on && n0 + c < N) ? dpre[(r0 + rr) * N + n0 + c] : 0.f;
        }
        __syncthreads();
#pragma unroll
        for (int rr = 0; rr < BR; ++rr) {
            float xv[4], gv[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) { xv[i] = xs[rr][ty * 4 + i]; gv[i] = gs[rr][tx * 4 + i]; }
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(xv[i], gv[j], acc[i][j]);
        }
        __syncthreads();
    }
    for (int i = 0; i < 4; ++i)
        for (int j = 0; j < 4; ++j) {
            const int kk = k0 + ty * 4 + i, n = n0 + tx * 4 + j;
            if (kk < Kx && n < N) atomicAdd(&dw[(int64_t)kk * N + n], acc[i][j]);
        }
}

// ---- dX of a layer -> the gradient of the layer's input rows ----
// A source row receives the self part of its own output row and a share of the neighbour part of every output row that
// aggregates it.  Instead of adding row by row with atomics (a read-modify-write of the target for every sampled
// entry), the entries of all layers are first turned round -- for every source row the list of (output row, weight) that
// name it: a count per source row, an exclusive scan, a fill; three kernels for all layers together, as none of it depends on
// a gradient -- and a warp then sums a source row's contributions in registers and stores the row once, through the ReLU of
// the layer below and into that layer's bias gradient on the way.
constexpr int kGradLight = 8;     // a source row named by more entries than this is cut into units of its own
constexpr int kGradUnit = 64;     // entries per unit
struct RevArgs {
    RowGeom g;
    int32_t l0;                        // first layer that hands its dX down
    int64_t out_at[MG_MAX_HOPS + 2];   // layer l's output rows are items [out_at[l], out_at[l + 1])
    int64_t in_at[MG_MAX_HOPS + 2];    // its source rows are places [in_at[l], in_at[l + 1]) of cnt
    int64_t ent_at[MG_MAX_HOPS + 2];   // its entries' places in pos
    int32_t rows_per_warp;             // of k_rev_entries: 4 to 32
    const int4* meta;                  // of the output rows: first entry, entries, first source row of the mini-batch (mg_layer_rows)
    const int32_t* ent_repr;
    uint32_t* cnt;                     // [in_at[k + 1] + 1]: counts, then (scanned) where the lists start
    uint32_t* pos;                     // an entry's place in its source row's list, left by the count for the fill
    int2* rev;                         // (output row, weight as float bits)
    int32_t sum_aggr;
    // the scan: a 64-bit state per tile (decoupled look-back), a tile counter
    uint64_t* state;
    uint32_t* ticket;
    // units of the rows with long lists: (row of the layer, its unit), per layer
    int64_t unit_at[MG_MAX_HOPS + 2];
    int2* units;
    uint32_t* n_units;                 // [k + 1]
    float* g_in[MG_MAX_HOPS + 1];      // the layer's source rows' gradients; rows of several units are cleared here
    int32_t d_in[MG_MAX_HOPS + 1];
    int32_t polls;                     // reads of a tile's state before the scan gives up
    uint32_t* bad;                     // set when it has: the lists are then wrong, and the kernels behind it leave them alone
    uint32_t* status;                  // the host's word
};

// A warp takes 32 output rows (fewer where there would not be a warp for every slot of the SMs), lane = row: its metadata is one load.  Their entries are then read as one stream, four per lane in flight,
// each lane looking up whose its entry is.  Bound by the scattered atomics and list places in L2.  (Eight lanes per row, each row
// found by a search over the mini-batches, took 2 x 55 us for the 3.7M entries of 24 mini-batches, now 34 + 36.)
template <bool FILL>
__global__ void __launch_bounds__(kThreads) k_rev_entries(RevArgs a) {
    if (FILL && *a.bad) return;
    constexpr int U = 4;
    const int lane = threadIdx.x & 31;
    const int64_t total = a.out_at[a.g.k + 1], step = (int64_t)gridDim.x * (kThreads / 32) * a.rows_per_warp;
    for (int64_t i0 = (blockIdx.x * (int64_t)(kThreads / 32) + (threadIdx.x >> 5)) * a.rows_per_warp; i0 < total; i0 += step) {
        const int64_t i = min(i0 + lane, total - 1);
        int layer = a.l0;
        while (i >= a.out_at[layer + 1]) ++layer;
        const int4 m = __ldg(a.meta + i);
        const int32_t n = lane < a.rows_per_warp && i0 + lane < total ? m.z : 0;
        const int32_t end = (int32_t)warp_incl_scan((uint32_t)n), all = __shfl_sync(0xFFFFFFFFu, end, 31);
        const int32_t row = (int32_t)(i - a.out_at[layer]);
        const int32_t ent = m.y - (end - n);                        // entry j of the stream is ent + j of the arena
        const int64_t src0 = a.in_at[layer] + m.w;                  // row 0 of the mini-batch among the layer's source rows
        const int64_t pos0 = a.ent_at[layer] + ent;
        const float w = a.sum_aggr ? 1.f : 1.f / (float)m.z;
        for (int32_t j0 = 0; j0 < all; j0 += 32 * U) {
            int32_t repr[U], own[U];
            uint32_t at[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int32_t j = min(j0 + u * 32 + lane, all - 1);
                int o = 0;   // the first row whose entries end behind j
#pragma unroll
                for (int s = 16; s > 0; s >>= 1)
                    if (__shfl_sync(0xFFFFFFFFu, end, o + s - 1) <= j) o += s;
                own[u] = o;
                repr[u] = __ldg(a.ent_repr + __shfl_sync(0xFFFFFFFFu, ent, o) + j);
                if (FILL) at[u] = a.pos[__shfl_sync(0xFFFFFFFFu, pos0, o) + j];
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int64_t src = __shfl_sync(0xFFFFFFFFu, src0, own[u]) + repr[u];
                const bool on = j0 + u * 32 + lane < all;
                if (FILL) at[u] += a.cnt[src];
                else if (on) at[u] = atomicAdd(&a.cnt[src], 1u);
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int32_t j = j0 + u * 32 + lane;
                if (FILL) {
                    const int2 item = make_int2(__shfl_sync(0xFFFFFFFFu, row, own[u]), __shfl_sync(0xFFFFFFFFu, __float_as_int(w), own[u]));
                    if (j < all) a.rev[at[u]] = item;
                } else {
                    const int64_t p = __shfl_sync(0xFFFFFFFFu, pos0, own[u]) + j;
                    if (j < all) a.pos[p] = at[u];
                }
            }
        }
    }
}

// exclusive scan of the counts in place, the total behind them; the rows with long lists are cut into units on the way.
constexpr int kRevTile = kThreads * 16;
__global__ void __launch_bounds__(kThreads) k_rev_scan(RevArgs a) {
    __shared__ uint32_t part[kThreads / 32];
    __shared__ uint32_t sh_before;
    __shared__ int32_t sh_tile;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t n = a.in_at[a.g.k + 1], n_tiles = (n + kRevTile - 1) / kRevTile;
    if (threadIdx.x == 0) sh_tile = (int32_t)atomicAdd(a.ticket, 1u);   // (a block per tile)
    __syncthreads();
    const int32_t tile = sh_tile;
    const int64_t t0 = (int64_t)tile * kRevTile + (int64_t)threadIdx.x * 16;   // 16 consecutive elements per thread
    uint32_t v[16], s = 0, my_units = 0;
#pragma unroll
    for (int q = 0; q < 4; ++q) {   // (the counts start on a 16-byte boundary)
        uint4 x = make_uint4(0u, 0u, 0u, 0u);
        if (t0 + 4 * q + 3 < n) x = *reinterpret_cast<const uint4*>(a.cnt + t0 + 4 * q);
        else {
            if (t0 + 4 * q < n) x.x = a.cnt[t0 + 4 * q];
            if (t0 + 4 * q + 1 < n) x.y = a.cnt[t0 + 4 * q + 1];
            if (t0 + 4 * q + 2 < n) x.z = a.cnt[t0 + 4 * q + 2];
        }
        v[4 * q] = x.x; v[4 * q + 1] = x.y; v[4 * q + 2] = x.z; v[4 * q + 3] = x.w;
    }
#pragma unroll
    for (int i = 0; i < 16; ++i) { s += v[i]; if (v[i] > kGradLight) my_units += (v[i] + kGradUnit - 1) / kGradUnit; }
    const uint32_t inc = warp_incl_scan(s);
    if (lane == 31) part[warp] = inc;
    __syncthreads();
    if (warp == 0) {
        const uint32_t w = lane < kThreads / 32 ? part[lane] : 0u;
        const uint32_t wi = warp_incl_scan(w);
        const uint32_t total = __shfl_sync(0xFFFFFFFFu, wi, 31);
        if (lane < kThreads / 32) part[lane] = wi - w;
        bool gave_up = false;
        const uint32_t before = chain_tiles(a.state, tile, kChainTag, 0u, total, a.polls, &gave_up);
        if (gave_up) { *a.bad = 1u; *reinterpret_cast<volatile uint32_t*>(a.status) = MG_ROLE_REV_SCAN; }
        if (lane == 0) {
            sh_before = before;
            if (tile == n_tiles - 1) a.cnt[n] = before + total;
        }
    }
    __syncthreads();
    uint32_t run = sh_before + part[warp] + inc - s;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const uint4 x = make_uint4(run, run + v[4 * q], run + v[4 * q] + v[4 * q + 1], run + v[4 * q] + v[4 * q + 1] + v[4 * q + 2]);
        run = x.w + v[4 * q + 3];
        if (t0 + 4 * q + 3 < n) *reinterpret_cast<uint4*>(a.cnt + t0 + 4 * q) = x;
        else {
            if (t0 + 4 * q < n) a.cnt[t0 + 4 * q] = x.x;
            if (t0 + 4 * q + 1 < n) a.cnt[t0 + 4 * q + 1] = x.y;
            if (t0 + 4 * q + 2 < n) a.cnt[t0 + 4 * q + 2] = x.z;
        }
    }
    if (my_units == 0) return;
    // one atomic for the thread's units, or one per row where its rows belong to two layers
    int layer = a.l0;
    while (t0 >= a.in_at[layer + 1]) ++layer;
    const bool one_layer = t0 + 16 <= a.in_at[layer + 1];
    uint32_t at = one_layer ? atomicAdd(&a.n_units[layer], my_units) : 0u;
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        if (v[i] <= kGradLight) continue;
        while (t0 + i >= a.in_at[layer + 1]) ++layer;
        const int32_t row = (int32_t)(t0 + i - a.in_at[layer]);
        const uint32_t parts = (v[i] + kGradUnit - 1) / kGradUnit;
        if (!one_layer) at = atomicAdd(&a.n_units[layer], parts);
        for (uint32_t q = 0; q < parts; ++q) a.units[a.unit_at[layer] + at + q] = make_int2(row, (int32_t)q);
        at += parts;
        if (parts > 1) {
            float4* g = reinterpret_cast<float4*>(a.g_in[layer] + (int64_t)row * a.d_in[layer]);
            for (int c = 0; c < a.d_in[layer] / 4; ++c) g[c] = make_float4(0.f, 0.f, 0.f, 0.f);
        }
    }
}

struct GatherArgs {
    RowGeom g;
    int32_t layer;             // the layer whose dX is handed down (1 .. k); its inputs are the rows of layer - 1
    int64_t rows_in;
    const uint32_t* off;       // [rows_in + 1] where the rows' lists start
    const int2* rev;
    const int2* units;
    const uint32_t* n_units;
    const uint32_t* bad;       // the scan gave up: there are no lists
    const float* dx;           // [rows of layer, 2 d_in]
    int32_t d_in;
    const float* y;            // [rows_in, d_in] kept outputs of layer - 1 (RELU_ROWS), else null
    const uint32_t* positive;  // which of them are above zero, mg_positive_words (RELU_BITS), else null
    float* g_in;               // [rows_in, d_in]
    float* db;                 // [d_in] bias gradient of layer - 1 (with a ReLU)
};

// Bound by the latency of scattered 512-byte row reads.  A warp works on 128 columns of 16 consecutive source rows, or of one
// unit of a row with a long list (a hub of the graph is named by hundreds of entries; one warp reading them one after the
// other set the kernel's time).  Its contributions -- self parts and entries, row after row -- are first listed in shared
// memory, lane = row, and then read as one stream, U loads of 512 bytes in flight whatever rows they belong to, with the kept
// outputs of the rows that end among them beside, or, where the forward pass has left bits of them, one word per column for
// all rows of the group.  Rows of several units are added up by atomics: mask and bias are
// linear in the sum.  24 mini-batches of 1,000 targets on 2M nodes: 1.56M rows x 128 in 685 -> 367 us with eight loads in flight and three
// blocks per SM, 342 with six and four (four and five: 362), 543k + 92k rows x 256 in
// 445 -> 388 us (bits: 213 us); 8 mini-batches on 1M nodes, 181k + 34k rows x 256 in 250 -> 141 us (bits: 83 us).  (With the outputs
// read: four blocks per SM at 64 registers; three at 72 take 481 / 178 us.)
constexpr int kGradRows = 16, kGradItems = kGradRows * (kGradLight + 1);
static_assert(kGradItems >= kGradUnit + 1, "a unit's items fit the list");
constexpr int64_t kGradMaxRows = (1ll << 30) - 1;   // an item holds twice its output row, and one more, in 31 bits; the largest value means none
static_assert(2 * (kGradMaxRows - 1) + 1 < 0x7FFFFFFFll, "an output row's item is not the one that means none");
enum { RELU_NONE = 0, RELU_ROWS = 1, RELU_BITS = 2 };
template <int RELU>
__global__ void __launch_bounds__(kThreads, 4) k_grad_gather(GatherArgs a) {
    constexpr bool MASK = RELU != RELU_NONE;
    constexpr int U = RELU == RELU_NONE ? 6 : 4, kWarps = kThreads / 32;
    constexpr uint32_t kNone = 0x7FFFFFFFu;       // an item without a contribution
    __shared__ int2 items_sm[kWarps][kGradItems];   // 2 x output row + (1: its neighbour part), weight; sign: the row's last item
    __shared__ int32_t rows_sm[kWarps][kGradRows];
    __shared__ float sums[MASK ? 1024 : 1];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (*a.bad) return;
    int2* items = items_sm[warp];
    int32_t* rows = rows_sm[warp];
    const int n4 = a.d_in / 4;
    int blocks_log = 0;                           // column blocks of 128, a power of two of them (widths go up to 1,024)
    while ((128 << blocks_log) < a.d_in) ++blocks_log;
    const int c4 = (warp & ((1 << blocks_log) - 1)) * 32 + lane;
    const bool on = c4 < n4;
    const int32_t* rb_in = a.g.rowbase + (int64_t)(a.layer - 1) * (a.g.B + 1);
    const int32_t* rb_out = rb_in + (a.g.B + 1);
    const float4* __restrict__ dx = reinterpret_cast<const float4*>(a.dx) + c4;
    const float4 zero4 = make_float4(0.f, 0.f, 0.f, 0.f);
    float4 bias = zero4;
    if (MASK) {
        for (int c = threadIdx.x; c < 1024; c += kThreads) sums[c] = 0.f;
        __syncthreads();
    }
    // output row of source row s, -1 where it has none (rows of the farthest delta)
    auto self_of = [&](int64_t s) -> int32_t {
        int lo = 0, hi = a.g.B;
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if ((int64_t)rb_in[mid] <= s) lo = mid; else hi = mid;
        }
        const int32_t local = (int32_t)(s - rb_in[lo]);
        return local < rb_out[lo + 1] - rb_out[lo] ? rb_out[lo] + local : -1;
    };
    const int64_t n_units = *a.n_units, total = n_units + (a.rows_in + kGradRows - 1) / kGradRows;
    const int per_block = kWarps >> blocks_log;
    for (int64_t w = (int64_t)blockIdx.x * per_block + (warp >> blocks_log); w < total; w += (int64_t)gridDim.x * per_block) {
        int n_items = 0;
        bool add = false;
        if (w < n_units) {
            const int2 un = a.units[w];
            const uint32_t j0 = a.off[un.x], j1 = a.off[un.x + 1];
            const uint32_t first = j0 + (uint32_t)un.y * kGradUnit;
            const int n = (int)min((uint32_t)kGradUnit, j1 - first);
            const int32_t self = un.y == 0 ? self_of(un.x) : -1;
            const int at = self >= 0 ? 1 : 0;
            add = j1 - j0 > kGradUnit;
            n_items = n + at;
            for (int i = lane; i < n; i += 32) {
                const int2 r = a.rev[first + i];
                items[at + i] = make_int2((int)((2u * (uint32_t)r.x + 1u) | (i == n - 1 ? 0x80000000u : 0u)), r.y);
            }
            if (lane == 0) {
                rows[0] = un.x;
                if (at) items[0] = make_int2(2 * self, __float_as_int(1.f));
            }
        } else {
            const int64_t s = (w - n_units) * kGradRows + lane;
            uint32_t j0 = 0, c = kGradLight + 1;
            if (lane < kGradRows && s < a.rows_in) { j0 = a.off[s]; c = a.off[s + 1] - j0; }
            const bool mine = c <= kGradLight;
            const int32_t self = mine ? self_of(s) : -1;
            const int n = mine ? max(1, (int)c + (self >= 0 ? 1 : 0)) : 0;
            const uint32_t end = warp_incl_scan((uint32_t)n);
            n_items = (int)__shfl_sync(0xFFFFFFFFu, end, 31);
            const uint32_t rowmask = __ballot_sync(0xFFFFFFFFu, mine);
            if (mine) {
                int at = (int)end - n;
                if (self >= 0) items[at++] = make_int2(2 * self, __float_as_int(1.f));
                for (uint32_t q = 0; q < c; ++q) {
                    const int2 r = a.rev[j0 + q];
                    items[at++] = make_int2(2 * r.x + 1, r.y);
                }
                if (self < 0 && c == 0) items[at] = make_int2((int)kNone, 0);
                items[end - 1].x |= (int)0x80000000u;
                rows[__popc(rowmask & ((1u << lane) - 1u))] = (int32_t)s;
            }
        }
        // (16 consecutive rows that start at a multiple of 16, or one row: their bits share a word per column)
        uint4 pos = make_uint4(0u, 0u, 0u, 0u);
        if (RELU == RELU_BITS && on) {
            const int64_t row = w < n_units ? a.units[w].x : (w - n_units) * kGradRows;
            pos = __ldg(reinterpret_cast<const uint4*>(a.positive) + (row >> 5) * n4 + c4);
        }
        __syncwarp();
        float4 acc = zero4;
        int row_i = 0, row_l = 0;   // the row that the sums and the loads have come to
        for (int t = 0; t < n_items; t += U) {
            float4 v[U], yv[RELU == RELU_ROWS ? U : 1];
            int2 it[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                it[u] = items[min(t + u, n_items - 1)];
                const uint32_t src = (uint32_t)it[u].x & 0x7FFFFFFFu;
                v[u] = zero4;
                if (on && t + u < n_items && src != kNone) v[u] = __ldg(dx + (int64_t)src * n4);
                if (RELU == RELU_ROWS) {
                    yv[u] = zero4;
                    if (t + u < n_items && it[u].x < 0) {
                        if (on) yv[u] = __ldg(reinterpret_cast<const float4*>(a.y) + (int64_t)rows[row_l] * n4 + c4);
                        ++row_l;
                    }
                }
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if (t + u >= n_items) break;
                const float wt = __int_as_float(it[u].y);
                acc.x = fmaf(wt, v[u].x, acc.x); acc.y = fmaf(wt, v[u].y, acc.y); acc.z = fmaf(wt, v[u].z, acc.z); acc.w = fmaf(wt, v[u].w, acc.w);
                if (it[u].x >= 0) continue;
                if (MASK) {
                    if (RELU == RELU_ROWS)
                        acc = make_float4(yv[u].x > 0.f ? acc.x : 0.f, yv[u].y > 0.f ? acc.y : 0.f, yv[u].z > 0.f ? acc.z : 0.f, yv[u].w > 0.f ? acc.w : 0.f);
                    else {
                        const int bit = rows[row_i] & 31;
                        acc = make_float4(pos.x >> bit & 1u ? acc.x : 0.f, pos.y >> bit & 1u ? acc.y : 0.f, pos.z >> bit & 1u ? acc.z : 0.f,
                                          pos.w >> bit & 1u ? acc.w : 0.f);
                    }
                    bias.x += acc.x; bias.y += acc.y; bias.z += acc.z; bias.w += acc.w;
                }
                if (on) {
                    float4* dst = reinterpret_cast<float4*>(a.g_in) + (int64_t)rows[row_i] * n4 + c4;
                    if (add) atomicAdd(dst, acc);
                    else *dst = acc;
                }
                ++row_i;
                acc = zero4;
            }
        }
        __syncwarp();
    }
    if (MASK) {
        if (on) {
            atomicAdd(&sums[4 * c4], bias.x); atomicAdd(&sums[4 * c4 + 1], bias.y);
            atomicAdd(&sums[4 * c4 + 2], bias.z); atomicAdd(&sums[4 * c4 + 3], bias.w);
        }
        __syncthreads();
        for (int c = threadIdx.x; c < a.d_in; c += kThreads) atomicAdd(&a.db[c], sums[c]);
    }
}

struct PackedIdArgs {
    RowGeom g;
    const int32_t* nodes;
    int64_t n_rows;
    int32_t* ids;
};

__global__ void __launch_bounds__(kThreads) k_packed_ids(PackedIdArgs a) {
    for (int64_t row = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; row < a.n_rows; row += (int64_t)gridDim.x * blockDim.x) {
        int32_t b, local, node;
        locate_row(a.g, 0, row, &b, &local, &node);
        a.ids[row] = a.nodes[node];
    }
}

}  // namespace

static void launch_packed_ids(mg_ctx* ctx, const mg_dense* d, int32_t* ids_dev) {
    PackedIdArgs a{{d->n_batches, d->k, d->rowbase, d->cum, d->node_off}, d->nodes, d->h_hdr.rows_total[0], ids_dev};
    if (a.n_rows <= 0) return;
    k_packed_ids<<<mg_grid(ctx, 4), kThreads, 0, ctx->stream>>>(a);
    ctx->launches++;
}

extern "C" int mg_backward_begin(mg_ctx* ctx, mg_model* m, mg_dense* d, const float* d_out_dev, float* d_h0_dev, int32_t* ids_dev,
                                 float* grads_dev, void* grads_stream) {
    if (!ctx) return MG_ERR_ARG;
    int rc = forward_checks(ctx, m, d);
    if (rc) return rc;
    if (!d_out_dev) return mg_fail(ctx, MG_ERR_ARG, "null output gradient");
    if (!ctx->last_hk || ctx->last_fwd_model != m || ctx->last_fwd_dense != d)
        return mg_fail(ctx, MG_ERR_STATE, "mg_backward follows mg_forward of the same model and sample");
    if (!ctx->layers_kept) return mg_fail(ctx, MG_ERR_STATE, "the forward pass did not keep its intermediate layers: call mg_keep_layer_outputs(ctx, 1) first");
    MG_CUDA(ctx, cudaSetDevice(ctx->device));
    const int k = d->k, B = d->n_batches;
    cudaStream_t st = ctx->stream;
    if (grads_dev && (cudaStream_t)grads_stream != st) {   // the caller's buffers are as its stream leaves them
        MG_CUDA(ctx, cudaEventRecord(ctx->ev_user, (cudaStream_t)grads_stream));
        MG_CUDA(ctx, cudaStreamWaitEvent(st, ctx->ev_user));
    }
    // gradient block of the model (allocated once), cleared for this pass
    if (!m->g_block) {
        m->g_elems = 0;
        for (int l = 0; l < k; ++l) m->g_elems += (size_t)(2 * m->dims[l] + 1) * m->dims[l + 1];
        if (mg_malloc(ctx, (void**)&m->g_block, m->g_elems * sizeof(float)) != cudaSuccess) { cudaGetLastError(); m->g_block = nullptr; return mg_fail(ctx, MG_ERR_OOM, "gradient allocation failed"); }
        float* g = m->g_block;
        for (int l = 0; l < k; ++l) {
            m->g_w_cat[l] = g; g += (size_t)2 * m->dims[l] * m->dims[l + 1];
            m->g_bias[l] = g; g += m->dims[l + 1];
        }
    }
    MG_CUDA(ctx, mg_reads_wait(&m->g_reads, st));   // (the last pass's gradients may still be on their way to the caller)
    m->g_reads.queued = false;
    MG_CUDA(ctx, cudaMemsetAsync(m->g_block, 0, m->g_elems * sizeof(float), st));
    if (!m->zeros) {
        if (mg_malloc(ctx, (void**)&m->zeros, sizeof(float) * 2 * 1024) != cudaSuccess) { cudaGetLastError(); return mg_fail(ctx, MG_ERR_OOM, "gradient allocation failed"); }
        MG_CUDA(ctx, cudaMemsetAsync(m->zeros, 0, sizeof(float) * 2 * 1024, st));
    }
    // scratch: dH^1 .. dH^{k-1}, the X rows of a chunk (fp32 products only), dX of a layer, the turned-round entries of the layers whose dX is handed down
    size_t g_off[MG_MAX_HOPS + 1] = {0}, g_total = 0, h_off[MG_MAX_HOPS + 1] = {0}, h_total = 0;
    for (int l = 1; l < k; ++l) {
        g_off[l] = g_total; g_total += ((size_t)d->h_hdr.rows_total[l] * m->dims[l] + 7) / 8 * 8;   // (32-byte aligned starts)
        h_off[l] = h_total; h_total += (size_t)d->h_hdr.rows_total[l] * m->dims[l];
    }
    // (chunks 16 times the forward pass's: nothing here gains from a chunk that stays in L2, and fewer, longer launches
    // mean fewer atomic adds into the weight gradients: 18.2 -> 14.6 ms at 128 mini-batches of the 1M-node workload)
    const int64_t bw_mult = 16;
    int64_t max_x = 0, max_dx = 0;
    RevArgs ra;
    memset(&ra, 0, sizeof(ra));
    ra.l0 = d_h0_dev ? 1 : 2;
    for (int l = 1; l <= k; ++l) {
        if (m->precision == MG_GEMM_FP32)
            max_x = std::max<int64_t>(max_x, std::min<int64_t>(bw_mult * chunk_rows_for(m->dims[l - 1]), d->h_hdr.rows_total[l]) * 2 * m->dims[l - 1]);
        const bool down = l >= ra.l0;
        const int64_t entries = down ? d->h_hdr.ent_base[k - l + 1] : 0;
        if (down) max_dx = std::max<int64_t>(max_dx, (int64_t)d->h_hdr.rows_total[l] * 2 * m->dims[l - 1]);
        ra.out_at[l + 1] = ra.out_at[l] + (down ? d->h_hdr.rows_total[l] : 0);
        ra.in_at[l + 1] = ra.in_at[l] + (down ? d->h_hdr.rows_total[l - 1] : 0);
        ra.ent_at[l + 1] = ra.ent_at[l] + entries;
        ra.unit_at[l + 1] = ra.unit_at[l] + entries / kGradLight + 1;   // (a row of c > 8 entries has ceil(c / 64) <= c / 8 units)
    }
    const int64_t in_total = ra.in_at[k + 1], ent_total = ra.ent_at[k + 1];
    const int64_t rev_tiles = (in_total + kRevTile - 1) / kRevTile;
    if (ent_total >= (1ll << 32)) return mg_fail(ctx, MG_ERR_CAPACITY, "too many entries for one backward pass");
    for (int l = ra.l0; l <= k; ++l)
        if (d->h_hdr.rows_total[l] > kGradMaxRows) return mg_fail(ctx, MG_ERR_CAPACITY, "too many rows for one backward pass");
    if (ctx->bw_g_elems < g_total && (rc = mg_ensure(ctx, &ctx->bw_g, &ctx->bw_g_elems, g_total + g_total / 4 + 16))) return rc;
    if (ctx->bw_x_elems < (size_t)max_x && (rc = mg_ensure(ctx, &ctx->bw_x, &ctx->bw_x_elems, (size_t)max_x + 16))) return rc;
    if (ctx->bw_dx_elems < (size_t)max_dx && (rc = mg_ensure(ctx, &ctx->bw_dx, &ctx->bw_dx_elems, (size_t)max_dx + 16))) return rc;
    // one block.  Cleared by one memset: the scan's ticket, the unit counts, whether it gave up, its states, the counts; then the entries'
    // places, then the lists and units
    const size_t cnt_at = ((MG_MAX_HOPS + 4) + 2 * (size_t)rev_tiles + 3) / 4 * 4;
    const size_t cleared = cnt_at + (size_t)in_total + 1;
    const size_t rev_at = (cleared + (size_t)ent_total + 1) / 2 * 2;
    const size_t need_lists = rev_at + 2 * ((size_t)ent_total + (size_t)ra.unit_at[k + 1]);
    if (ctx->bw_lists_elems < need_lists && (rc = mg_ensure(ctx, &ctx->bw_lists, &ctx->bw_lists_elems, need_lists + need_lists / 4 + 16))) return rc;
    const RowGeom geom{B, k, d->rowbase, d->cum, d->node_off};
    const bool half = ctx->feat_dtype == MG_DTYPE_F16;
    const int grid = mg_grid(ctx, 8);
    if (!ctx->meta_left) {   // (the forward pass was in fp32, or of few rows that its layers looked up themselves)
        int64_t meta_at[MG_MAX_HOPS + 2] = {0};
        if ((rc = row_metadata(ctx, d, meta_at))) return rc;
    }
    // (behind the last layer's products: the scan clears rows of the inputs' gradients, and d_h0_dev may lie where d_out_dev does)
    auto turn_entries_round = [&]() -> int {
        ra.g = geom;
        ra.meta = ctx->ws_meta + (ra.l0 > 1 ? (int64_t)d->h_hdr.rows_total[1] : 0);
        ra.ent_repr = d->ent_repr; ra.sum_aggr = m->sum_aggr ? 1 : 0;
        ra.ticket = ctx->bw_lists;
        ra.n_units = ra.ticket + 1;
        static_assert(MG_MAX_HOPS % 2 == 0, "the states are 8-byte aligned behind the counters");
        ra.state = reinterpret_cast<uint64_t*>(ctx->bw_lists + MG_MAX_HOPS + 4);
        ra.cnt = ctx->bw_lists + cnt_at;
        ra.pos = ra.cnt + in_total + 1;
        ra.rev = reinterpret_cast<int2*>(ctx->bw_lists + rev_at);
        ra.units = ra.rev + ent_total;
        ra.bad = ra.n_units + MG_MAX_HOPS + 1;
        const char* polls = getenv("MG_REV_POLLS");
        ra.polls = polls ? atoi(polls) : kChainPolls;
        ra.status = ctx->d_flags;
        for (int l = ra.l0; l <= k; ++l) { ra.g_in[l] = l > 1 ? ctx->bw_g + g_off[l - 1] : d_h0_dev; ra.d_in[l] = m->dims[l - 1]; }
        MG_CUDA(ctx, cudaMemsetAsync(ctx->bw_lists, 0, sizeof(uint32_t) * cleared, st));
        ra.rows_per_warp = 4;
        while (ra.rows_per_warp < 32 && ra.out_at[k + 1] > (int64_t)ra.rows_per_warp * grid * (kThreads / 32)) ra.rows_per_warp *= 2;
        const int64_t per_block = (int64_t)ra.rows_per_warp * (kThreads / 32);
        const int rgrid = (int)std::min<int64_t>(grid, (ra.out_at[k + 1] + per_block - 1) / per_block);
        k_rev_entries<false><<<rgrid, kThreads, 0, st>>>(ra);
        k_rev_scan<<<(unsigned)rev_tiles, kThreads, 0, st>>>(ra);
        k_rev_entries<true><<<rgrid, kThreads, 0, st>>>(ra);
        ctx->launches += 3;
        return MG_OK;
    };
    bool turned = false;
    for (int l = k; l >= 1; --l) {
        const int d_in = m->dims[l - 1], d_out = m->dims[l];
        const int64_t M = d->h_hdr.rows_total[l];
        // dPre of the last layer is the caller's gradient; below it, the gather of the layer above has already gone through
        // the ReLU and summed the bias gradient
        const float* dpre_all = l == k ? d_out_dev : ctx->bw_g + g_off[l];
        if (l == k && M > 0) {
            // (few blocks: every one ends with an atomic add per column; 8,000 x 256 in 1,184 blocks took 13 us, in 148 6.5 us)
            const int blocks = (int)std::min<int64_t>(ctx->n_sms, (M + kThreads / (d_out / 4) - 1) / (kThreads / (d_out / 4)));
            k_grad_bias<<<blocks, kThreads, 0, st>>>(d_out_dev, m->g_bias[l - 1], M, d_out);
            ctx->launches++;
        }
        const float* h_prev = l > 1 ? ctx->ws_h[0] + h_off[l - 1] : nullptr;
        float* g_in = l > 1 ? ctx->bw_g + g_off[l - 1] : d_h0_dev;
        int64_t meta_at = 0;   // the layer's rows in ws_meta
        for (int q = 1; q < l; ++q) meta_at += d->h_hdr.rows_total[q];
        if (m->precision == MG_GEMM_TF32) {
            // dW += X^T dPre with X brought together inside the kernel; the row metadata is what mg_forward of this very model and sample left, or
            // was made above where its layers did without
            if ((rc = mg_layer_grad_weights(ctx, d, l, d_in, d_out, h_prev, dpre_all, ctx->ws_meta + meta_at, m->sum_aggr ? 1 : 0,
                                            ctx->agg_at[l] >= 0 && ctx->agg_sum == m->sum_aggr ? reinterpret_cast<const float*>(ctx->ws_saved + ctx->agg_at[l]) : nullptr,
                                            m->g_w_cat[l - 1]))) return rc;
            // dX = dPre W^T on the tensor cores: the K-major operand the kernel wants is W itself ([2 d_in, d_out])
            if (g_in && (rc = mg_gemm_tf32(ctx, dpre_all, m->w_cat[l - 1], m->zeros, ctx->bw_dx, M, 2 * d_in, d_out, false))) return rc;
        }
        const int64_t chunk = bw_mult * chunk_rows_for(d_in);
        for (int64_t r0 = 0; r0 < M && m->precision == MG_GEMM_FP32; r0 += chunk) {
            const int64_t r1 = std::min(M, r0 + chunk), rows = r1 - r0;
            AggArgs a;
            a.B = B; a.k = k; a.layer = l; a.d_in = d_in;
            a.row_lo = (int32_t)r0; a.row_hi = (int32_t)r1;
            a.rowbase_out = d->rowbase + (size_t)l * (B + 1);
            a.rowbase_in = d->rowbase + (size_t)(l - 1) * (B + 1);
            a.cum = d->cum; a.node_off = d->node_off; a.nodes = d->nodes;
            a.ent_off = d->ent_off; a.ent_nbrs = d->ent_nbrs; a.ent_repr = d->ent_repr;
            a.h_prev = h_prev;
            a.slots = ctx->slots; a.feat = mg_feat_geom(ctx); a.row_bytes = ctx->row_bytes;
            a.x = ctx->bw_x;
            a.round_tf32 = 0;
            a.sum_aggr = m->sum_aggr ? 1 : 0;
            if (l == 1) { if (half) launch_aggregate<true, true>(a, grid, st); else launch_aggregate<true, false>(a, grid, st); }
            else launch_aggregate<false, false>(a, grid, st);
            const float* dpre = dpre_all + r0 * d_out;
            const unsigned slices = (unsigned)((rows + kGradRowsPerBlock - 1) / kGradRowsPerBlock);
            dim3 gw((unsigned)((2 * d_in + 63) / 64), (unsigned)((d_out + 63) / 64), slices);
            k_grad_weights<<<gw, 256, 0, st>>>(ctx->bw_x, dpre, m->g_w_cat[l - 1], rows, 2 * d_in, d_out);
            ctx->launches += 2;
            if (!g_in) continue;   // layer 1 without a gradient of the base representations
            dim3 gx((unsigned)((rows + 63) / 64), (unsigned)((2 * d_in + 63) / 64));
            k_gemm_fp32<false><<<gx, 256, 0, st>>>(dpre, m->w_cat_t[l - 1], m->zeros, ctx->bw_dx + r0 * 2 * d_in, rows, 2 * d_in, d_out);
            ctx->launches++;
        }
        const int64_t rows_in = d->h_hdr.rows_total[l - 1];
        if (!g_in || rows_in == 0) continue;
        if (!turned && (rc = turn_entries_round())) return rc;
        turned = true;
        // dX -> the gradient of the layer's input rows
        const bool bits = l > 1 && ctx->positive_at[l - 1] >= 0;
        GatherArgs ga{geom, l, rows_in, ra.cnt + ra.in_at[l], ra.rev, ra.units + ra.unit_at[l], ra.n_units + l, ra.bad, ctx->bw_dx, d_in,
                      l > 1 ? ctx->ws_h[0] + h_off[l - 1] : nullptr, bits ? ctx->ws_saved + ctx->positive_at[l - 1] : nullptr, g_in, l > 1 ? m->g_bias[l - 2] : nullptr};
        // (groups of 16 rows, a warp per 128 columns; the units come on top, the loop takes what does not fit the grid)
        const int64_t warps = (rows_in + kGradRows - 1) / kGradRows * std::max(1, (d_in + 127) / 128);
        const int ggrid = (int)std::max<int64_t>(1, std::min<int64_t>(mg_grid(ctx, l > 1 ? 4 : 8), (warps + kThreads / 32 - 1) / (kThreads / 32) + 16));
        if (bits) k_grad_gather<RELU_BITS><<<ggrid, kThreads, 0, st>>>(ga);
        else if (l > 1) k_grad_gather<RELU_ROWS><<<ggrid, kThreads, 0, st>>>(ga);
        else k_grad_gather<RELU_NONE><<<ggrid, kThreads, 0, st>>>(ga);
        ctx->launches++;
    }
    if (ids_dev) launch_packed_ids(ctx, d, ids_dev);
    if (!ctx->ev_backward) MG_CUDA(ctx, cudaEventCreateWithFlags(&ctx->ev_backward, cudaEventDisableTiming));
    MG_CUDA(ctx, cudaGetLastError());
    MG_CUDA(ctx, cudaEventRecord(ctx->ev_backward, st));
    if (grads_dev) {
        cudaStream_t gs = (cudaStream_t)grads_stream;
        if (gs != st) MG_CUDA(ctx, cudaStreamWaitEvent(gs, ctx->ev_backward));
        MG_CUDA(ctx, cudaMemcpyAsync(grads_dev, m->g_block, m->g_elems * sizeof(float), cudaMemcpyDeviceToDevice, gs));
        if (gs != st) MG_CUDA(ctx, mg_reads_add(&m->g_reads, gs));
    }
    return MG_OK;
}

extern "C" int mg_backward_end(mg_ctx* ctx) {
    if (!ctx) return MG_ERR_ARG;
    if (!ctx->ev_backward) return mg_fail(ctx, MG_ERR_STATE, "mg_backward_begin has not run");
    MG_CUDA(ctx, cudaSetDevice(ctx->device));
    MG_CUDA(ctx, cudaEventSynchronize(ctx->ev_backward));
    return mg_gemm_tf32_status(ctx);
}

extern "C" int mg_backward(mg_ctx* ctx, mg_model* m, mg_dense* d, const float* d_out_dev, float* d_h0_dev) {
    if (int rc = mg_backward_begin(ctx, m, d, d_out_dev, d_h0_dev, nullptr, nullptr, nullptr)) return rc;
    return mg_backward_end(ctx);
}

extern "C" int mg_model_grads(const mg_model* m, int32_t layer, const float** d_w_self, const float** d_w_nbr, const float** d_bias) {
    if (!m) return MG_ERR_ARG;
    if (layer < 1 || layer > m->k) return mg_fail(m->ctx, MG_ERR_ARG, "layer must be in [1, k]");
    if (!m->g_w_cat[layer - 1]) return mg_fail(m->ctx, MG_ERR_STATE, "mg_backward has not run");
    const size_t half_elems = (size_t)m->dims[layer - 1] * m->dims[layer];
    if (d_w_self) *d_w_self = m->g_w_cat[layer - 1];
    if (d_w_nbr) *d_w_nbr = m->g_w_cat[layer - 1] + half_elems;
    if (d_bias) *d_bias = m->g_bias[layer - 1];
    return MG_OK;
}

static int optimizer_checks(mg_ctx* ctx, const mg_model* m) {
    if (!m || m->ctx != ctx) return mg_fail(ctx, MG_ERR_ARG, "bad model handle");
    if (!m->g_block) return mg_fail(ctx, MG_ERR_STATE, "mg_backward has not run");
    return MG_OK;
}

extern "C" int mg_model_adagrad_step(mg_ctx* ctx, mg_model* m, float lr, float eps) {
    if (!ctx) return MG_ERR_ARG;
    if (int rc = optimizer_checks(ctx, m)) return rc;
    if (!(eps > 0.f)) return mg_fail(ctx, MG_ERR_ARG, "eps must be positive");
    MG_CUDA(ctx, cudaSetDevice(ctx->device));
    if (!m->s_block) {   // accumulated squared gradients start at zero
        if (mg_malloc(ctx, (void**)&m->s_block, m->g_elems * sizeof(float)) != cudaSuccess) {
            cudaGetLastError();
            m->s_block = nullptr;
            return mg_fail(ctx, MG_ERR_OOM, "optimizer state allocation failed");
        }
        MG_CUDA(ctx, cudaMemsetAsync(m->s_block, 0, m->g_elems * sizeof(float), ctx->stream));
    }
    launch_weights<W_ADAGRAD>(ctx, m, lr, eps);
    MG_CUDA(ctx, cudaGetLastError());
    MG_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
    return MG_OK;
}

extern "C" int mg_model_sgd_step(mg_ctx* ctx, mg_model* m, float lr) {
    if (!ctx) return MG_ERR_ARG;
    if (int rc = optimizer_checks(ctx, m)) return rc;
    MG_CUDA(ctx, cudaSetDevice(ctx->device));
    launch_weights<W_SGD>(ctx, m, lr, 0.f);
    MG_CUDA(ctx, cudaGetLastError());
    MG_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
    return MG_OK;
}

namespace {

struct EmbSgdArgs {
    RowGeom g;
    const int32_t* nodes;
    const float* grad;          // [n_rows, dim] packed like H^0
    int64_t n_rows;
    char* slots;
    FeatGeom feat;
    int64_t row_bytes;
    int32_t dim;
    float lr;
};

// base representation of node(row) -= lr * grad[row]; a node of several mini-batches receives several updates.  Bound by
// the gradient rows coming in and the reductions in L2: a warp looks `group` consecutive rows up at once (lane = row: a
// binary search and two look-ups per row otherwise stood between any two rows), then reads four rows ahead of their
// 16-byte reductions (1.56M rows x 128 onto 2M nodes: 538 -> 294 us against a row and 4-byte reductions at a time).
// (A borrowed table or the caller's gradient rows may start anywhere: then 4 bytes at a time.)
__global__ void __launch_bounds__(kThreads) k_embedding_sgd(EmbSgdArgs a, int group, bool grad_aligned, bool table_aligned) {
    const int lane = threadIdx.x & 31;
    const int n4 = a.dim / 4;
    const int64_t warps = (int64_t)gridDim.x * (kThreads / 32);
    for (int64_t s0 = (blockIdx.x * (int64_t)(kThreads / 32) + (threadIdx.x >> 5)) * group; s0 < a.n_rows; s0 += warps * group) {
        const int n = (int)min((int64_t)group, a.n_rows - s0);
        int64_t at = 0;
        if (lane < n) {
            int32_t b, local, node;
            locate_row(a.g, 0, s0 + lane, &b, &local, &node);
            at = feat_row(a.feat, a.nodes[node]);
        }
        for (int c = lane; c - lane < n4; c += 32)
            for (int r = 0; r < n; r += 4) {
                float4 v[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    v[u] = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (r + u >= n || c >= n4) continue;
                    const float* g = a.grad + (s0 + r + u) * a.dim + 4 * c;
                    v[u] = grad_aligned ? __ldcs(reinterpret_cast<const float4*>(g)) : make_float4(g[0], g[1], g[2], g[3]);
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int64_t row = __shfl_sync(0xFFFFFFFFu, at, min(r + u, 31));
                    if (v[u].x == 0.f && v[u].y == 0.f && v[u].z == 0.f && v[u].w == 0.f) continue;
                    const float4 step = make_float4(-a.lr * v[u].x, -a.lr * v[u].y, -a.lr * v[u].z, -a.lr * v[u].w);
                    float* dst = reinterpret_cast<float*>(a.slots + row * a.row_bytes) + 4 * c;
                    if (table_aligned) atomicAdd(reinterpret_cast<float4*>(dst), step);
                    else { atomicAdd(dst, step.x); atomicAdd(dst + 1, step.y); atomicAdd(dst + 2, step.z); atomicAdd(dst + 3, step.w); }
                }
            }
    }
}

}  // namespace

extern "C" int mg_apply_embedding_sgd(mg_ctx* ctx, mg_dense* d, const float* d_h0_dev, float lr) {
    if (!ctx) return MG_ERR_ARG;
    if (!d || !d_h0_dev) return mg_fail(ctx, MG_ERR_ARG, "null argument");
    if (d->pending) return mg_fail(ctx, MG_ERR_STATE, "a sample is in flight on this mg_dense: call mg_sample_many_end first");
    if (!d->valid) return mg_fail(ctx, MG_ERR_STATE, "mg_dense holds no completed sample");
    if (d->ctx != ctx) return mg_fail(ctx, MG_ERR_ARG, "handle belongs to another context");
    if (!ctx->slots || ctx->feat_dim <= 0) return mg_fail(ctx, MG_ERR_STATE, "no feature table loaded");
    if (ctx->feat_dtype != MG_DTYPE_F32) return mg_fail(ctx, MG_ERR_ARG, "base representations are updated in fp32 tables only");
    if (int rs = mg_check_sample_residency(ctx, d)) return rs;
    MG_CUDA(ctx, cudaSetDevice(ctx->device));
    EmbSgdArgs a{{d->n_batches, d->k, d->rowbase, d->cum, d->node_off}, d->nodes, d_h0_dev, d->h_hdr.rows_total[0], ctx->slots,
                 mg_feat_geom(ctx), ctx->row_bytes, ctx->feat_dim, lr};
    if (a.n_rows > 0) {
        int group = 4;   // rows a warp looks up at once: fewer where there would not be a group for every warp of the grid
        while (group < 32 && a.n_rows > (int64_t)group * mg_grid(ctx, 8) * (kThreads / 32)) group *= 2;
        const int64_t groups = (a.n_rows + group - 1) / group;
        const int blocks = (int)std::min<int64_t>(mg_grid(ctx, 8), (groups + kThreads / 32 - 1) / (kThreads / 32));
        k_embedding_sgd<<<blocks, kThreads, 0, ctx->stream>>>(a, group, reinterpret_cast<uintptr_t>(d_h0_dev) % 16 == 0,
                                                              reinterpret_cast<uintptr_t>(ctx->slots) % 16 == 0);
        ctx->launches++;
    }
    // with host backing the updated slots go back to the host table when their partitions are evicted
    ctx->dirty_part.assign(ctx->n_parts, 0);
    for (int p = 0; p < ctx->n_parts; ++p) ctx->dirty_part[p] = ctx->slot_of_part[p] >= 0 ? 1 : 0;
    MG_CUDA(ctx, cudaGetLastError());
    MG_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
    return MG_OK;
}

extern "C" int mg_dense_packed_ids(mg_ctx* ctx, mg_dense* d, int32_t* ids_dev) {
    if (!ctx) return MG_ERR_ARG;
    if (!d || !ids_dev) return mg_fail(ctx, MG_ERR_ARG, "null argument");
    if (d->pending) return mg_fail(ctx, MG_ERR_STATE, "a sample is in flight on this mg_dense: call mg_sample_many_end first");
    if (!d->valid) return mg_fail(ctx, MG_ERR_STATE, "mg_dense holds no completed sample");
    MG_CUDA(ctx, cudaSetDevice(ctx->device));
    launch_packed_ids(ctx, d, ids_dev);
    MG_CUDA(ctx, cudaGetLastError());
    MG_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
    return MG_OK;
}

// ---------------------------------------------------------------------------------------
// Forward pass that allocates nothing (the paper has no counterpart).
//
// All temporaries live in one file-scope device array that every GPU loading this library
// holds until the process exits:
//   [0, kNoAllocStagingBytes)                     the [self | mean] staging rows of one chunk
//   [kNoAllocStagingBytes, MG_NOALLOC_SCRATCH_BYTES)  the intermediate layer outputs H^1 .. H^{k-1}
// Nothing in it has to start at zero: every element a kernel reads was written earlier in the
// same call (rows past the end of a tile are zero-filled by the TMA load, not read from here).
// ---------------------------------------------------------------------------------------
static __device__ __align__(256) unsigned char g_noalloc_scratch[MG_NOALLOC_SCRATCH_BYTES];

namespace {
constexpr size_t kNoAllocStagingBytes = 4u << 20;
constexpr int kNoAllocMaxDevices = 64;
unsigned char* g_noalloc_ptr[kNoAllocMaxDevices] = {nullptr};
}  // namespace

extern "C" int mg_forward_noalloc(mg_ctx* ctx, const mg_model* m, mg_dense* d, float* out_dev) {
    if (!ctx) return MG_ERR_ARG;
    int rc = forward_checks(ctx, m, d);
    if (rc) return rc;
    if (!out_dev) return mg_fail(ctx, MG_ERR_ARG, "null output");
    if (ctx->device < 0 || ctx->device >= kNoAllocMaxDevices) return mg_fail(ctx, MG_ERR_ARG, "device ordinal above %d", kNoAllocMaxDevices - 1);
    MG_CUDA(ctx, cudaSetDevice(ctx->device));
    // once per device, with that device current: the array's name is only a host-side handle, the
    // kernels need its device address
    if (!g_noalloc_ptr[ctx->device]) {
        unsigned char* p = nullptr;
        const cudaError_t e = cudaGetSymbolAddress((void**)&p, g_noalloc_scratch);
        if (e != cudaSuccess || !p) return mg_cuda_fail(ctx, e, "cudaGetSymbolAddress(g_noalloc_scratch)");
        g_noalloc_ptr[ctx->device] = p;
    }
    unsigned char* scratch = g_noalloc_ptr[ctx->device];
    const int k = d->k, B = d->n_batches;
    cudaStream_t st = ctx->stream;

    // intermediates H^1 .. H^{k-1} must fit behind the staging area
    size_t off[MG_MAX_HOPS + 1] = {0};
    size_t inter_floats = 0;
    for (int l = 1; l < k; ++l) {
        off[l] = inter_floats;
        inter_floats += (size_t)d->h_hdr.rows_total[l] * m->dims[l];
    }
    const size_t inter_cap = (MG_NOALLOC_SCRATCH_BYTES - kNoAllocStagingBytes) / sizeof(float);
    if (inter_floats > inter_cap)
        return mg_fail(ctx, MG_ERR_CAPACITY,
                       "mg_forward_noalloc: intermediate layer outputs need %zu bytes, the built-in scratch holds %zu "
                       "(MG_NOALLOC_SCRATCH_BYTES = %u in total); use mg_forward or fewer mini-batches per call",
                       inter_floats * sizeof(float), inter_cap * sizeof(float), (unsigned)MG_NOALLOC_SCRATCH_BYTES);
    float* staging = reinterpret_cast<float*>(scratch);
    float* inter = reinterpret_cast<float*>(scratch + kNoAllocStagingBytes);

    const bool half = ctx->feat_dtype == MG_DTYPE_F16;
    for (int l = 1; l <= k; ++l) {
        const int d_in = m->dims[l - 1], d_out = m->dims[l];
        const int64_t M = d->h_hdr.rows_total[l];
        float* h_out = l == k ? out_dev : inter + off[l];
        const float* h_prev = l > 1 ? inter + off[l - 1] : nullptr;
        int64_t chunk = (int64_t)(kNoAllocStagingBytes / sizeof(float)) / (2 * d_in);
        chunk = chunk / 128 * 128;
        if (chunk < 128) return mg_fail(ctx, MG_ERR_CAPACITY, "mg_forward_noalloc: layer width %d too large for the staging area", d_in);
        for (int64_t r0 = 0; r0 < M; r0 += chunk) {
            const int64_t r1 = std::min(M, r0 + chunk);
            AggArgs a;
            a.B = B; a.k = k; a.layer = l; a.d_in = d_in;
            a.row_lo = (int32_t)r0; a.row_hi = (int32_t)r1;
            a.rowbase_out = d->rowbase + (size_t)l * (B + 1);
            a.rowbase_in = d->rowbase + (size_t)(l - 1) * (B + 1);
            a.cum = d->cum; a.node_off = d->node_off; a.nodes = d->nodes;
            a.ent_off = d->ent_off; a.ent_nbrs = d->ent_nbrs; a.ent_repr = d->ent_repr;
            a.h_prev = h_prev;
            a.slots = ctx->slots; a.feat = mg_feat_geom(ctx); a.row_bytes = ctx->row_bytes;
            a.x = staging;
            a.round_tf32 = m->precision == MG_GEMM_TF32;
            a.sum_aggr = m->sum_aggr ? 1 : 0;
            const int grid = mg_grid(ctx, 8);
            if (l == 1) { if (half) launch_aggregate<true, true>(a, grid, st); else launch_aggregate<true, false>(a, grid, st); }
            else launch_aggregate<false, false>(a, grid, st);
            ctx->launches++;
            const int64_t rows = r1 - r0;
            const bool relu = l < k;
            if (m->precision == MG_GEMM_FP32) {
                dim3 g2((unsigned)((rows + 63) / 64), (unsigned)((d_out + 63) / 64));
                if (relu) k_gemm_fp32<true><<<g2, 256, 0, st>>>(staging, m->w_cat[l - 1], m->bias[l - 1], h_out + r0 * d_out, rows, d_out, 2 * d_in);
                else k_gemm_fp32<false><<<g2, 256, 0, st>>>(staging, m->w_cat[l - 1], m->bias[l - 1], h_out + r0 * d_out, rows, d_out, 2 * d_in);
                ctx->launches++;
            } else {
                rc = mg_gemm_tf32(ctx, staging, m->w_cat_t[l - 1], m->bias[l - 1], h_out + r0 * d_out, rows, d_out, 2 * d_in, relu);
                if (rc) return rc;
            }
        }
    }
    MG_CUDA(ctx, cudaGetLastError());
    MG_CUDA(ctx, cudaStreamSynchronize(st));
    if (m->precision == MG_GEMM_TF32) return mg_gemm_tf32_status(ctx);
    return MG_OK;
}

extern "C" int mg_keep_layer_outputs(mg_ctx* ctx, int enable) {
    if (!ctx) return MG_ERR_ARG;
    ctx->keep_layers = enable != 0;
    return MG_OK;
}

extern "C" int mg_set_layer_window(mg_ctx* ctx, int32_t mini_batches) {
    if (!ctx) return MG_ERR_ARG;
    if (mini_batches < 0) return mg_fail(ctx, MG_ERR_ARG, "negative window");
    ctx->layer_window_batches = mini_batches;
    return MG_OK;
}
