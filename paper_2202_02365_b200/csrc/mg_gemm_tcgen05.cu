// TF32 tensor-core GEMM for the GraphSage linear layers on sm_100a:
//     out[M, N] = act(x[M, K] . w_t[N, K]^T + bias)
// x is the [self | mean] staging matrix (K-major), w_t the K-major copy of [W_self; W_nbr].
// Both operands are already rounded to the nearest TF32 value by their producers.
//
// One CTA computes a 128 x BN tile (BN = N rounded up to 16, at most 256; wider outputs use
// several N tiles).  A producer thread streams 32-float K slices of both operands into a ring
// of 128-byte-swizzled shared-memory stages with TMA (no multicast); one thread issues
// tcgen05.mma kind::tf32 with the fp32 accumulator in tensor memory; four epilogue warps read
// the accumulator with tcgen05.ld, add the bias, apply ReLU and store.  Two CTAs fit on an SM,
// so one tile's epilogue overlaps the other's main loop.  Every mbarrier wait is bounded: on a
// time-out the kernel records an error code, still frees its tensor memory and returns.

#include <cuda.h>

#include <algorithm>

#include "mg_internal.cuh"
#include "mg_tcgen05.cuh"

namespace {

constexpr int BM = 128;
constexpr int BK = 32;                       // floats per stage row = 128 bytes = one swizzle row
constexpr int kGemmThreads = 192;            // warp 0 TMA, warp 1 MMA + TMEM, warps 2..5 epilogue

using namespace tc;

struct GemmParams {
    float* out;
    const float* bias;
    int64_t M;
    int32_t N, K, BN, stages, tmem_cols, relu;
    uint32_t* error;  // 0 = ok, else the role that gave up waiting
};

__global__ void __launch_bounds__(kGemmThreads)
k_gemm_tf32(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b, GemmParams p) {
    extern __shared__ uint8_t smem_raw[];
    __shared__ uint64_t full_bar[8], empty_bar[8], acc_bar;
    __shared__ uint32_t tmem_slot;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t m0 = (int64_t)blockIdx.x * BM;
    const int n0 = blockIdx.y * p.BN;
    const int kt_total = (p.K + BK - 1) / BK;   // K steps
    const uint32_t a_bytes = BM * BK * 4, b_bytes = (uint32_t)p.BN * BK * 4;
    uint8_t* stage_base = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    const uint32_t stage_bytes = a_bytes + b_bytes;  // both multiples of 1024

    if (threadIdx.x == 0) {
        for (int s = 0; s < p.stages; ++s) { mbar_init(&full_bar[s], 1); mbar_init(&empty_bar[s], 1); }
        mbar_init(&acc_bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(&map_a) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(&map_b) : "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)), "r"((uint32_t)p.tmem_cols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = tmem_slot;

    if (warp == 0) {
        if (lane == 0) {
            for (int kt = 0; kt < kt_total; ++kt) {
                const int s = kt % p.stages;
                if (kt >= p.stages && !mbar_wait(&empty_bar[s], ((kt / p.stages) - 1) & 1)) { report(p.error, 1u); break; }
                uint8_t* sa = stage_base + (size_t)s * stage_bytes;
                mbar_expect_tx(&full_bar[s], stage_bytes);
                tma_load_2d(sa, &map_a, &full_bar[s], kt * BK, (int)m0);
                tma_load_2d(sa + a_bytes, &map_b, &full_bar[s], kt * BK, n0);
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        if (lane == 0) {
            // instruction descriptor: fp32 accumulator, TF32 x TF32, both K-major, M = 128, N = BN
            const uint32_t idesc = (1u << 4) | (2u << 7) | (2u << 10) | ((uint32_t)(p.BN >> 3) << 17) | ((uint32_t)(BM >> 4) << 24);
            bool ok = true;
            for (int kt = 0; kt < kt_total && ok; ++kt) {
                const int s = kt % p.stages;
                if (!mbar_wait(&full_bar[s], (kt / p.stages) & 1)) { report(p.error, 2u); ok = false; break; }
                tc_fence_after();
                const uint32_t sa = smem_u32(stage_base + (size_t)s * stage_bytes);
                const uint64_t da = smem_desc_sw128(sa), db = smem_desc_sw128(sa + a_bytes);
#pragma unroll
                for (int kk = 0; kk < BK / 8; ++kk)   // one instruction consumes 8 TF32 values (32 bytes) of K
                    mma_tf32(tmem_base, da + (uint64_t)(kk * 2), db + (uint64_t)(kk * 2), idesc, (kt | kk) ? 1u : 0u);
                mma_commit(&empty_bar[s]);   // the stage may be refilled once these MMAs have read it
            }
            mma_commit(&acc_bar);            // accumulator complete (arrives even after a time-out)
        }
        __syncwarp();
    } else {
        const bool ok = mbar_wait(&acc_bar, 0);
        if (!ok && lane == 0) report(p.error, 3u);
        tc_fence_after();
        const int lane_group = warp & 3;                 // tensor-memory lanes this warp may read
        const int64_t row0 = m0 + lane_group * 32;
        // the operand ring is idle once the accumulator is complete: its first 17 KiB serve as the four
        // warps' transpose buffers for coalesced stores
        float* out_stage = reinterpret_cast<float*>(stage_base);
        if (ok) {
            for (int c0 = 0; c0 < p.BN; c0 += 32) {
                uint32_t v[32];
                tmem_ld_32(tmem_base + ((uint32_t)(lane_group * 32) << 16) + (uint32_t)c0, v);
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                if (row0 >= p.M) continue;
                store_slice_coalesced(v, out_stage + lane_group * (32 * 33), p.bias, p.out, row0, p.M, p.N, n0 + c0, p.relu != 0);
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"((uint32_t)p.tmem_cols) : "memory");
    }
}

// The same product for K up to 256: persistent CTA pairs keep their columns' weights in shared memory and stream rows.
//
// Bound by DRAM (rows in, rows out).  The kernel above loads the weights anew for every 128 rows -- 256 KB of weights for 128 KB of rows at
// K = N = 256 --, has two ring stages beside them, and a CTA stores only once it has loaded.  Here a pair owns up to 256 output columns
// (each CTA holds the weights of half of them, cta_group::2) and every n-th block of 256 rows, 128 per CTA, so rows come in once for 256
// columns.  K slices of rows come through a ring of four, and two accumulators in tensor memory let the stores (TMA, through two 32 x 32
// tiles per warp) of one block run under the products of the next.  543k rows (K = N = 256) and 92k rows (K = 256, N = 512): 334 -> 271 us.
// (Single CTAs with 128 columns each, rows read once per CTA: 311 us.)
constexpr int kWideStages = 4, kWideMaxK = 256, kWideCols = 256;

struct WideParams {
    const float* bias;
    int64_t M;
    int32_t N, BN, kt, n_tiles, tmem_cols, relu;   // kt: K slices of 32; n_tiles: column blocks
    uint32_t* error;
};

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kGemmThreads)
k_gemm_tf32_rows(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b, const __grid_constant__ CUtensorMap map_out,
                 WideParams p) {
    extern __shared__ uint8_t smem_raw[];
    __shared__ uint64_t b_full[kWideMaxK / BK], a_full[kWideStages], a_empty[kWideStages], acc_full[2], acc_empty[2];
    __shared__ uint32_t tmem_slot;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = cluster_ctarank(), pair = blockIdx.x >> 1;   // rank 0, the leader, issues the MMAs
    const bool leader = rank == 0;
    const int n0 = (int)(pair % p.n_tiles) * p.BN, half_n = p.BN / 2;
    const int64_t first = pair / p.n_tiles, step = (gridDim.x >> 1) / p.n_tiles;   // (a multiple of n_tiles pairs)
    const int64_t m_tiles = (p.M + 2 * BM - 1) / (2 * BM);
    auto row_of = [&](uint32_t it) -> int64_t { return (first + (int64_t)it * step) * (2 * BM) + rank * BM; };   // (past the end: read as zeros, not stored)
    const uint32_t my = first < m_tiles ? (uint32_t)((m_tiles - first + step - 1) / step) : 0u;
    constexpr uint32_t a_bytes = BM * BK * 4;
    const uint32_t b_bytes = (uint32_t)half_n * BK * 4;   // (both multiples of 1024)
    uint8_t* out_base = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint8_t* a_base = out_base + 4 * 2 * 4096;
    uint8_t* b_base = a_base + kWideStages * a_bytes;
    if (threadIdx.x == 0) {
        for (int s = 0; s < kWideMaxK / BK; ++s) mbar_init(&b_full[s], 1);
        for (int s = 0; s < kWideStages; ++s) { mbar_init(&a_full[s], 1); mbar_init(&a_empty[s], 1); }
        for (int s = 0; s < 2; ++s) { mbar_init(&acc_full[s], 1); mbar_init(&acc_empty[s], 2 * 4); }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(&map_a) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(&map_b) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(&map_out) : "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)), "r"((uint32_t)p.tmem_cols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    cluster_sync_all();   // barriers of both CTAs are initialised before anyone arrives on a remote one
    tc_fence_after();
    const uint32_t tmem_base = tmem_slot, acc_cols = (uint32_t)p.tmem_cols / 2;

    if (warp == 0) {
        if (lane == 0) {
            uint32_t cnt = 0, b_loaded = 0;
            bool ok = true;
            for (uint32_t it = 0; it < my && ok; ++it)
                for (int kt = 0; kt < p.kt; ++kt, ++cnt) {
                    const int s = cnt % kWideStages;
                    if (it == 0) {
                        if (leader) mbar_expect_tx(&b_full[kt], 2 * b_bytes);   // (both CTAs' bytes are counted on the leader's barriers)
                        tma_load_2d_pair(b_base + (size_t)kt * b_bytes, &map_b, mapa_u32(smem_u32(&b_full[kt]), 0), kt * BK, n0 + (int)rank * half_n);
                        ++b_loaded;
                    }
                    if (cnt >= (uint32_t)kWideStages && !mbar_wait(&a_empty[s], ((cnt / kWideStages) - 1) & 1)) { report(p.error, 1u); ok = false; break; }
                    if (leader) mbar_expect_tx(&a_full[s], 2 * a_bytes);
                    tma_load_2d_pair(a_base + (size_t)s * a_bytes, &map_a, mapa_u32(smem_u32(&a_full[s]), 0), kt * BK, (int)row_of(it));
                }
            // nothing of the pair's may be in flight when it ends
            for (uint32_t i = 0; leader && i < b_loaded; ++i) if (!mbar_wait(&b_full[i], 0)) report(p.error, 4u);
            for (uint32_t i = cnt >= (uint32_t)kWideStages ? cnt - kWideStages : 0; leader && i < cnt; ++i)
                if (!mbar_wait(&a_full[i % kWideStages], (i / kWideStages) & 1)) report(p.error, 4u);
        }
        __syncwarp();
    } else if (warp == 1) {
        if (lane == 0 && leader) {
            const uint32_t idesc = (1u << 4) | (2u << 7) | (2u << 10) | ((uint32_t)(p.BN >> 3) << 17) | ((uint32_t)(2 * BM >> 4) << 24);
            uint32_t cnt = 0;
            bool ok = true;
            for (uint32_t it = 0; it < my && ok; ++it) {
                const uint32_t buf = it & 1, d_tmem = tmem_base + buf * acc_cols;
                if (it >= 2 && !mbar_wait(&acc_empty[buf], ((it >> 1) - 1) & 1)) { report(p.error, 5u); break; }
                tc_fence_after();
                for (int kt = 0; kt < p.kt; ++kt, ++cnt) {
                    const int s = cnt % kWideStages;
                    if ((it == 0 && !mbar_wait(&b_full[kt], 0)) || !mbar_wait(&a_full[s], (cnt / kWideStages) & 1)) { report(p.error, 2u); ok = false; break; }
                    tc_fence_after();
                    const uint64_t da = smem_desc_sw128(smem_u32(a_base + (size_t)s * a_bytes)), db = smem_desc_sw128(smem_u32(b_base + (size_t)kt * b_bytes));
#pragma unroll
                    for (int kk = 0; kk < BK / 8; ++kk)
                        mma_tf32_pair(d_tmem, da + (uint64_t)(kk * 2), db + (uint64_t)(kk * 2), idesc, (kt | kk) ? 1u : 0u);
                    mma_commit_pair(&a_empty[s]);
                }
                if (ok) mma_commit_pair(&acc_full[buf]);
            }
        }
        __syncwarp();
    } else {
        const int quarter = warp & 3;   // tensor-memory lanes this warp may read
        uint8_t* stage = out_base + quarter * 2 * 4096;
        uint32_t boxes = 0;
        bool ok = true;
        for (uint32_t it = 0; it < my && ok; ++it) {
            const uint32_t buf = it & 1;
            if (!mbar_wait(&acc_full[buf], (it >> 1) & 1)) { if (lane == 0) report(p.error, 3u); ok = false; }
            ok = __all_sync(0xFFFFFFFFu, ok);
            if (!ok) break;
            tc_fence_after();
            const int64_t row0 = row_of(it) + quarter * 32;
            for (int c0 = 0; c0 < p.BN; c0 += 32) {
                uint32_t v[32];
                tmem_ld_32(tmem_base + buf * acc_cols + ((uint32_t)(quarter * 32) << 16) + (uint32_t)c0, v);
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                if (row0 >= p.M || n0 + c0 >= p.N) continue;
                uint8_t* box = stage + (boxes++ & 1) * 4096;
                if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");   // the box before last has left the tile
                __syncwarp();
#pragma unroll
                for (int c = 0; c < 8; ++c) {   // lane = row of the box, 128-byte swizzle
                    const int n = n0 + c0 + 4 * c;
                    const float4 b = n < p.N ? __ldg(reinterpret_cast<const float4*>(p.bias + n)) : make_float4(0.f, 0.f, 0.f, 0.f);
                    float4 o = make_float4(__uint_as_float(v[4 * c]) + b.x, __uint_as_float(v[4 * c + 1]) + b.y, __uint_as_float(v[4 * c + 2]) + b.z,
                                           __uint_as_float(v[4 * c + 3]) + b.w);
                    if (p.relu) { o.x = fmaxf(o.x, 0.f); o.y = fmaxf(o.y, 0.f); o.z = fmaxf(o.z, 0.f); o.w = fmaxf(o.w, 0.f); }
                    *reinterpret_cast<float4*>(box + lane * 128 + ((c ^ (lane & 7)) << 4)) = o;
                }
                fence_async_smem();
                __syncwarp();
                if (lane == 0) {   // (rows past the end and columns past the width are clipped by the tensor map)
                    tma_store_2d(&map_out, box, n0 + c0, (int)row0);
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
        if (lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
        __syncwarp();
    }
    tc_fence_before();
    cluster_sync_all();   // neither CTA leaves (or frees tensor memory) while the other may still signal or read it
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"((uint32_t)p.tmem_cols) : "memory");
    }
}

}  // namespace

// the persistent form (M rows, K <= 256, out and bias 16-byte aligned)
static int gemm_rows(mg_ctx* ctx, const float* x, const float* w_t, const float* bias, float* out, int64_t M, int N, int K, bool relu) {
    WideParams p;
    p.bias = bias; p.M = M; p.N = N; p.relu = relu ? 1 : 0; p.error = ctx->d_flags;
    p.BN = std::min(kWideCols, (N + 31) / 32 * 32);
    p.kt = (K + BK - 1) / BK;
    p.n_tiles = (N + p.BN - 1) / p.BN;
    p.tmem_cols = 64;
    while (p.tmem_cols < 2 * p.BN) p.tmem_cols <<= 1;
    CUtensorMap ma, mb, mo;
    if (!make_map_f32(&ma, x, M, K, BM) || !make_map_f32(&mb, w_t, N, K, p.BN / 2) || !make_map_f32(&mo, out, M, N, 32))
        return mg_fail(ctx, MG_ERR_CUDA, "cuTensorMapEncodeTiled failed (M %lld N %d K %d)", (long long)M, N, K);
    const int fixed = 4 * 2 * 4096 + kWideStages * BM * BK * 4 + 1024;
    const int smem = fixed + p.kt * (p.BN / 2) * BK * 4;
    MG_CUDA(ctx, mg_smem_limit(ctx, (const void*)k_gemm_tf32_rows, fixed + kWideMaxK * (kWideCols / 2) * 4));
    const int64_t m_tiles = (M + 2 * BM - 1) / (2 * BM);
    const int64_t per = std::min<int64_t>(m_tiles, std::max(1, ctx->n_sms / 2 / p.n_tiles));
    k_gemm_tf32_rows<<<(unsigned)(2 * per * p.n_tiles), kGemmThreads, smem, ctx->stream>>>(ma, mb, mo, p);
    ctx->launches++;
    MG_CUDA(ctx, cudaGetLastError());
    return MG_OK;
}

int mg_gemm_tf32(mg_ctx* ctx, const float* x, const float* w_t, const float* bias, float* out, int64_t M, int N, int K, bool relu) {
    if (M <= 0) return MG_OK;
    if (K % 4 != 0 || N % 4 != 0) return mg_fail(ctx, MG_ERR_ARG, "GEMM sizes must be multiples of 4");
    // (longer rows' weights do not fit shared memory beside the ring; a caller's output may start anywhere; a pair with fewer than four
    // blocks of rows waits longer for its weights than it saves: 34k + 8k rows 46 -> 49 us, 10k rows of 100 columns 7.8 -> 9.3)
    const int64_t row_blocks = (M + 2 * BM - 1) / (2 * BM) * ((N + kWideCols - 1) / kWideCols);
    if (K <= kWideMaxK && row_blocks >= 4 * (ctx->n_sms / 2) && ((reinterpret_cast<uintptr_t>(out) | reinterpret_cast<uintptr_t>(bias)) & 15) == 0)
        return gemm_rows(ctx, x, w_t, bias, out, M, N, K, relu);
    GemmParams p;
    p.out = out; p.bias = bias; p.M = M; p.N = N; p.K = K; p.relu = relu ? 1 : 0; p.error = ctx->d_flags;
    p.BN = std::min(256, (N + 15) / 16 * 16);
    p.tmem_cols = 32;
    while (p.tmem_cols < p.BN) p.tmem_cols <<= 1;
    const int stage_bytes = BM * BK * 4 + p.BN * BK * 4;
    p.stages = std::max(1, std::min({(K + BK - 1) / BK, 8, (96 * 1024) / stage_bytes}));
    const size_t smem = (size_t)p.stages * stage_bytes + 1024;
    CUtensorMap ma, mb;
    if (!make_map_f32(&ma, x, M, K, BM) || !make_map_f32(&mb, w_t, N, K, p.BN))
        return mg_fail(ctx, MG_ERR_CUDA, "cuTensorMapEncodeTiled failed (M %lld N %d K %d)", (long long)M, N, K);
    MG_CUDA(ctx, mg_smem_limit(ctx, (const void*)k_gemm_tf32, 100 * 1024));
    dim3 grid((unsigned)((M + BM - 1) / BM), (unsigned)((N + p.BN - 1) / p.BN));
    k_gemm_tf32<<<grid, kGemmThreads, smem, ctx->stream>>>(ma, mb, p);
    ctx->launches++;
    MG_CUDA(ctx, cudaGetLastError());
    return MG_OK;
}

// After the stream has drained: MG_ERR_TIMEOUT if a kernel gave up waiting (the word is cleared).
int mg_gemm_tf32_status(mg_ctx* ctx) {
    const uint32_t flag = *static_cast<volatile uint32_t*>(ctx->h_flags);
    if (!flag) return MG_OK;
    *ctx->h_flags = 0;
    if (flag == MG_ROLE_REV_SCAN) return mg_fail(ctx, MG_ERR_TIMEOUT, "the scan of the backward pass's entry lists gave up waiting");
    return mg_fail(ctx, MG_ERR_TIMEOUT, "tensor-core GEMM gave up waiting on a barrier (role %u)", flag);
}
