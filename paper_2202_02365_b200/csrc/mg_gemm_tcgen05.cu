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

}  // namespace

int mg_gemm_tf32(mg_ctx* ctx, const float* x, const float* w_t, const float* bias, float* out, int64_t M, int N, int K, bool relu) {
    if (M <= 0) return MG_OK;
    if (K % 4 != 0 || N % 4 != 0) return mg_fail(ctx, MG_ERR_ARG, "GEMM sizes must be multiples of 4");
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
