// The weight gradients of the proposal network on the fifth-generation tensor
// cores, both in one launch:
//
//     dW1 += dZ1^T X   (128 x 384),     dW2 += dZ2^T H1   (128 x 128)
//
// with the batch as K.  The operands come transposed from the rows' kernel
// (dZ1T, dZ2T: [128][rows]; XT: [384][rows]; H1T: [128][rows]; BF16, K-major).
// A block of 128 threads takes one 128 x 64 tile of dW1 (six) or dW2 (two) and
// a part of the rows, so that the batch is split over about two blocks per SM.
// Thread 0 streams the rows in chunks of 64 through four stages: a chunk of A
// (128 x 128 bytes) and of B (64 x 128 bytes) is one TMA box each, with the
// 128-byte swizzle the MMA descriptors name.  Four tcgen05.mma (K = 16) per
// chunk go into one TMEM accumulator, whose FP32 tile the four warps then add
// into the gradient, four columns per reduction.  Rows past the batch are
// filled with zeros by the copies.  Every wait is bounded: a wait that gives up
// raises the caller's error flag and the block leaves without adding.
//
// Bound by latency (a block has four chunks of a batch of 8,192 rows).  As two
// GEMMs with boxes of 16-byte rows, after four transposes through memory, this
// took 63 us of a training step of 8,192 rows.
#include <cuda.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>

#include "gamma_internal.h"
#include "gamma_tc.cuh"

namespace gk {

using bf16 = __nv_bfloat16;

namespace {

constexpr int kGemmBM = 128;             // rows of a tile (MMA M: the output features)
constexpr int kGemmBN = 64;              // columns of a tile
constexpr int kGemmBK = 64;              // batch rows per stage
constexpr int kGemmStages = 4;           // stages in flight
constexpr int kTiles1 = kInPad / kGemmBN, kTiles2 = kH / kGemmBN;

struct __align__(1024) GemmSmem {
    bf16 A[kGemmStages][kGemmBM * kGemmBK];   // 128 rows x 128 bytes per stage (128-byte swizzle)
    bf16 B[kGemmStages][kGemmBN * kGemmBK];   // 64 rows x 128 bytes
    uint64_t full[kGemmStages], empty[kGemmStages], done;
    uint32_t tmem;
    int ok;
};

__device__ __forceinline__ void red_add4(float* p, float a, float b, float c, float d)
{
    asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(a), "f"(b), "f"(c), "f"(d)
                 : "memory");
}

__global__ void __launch_bounds__(128, 1)
    k_wgrad(const __grid_constant__ WgradMaps maps, int nchunks, int chunks_per_split, float* __restrict__ gW1,
            float* __restrict__ gW2, unsigned* flags)
{
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char* base = smem_raw + ((1024u - (smem_addr(smem_raw) & 1023u)) & 1023u);
    GemmSmem& S = *reinterpret_cast<GemmSmem*>(base);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const bool first = blockIdx.x < kTiles1;                  // a tile of dW1, else of dW2
    const int n0 = (first ? (int)blockIdx.x : (int)blockIdx.x - kTiles1) * kGemmBN;
    const int c0 = blockIdx.y * chunks_per_split;
    const int nloc = min(nchunks, c0 + chunks_per_split) - c0;
    if (nloc <= 0) return;                                    // block-uniform: an empty part
    if (tid == 0) {
        for (int b = 0; b < kGemmStages; ++b) {
            mbar_init(&S.full[b], 1);
            mbar_init(&S.empty[b], 1);
        }
        mbar_init(&S.done, 1);
        mbar_fence_init();
        S.ok = 1;
    }
    if (warp == 0) {
        tmem_alloc(&S.tmem, kGemmBN);
        tmem_relinquish();
    }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tm = S.tmem;
    if (tid == 0) {
        constexpr uint32_t kId = idesc_bf16_f32(kGemmBM, kGemmBN);
        constexpr uint32_t kBytes = (kGemmBM + kGemmBN) * kGemmBK * 2;
        const CUtensorMap* am = first ? &maps.dz1 : &maps.dz2;
        const CUtensorMap* bm = first ? &maps.x : &maps.h1;
        bool ok = true;
        int loaded = 0, used = 0;                             // chunks requested, chunks seen landed
        auto load = [&](int i) {
            const int s = i % kGemmStages;
            if (i >= kGemmStages) ok = mbar_wait_bounded(&S.empty[s], (i / kGemmStages - 1) & 1u);
            if (!ok) return;
            mbar_arrive_expect_tx(&S.full[s], kBytes);
            const int k0 = (c0 + i) * kGemmBK;
            tma_load_2d(S.A[s], am, k0, 0, &S.full[s]);
            tma_load_2d(S.B[s], bm, k0, n0, &S.full[s]);
            ++loaded;
        };
        for (int i = 0; i < kGemmStages - 1 && i < nloc && ok; ++i) load(i);
        for (int i = 0; i < nloc && ok; ++i) {
            if (i + kGemmStages - 1 < nloc) load(i + kGemmStages - 1);
            if (!ok) break;
            const int s = i % kGemmStages;
            ok = mbar_wait_bounded(&S.full[s], (i / kGemmStages) & 1u);
            if (!ok) break;
            ++used;
            tc_fence_after_sync();
            const uint32_t aa = smem_addr(S.A[s]), ba = smem_addr(S.B[s]);
#pragma unroll
            for (int kk = 0; kk < kGemmBK; kk += 16)
                tc_mma_bf16(tm, smem_desc_sw128(aa, kk * 2), smem_desc_sw128(ba, kk * 2), kId, (i | kk) != 0);
            tc_commit(&S.empty[s]);
        }
        tc_commit(&S.done);
        if (!ok) {
            S.ok = 0;
            // let this block's copies land before it leaves
            for (int i = used; i < loaded; ++i) mbar_wait_bounded(&S.full[i % kGemmStages], (i / kGemmStages) & 1u);
        }
    }
    // every thread waits for the accumulator (bounded), then the epilogue
    const bool landed = mbar_wait_bounded(&S.done, 0u);
    const bool ok = __syncthreads_and(landed) && S.ok;        // block-uniform
    tc_fence_after_sync();
    if (ok) {
        const int row = 32 * warp + lane;
        float* dst = first ? gW1 + (long long)row * kInPad + n0 : gW2 + (long long)row * kH + n0;
#pragma unroll
        for (int j = 0; j < kGemmBN; j += 32) {
            float v[32];
            tmem_ld32(tm + ((uint32_t)(32 * warp) << 16) + (uint32_t)j, v);
#pragma unroll
            for (int u = 0; u < 32; u += 4) red_add4(dst + j + u, v[u], v[u + 1], v[u + 2], v[u + 3]);
        }
    } else if (tid == 0) {
        atomicOr(flags, kFlagTimeout);
    }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    if (warp == 0) tmem_dealloc(tm, kGemmBN);
}

}  // namespace

bool encode_wgrad_maps(WgradMaps* maps, const bf16* dZ1T, const bf16* XT, const bf16* dZ2T, const bf16* H1T,
                       long long M, long long Mp)
{
    const unsigned long long rows = (unsigned long long)M, stride = (unsigned long long)Mp * 2;
    return encode_bf16_2d(&maps->dz1, dZ1T, rows, kH, stride, kGemmBK, kGemmBM, true) &&
           encode_bf16_2d(&maps->x, XT, rows, kInPad, stride, kGemmBK, kGemmBN, true) &&
           encode_bf16_2d(&maps->dz2, dZ2T, rows, kH, stride, kGemmBK, kGemmBM, true) &&
           encode_bf16_2d(&maps->h1, H1T, rows, kH, stride, kGemmBK, kGemmBN, true);
}

cudaError_t launch_wgrad(const WgradMaps& maps, long long M, float* gW1, float* gW2, unsigned* flags,
                         cudaStream_t s)
{
    const size_t smem = sizeof(GemmSmem) + 1024;              // room to align the base to 1 KB
    cudaError_t e = cudaFuncSetAttribute(k_wgrad, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    const int nchunks = (int)((M + kGemmBK - 1) / kGemmBK), tiles = kTiles1 + kTiles2;
    // about two blocks per SM, with at least four chunks each
    int splits = std::max(1, std::min((2 * device_sm_count() + tiles - 1) / tiles, nchunks / 4));
    const int per = (nchunks + splits - 1) / splits;
    splits = (nchunks + per - 1) / per;
    k_wgrad<<<dim3((unsigned)tiles, (unsigned)splits), 128, smem, s>>>(maps, nchunks, per, gW1, gW2, flags);
    return cudaGetLastError();
}

}  // namespace gk
