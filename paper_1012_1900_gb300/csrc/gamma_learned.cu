// Learned proposal for the gamma search: patch features, labels from the exact
// search, a 375-128-128-4 BF16 network trained and run with hand-written
// tensor-core kernels, and the seeding pass that turns its proposal into an
// exact upper bound before the table walk.
//
// None of this is in the paper.  The network never decides a result: its
// proposed nearest point only selects cells whose faces are evaluated
// exactly, and the distance found is a true distance to the evaluation
// surface, hence a valid upper bound on gamma.  The exact walk (Algorithm A1
// step 4) then runs unchanged from that bound.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math.h>

#include <algorithm>
#include <cstdio>
#include <cstring>
#include <new>
#include <vector>

#include "../../include/gamma.h"
#include "gamma_cell.cuh"
#include "gamma_internal.h"
#include "gamma_launch.cuh"
#include "gamma_mlp.cuh"
#include "gamma_plane.cuh"
#include "gamma_tc.cuh"

namespace gk {

using bf16 = __nv_bfloat16;

// --------------------------------------------------------------------------
// Features
// --------------------------------------------------------------------------

// The kInPad features of reference voxel v as one row: channel f / 125 over the
// 5^N patch p = v + o, o in {-2..2}^N (patch index f % 125, x fastest):
//   0: (D_e(p) - D_r(v)) / dD          clamped to [-16, 16]
//   1: |grad D_e(p)| * dta / dD        clamped to [0, 32]
//   2: |grad D_r(p)| * dta / dD        clamped to [0, 32]
// (gradients by central differences inside, one-sided at the grid edge); zero
// outside the grid and for f >= 375 (2D uses the first 25 of each 125).  One
// warp per row: it stages the 7^N neighbourhood of the voxel (the patch and the
// neighbours its gradients use) of both doses in shared memory (be, br), then
// each lane takes patch points and computes their three channels together.
constexpr int kBoxW = kPatch + 2;                    // 7
template <int N>
struct FeatBox {
    static constexpr int ELEMS = N == 3 ? kBoxW * kBoxW * kBoxW : kBoxW * kBoxW;
};

template <int N>
__device__ __forceinline__ void row_features(const Problem& P, unsigned v, float dr, float inv, float* be,
                                             float* br, bf16* __restrict__ xr)
{
    constexpr int E = FeatBox<N>::ELEMS;
    constexpr int NP = N == 3 ? 125 : 25;            // patch points used
    const int lane = threadIdx.x & 31;
    const int bst[3] = {1, kBoxW, kBoxW * kBoxW};
    const int x = (int)(v % (unsigned)P.nx);
    const unsigned r1 = v / (unsigned)P.nx;
    const int y = (int)(r1 % (unsigned)P.ny), z = (int)(r1 / (unsigned)P.ny);
    const int n[3] = {P.nx, P.ny, P.nz};
    float c1[3], c2[3];                                   // one-sided and central factors
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        c1[a] = 1.f / P.hn[a];
        c2[a] = 0.5f / P.hn[a];
    }
    // ---- the 7^N box around v (offsets -3 .. 3); outside the grid: 0 ----
    __syncwarp();
#pragma unroll 4
    for (int e = lane; e < E; e += 32) {
        const int ox = e % kBoxW - 3, oy = (e / kBoxW) % kBoxW - 3, oz = N == 3 ? e / (kBoxW * kBoxW) - 3 : 0;
        const int px = x + ox, py = y + oy, pz = z + oz;
        const bool in = (unsigned)px < (unsigned)P.nx && (unsigned)py < (unsigned)P.ny &&
                        (N == 2 || (unsigned)pz < (unsigned)P.nz);
        const long long p = ((long long)pz * P.ny + py) * P.nx + px;
        be[e] = in ? __ldg(P.ev + p) : 0.f;
        br[e] = in ? __ldg(P.ref + p) : 0.f;
    }
    __syncwarp();
    // ---- the three channels of one patch point per lane ----
    for (int pi = lane; pi < 125; pi += 32) {
        float f0 = 0.f, f1 = 0.f, f2 = 0.f;
        if (pi < NP) {
            const int o[3] = {pi % 5 - 2, (pi / 5) % 5 - 2, N == 3 ? pi / 25 - 2 : 0};
            const int c[3] = {x + o[0], y + o[1], z + o[2]};
            if ((unsigned)c[0] < (unsigned)P.nx && (unsigned)c[1] < (unsigned)P.ny &&
                (N == 2 || (unsigned)c[2] < (unsigned)P.nz)) {
                const int bi = ((o[2] + (N == 3 ? 3 : 0)) * kBoxW + (o[1] + 3)) * kBoxW + (o[0] + 3);
                f0 = fminf(fmaxf((be[bi] - dr) * inv, -16.f), 16.f);
                // the gradients of both doses (central differences inside,
                // one-sided at the grid edge)
                float se = 0.f, sr = 0.f;
#pragma unroll
                for (int a = 0; a < N; ++a) {
                    float de, dq;
                    if (c[a] > 0 && c[a] < n[a] - 1) {
                        de = (be[bi + bst[a]] - be[bi - bst[a]]) * c2[a];
                        dq = (br[bi + bst[a]] - br[bi - bst[a]]) * c2[a];
                    } else if (c[a] == 0) {
                        de = (be[bi + bst[a]] - be[bi]) * c1[a];
                        dq = (br[bi + bst[a]] - br[bi]) * c1[a];
                    } else {
                        de = (be[bi] - be[bi - bst[a]]) * c1[a];
                        dq = (br[bi] - br[bi - bst[a]]) * c1[a];
                    }
                    se = fmaf(de, de, se);
                    sr = fmaf(dq, dq, sr);
                }
                f1 = fminf(sqrtf(se) * inv, 32.f);
                f2 = fminf(sqrtf(sr) * inv, 32.f);
            }
        }
        xr[pi] = __float2bfloat16(f0);
        xr[125 + pi] = __float2bfloat16(f1);
        xr[250 + pi] = __float2bfloat16(f2);
    }
    if (lane < kInPad - kIn) xr[kIn + lane] = __float2bfloat16(0.f);
}

// Queue items past the cost gate (bucket >= min_bucket), into P.seed_list.
__global__ void __launch_bounds__(256) k_seed_select(const __grid_constant__ Problem P, int min_bucket)
{
    grid_release();
    grid_wait();
    const unsigned total = min(P.ctr->tail_count, P.tail_cap);
    const int lane = threadIdx.x & 31;
    const unsigned stride = gridDim.x * blockDim.x;
    for (unsigned c0 = blockIdx.x * blockDim.x; c0 < total; c0 += stride) {
        const unsigned i = c0 + threadIdx.x;
        const bool take = i < total && (int)P.tail_bucket[i] >= min_bucket;
        const unsigned m = __ballot_sync(0xffffffffu, take);
        unsigned base = 0;
        if (lane == 0 && m) base = atomicAdd(&P.ctr->seed_count, (unsigned)__popc(m));
        base = __shfl_sync(0xffffffffu, base, 0);
        if (take) P.seed_list[base + __popc(m & ((1u << lane) - 1u))] = i;
    }
}

// Features of listed voxels, one warp per row.  Bound by the latency of its
// loads and the stores of 768 bytes per row; eight features per thread, each
// with its own index arithmetic and loads, took 25.5 us for 4,096 rows of a
// 200x200x150 pair.
template <int N>
__global__ void __launch_bounds__(256) k_features(const __grid_constant__ Problem P,
                                                  const unsigned* __restrict__ vox, long long n,
                                                  bf16* __restrict__ X)
{
    __shared__ float sh_e[8][FeatBox<N>::ELEMS], sh_r[8][FeatBox<N>::ELEMS];
    const int wi = threadIdx.x >> 5;
    const float dnorm = resolve_dnorm(P);
    for (long long i = (long long)blockIdx.x * 8 + wi; i < n; i += (long long)gridDim.x * 8) {
        const unsigned v = vox[i];
        const float dr = __ldg(P.ref + v);
        const float dD = P.dd_frac * (P.local ? dr : dnorm);
        row_features<N>(P, v, dr, dD > 0.f ? 1.0f / dD : 0.f, sh_e[wi], sh_r[wi], X + i * kInPad);
    }
}

// --------------------------------------------------------------------------
// Cells around an arbitrary offset (labels and seeds)
// --------------------------------------------------------------------------

template <int N>
__device__ __forceinline__ bool load_cell(const Problem& P, int x, int y, int z, int cx, int cy,
                                          int cz, float dr, float inv, float (&q)[8], uint32_t& ok)
{
    const int px = x + cx, py = y + cy, pz = z + cz;
    if ((unsigned)px >= (unsigned)P.nx || (unsigned)py >= (unsigned)P.ny ||
        (N == 3 && (unsigned)pz >= (unsigned)P.nz))
        return false;
    const bool ex = px + 1 < P.nx, ey = py + 1 < P.ny, ez = N == 3 && pz + 1 < P.nz;
    const long long sy = P.nx, sz = (long long)P.nx * P.ny;
    const long long p = (long long)pz * sz + (long long)py * sy + px;
    ok = 0;
#pragma unroll
    for (int u = 0; u < 8; ++u) {
        q[u] = kNaN;
        if (u < (1 << N)) {
            const bool present = (!(u & 1) || ex) && (!(u & 2) || ey) && (!(u & 4) || ez);
            if (present) {
                const long long o = p + ((u & 1) ? 1 : 0) + ((u & 2) ? sy : 0) + ((u & 4) ? sz : 0);
                q[u] = (__ldg(P.ev + o) - dr) * inv;
                ok |= 1u << u;
            }
        }
    }
    return true;
}

// Labels: for each listed voxel, the nearest point of the evaluation surface
// (over the cells up to the gamma already computed) as an offset in normalised
// spatial units, and log(gamma + 1e-3).  Rows whose search would leave the
// table, or whose voxel is not evaluated, get NaN.
//
// One warp per voxel, a cell per lane and round: first the 2^N cells whose box
// contains the voxel (the table keys them by their faces off the voxel only),
// then the table.  A cell whose key and dose gap, or whose plane_bound, put it
// beyond the gamma known is passed over; of the others the first in that order
// with the smallest distance gives the point.  Bound by the latency of a few
// rounds.  One thread per voxel that evaluated every cell took 184 us for 4,096
// voxels of a 200x200x150 pair at 2 %/2 mm (32 blocks, one warp per scheduler).
template <int N>
__global__ void __launch_bounds__(128) k_labels(const __grid_constant__ Problem P,
                                                const float* __restrict__ gmap,
                                                const unsigned* __restrict__ vox, long long n,
                                                float* __restrict__ T)
{
    const int lane = threadIdx.x & 31;
    const float dnorm = P.dose_norm > 0.f ? P.dose_norm : fdec(P.ctr->dnorm_enc);
    const float hn2[3] = {P.mt.hn2[0], P.mt.hn2[1], P.mt.hn2[2]};
    const float kap[3] = {P.mt.kappa[1], P.mt.kappa[2], P.mt.kappa[4]};
    for (long long i = (long long)blockIdx.x * 4 + (threadIdx.x >> 5); i < n; i += (long long)gridDim.x * 4) {
        const unsigned v = vox[i];                            // warp-uniform
        const float gs = gmap[v];
        float* t = T + 4 * i;
        if (!(gs >= 0.f) || gs > P.r_cover) {
            if (lane < 4) t[lane] = kNaN;
            continue;
        }
        const int x = (int)(v % (unsigned)P.nx);
        const unsigned r1 = v / (unsigned)P.nx;
        const int y = (int)(r1 % (unsigned)P.ny), z = (int)(r1 / (unsigned)P.ny);
        const float dr = __ldg(P.ref + v);
        const float inv = 1.0f / (P.dd_frac * (P.local ? dr : dnorm));
        const float lim = gs * (1.f + 1e-5f) + 1e-6f;
        // a cell beyond this squared distance cannot hold the nearest point
        // (the bounds' own rounding is some 1e-5 of it)
        const float lim2 = lim * lim * (1.f + 1e-4f);
        float best = kInf, fv[3] = {0.f, 0.f, 0.f};
        // (a map that holds less than the distance found: again, every cell)
        for (int all = 0; all < 2 && !(best <= lim2); ++all)
            for (int base = 0;; base += 32) {
                const int k = base + lane - (1 << N);             // < 0: the cells around the voxel
                int cx = 0, cy = 0, cz = 0;
                float key = 0.f;
                bool in = false;
                if (k < 0) {
                    const int c = k + (1 << N);
                    cx = -(c & 1);
                    cy = -((c >> 1) & 1);
                    cz = N == 3 ? -((c >> 2) & 1) : 0;
                    in = true;
                } else if (k < P.ntable) {
                    const TableEntry e = P.table[k];
                    key = e.key;
                    in = key <= lim;
                    cx = unpack10(e.off, 0);
                    cy = unpack10(e.off, 10);
                    cz = unpack10(e.off, 20);
                }
                if (!__any_sync(0xffffffffu, in)) break;          // keys only grow
                if (k >= 0 && cx >= -1 && cx <= 0 && cy >= -1 && cy <= 0 && cz >= -1 && cz <= 0) in = false;
                float q[8], d2 = kInf, foot[3] = {0.f, 0.f, 0.f};
                uint32_t ok = 0;
                if (in) in = load_cell<N>(P, x, y, z, cx, cy, cz, dr, inv, q, ok);
                if (in && !all) {
                    float qlo = kInf, qhi = -kInf;
#pragma unroll
                    for (int u = 0; u < (1 << N); ++u) {          // (NaN: no such vertex)
                        qlo = fminf(qlo, q[u]);
                        qhi = fmaxf(qhi, q[u]);
                    }
                    const float gap = max3(qlo, -qhi, 0.f);
                    in = !(fmaf(gap, gap, key * key) > lim2);
                    if (in && ok == (1u << (1 << N)) - 1u) {
                        const float c[3] = {(float)cx, (float)cy, (float)cz};
                        in = !(plane_bound<N>(q, c, 0.f, 1.f, hn2, kap) > lim2);
                    }
                }
                if (in) {
                    CellGeom<float> g;
                    cell_geom<N, float>(cx, cy, cz, P.mt, g);
                    cell_argmin<N, float>(q, g, P.mt, d2, foot);
                }
                // the smallest, and of equal ones the first
                const unsigned bits = __float_as_uint(d2 + 0.f);
                const unsigned m = __reduce_min_sync(0xffffffffu, bits);
                if (m < __float_as_uint(best)) {
                    best = __uint_as_float(m);
                    const int src = __ffs(__ballot_sync(0xffffffffu, bits == m)) - 1;
                    fv[0] = __shfl_sync(0xffffffffu, cx + foot[0], src);
                    fv[1] = __shfl_sync(0xffffffffu, cy + foot[1], src);
                    fv[2] = __shfl_sync(0xffffffffu, cz + foot[2], src);
                }
            }
        if (lane == 0) {
            t[0] = fv[0] * P.hn[0];
            t[1] = fv[1] * P.hn[1];
            t[2] = N == 3 ? fv[2] * P.hn[2] : 0.f;
            t[3] = logf(gs + 1e-3f);
        }
    }
}

// --------------------------------------------------------------------------
// Optimiser
// --------------------------------------------------------------------------

// Where parameter i goes among the BF16 copies of the weights (W2 also
// transposed, for dH1): nothing for the biases.
struct WeightCopies {
    bf16 *W1h, *W2h, *W2Th, *W3h;
    int off_w2, off_w3;                    // first parameters of W2 and W3 (W1 starts at 0)
    __device__ __forceinline__ void put(int i, float p) const
    {
        const bf16 v = __float2bfloat16(p);
        if (i < kH * kInPad) {
            W1h[i] = v;
        } else if (i >= off_w2 && i < off_w2 + kH * kH) {
            const int k = i - off_w2;
            W2h[k] = v;
            W2Th[(k % kH) * kH + k / kH] = v;
        } else if (i >= off_w3 && i < off_w3 + kOutPad * kH) {
            W3h[i - off_w3] = v;
        }
    }
};

// Adam on the FP32 master parameters, and their BF16 copies; padded entries
// (mask == 0) stay zero.
__global__ void __launch_bounds__(256) k_adam(int n, float* __restrict__ p, const float* __restrict__ g,
                                              float* __restrict__ m, float* __restrict__ v,
                                              const unsigned char* __restrict__ mask, WeightCopies copies,
                                              float lr, float b1, float b2, float eps, float c1, float c2)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        if (!mask[i]) continue;
        const float gi = g[i];
        const float mi = b1 * m[i] + (1.f - b1) * gi;
        const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
        m[i] = mi;
        v[i] = vi;
        const float pi = p[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
        p[i] = pi;
        copies.put(i, pi);
    }
}

// The BF16 copies of all parameters.
__global__ void __launch_bounds__(256) k_cast_weights(int n, const float* __restrict__ p, WeightCopies copies)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) copies.put(i, p[i]);
}

// --------------------------------------------------------------------------
// Network inference on the fifth-generation tensor cores (tcgen05)
//
// One block per SM keeps the three weight matrices resident in shared memory
// and runs 128 feature rows at a time, each of its warps in one role:
//   warp 8   copies the rows: 64-column panels of 128 rows x 128 bytes by TMA
//            (128-byte swizzle) through three stages, always three ahead;
//   warp 9   issues layer 1, X W1^T over the six panels, into two accumulators
//            in turn (TMEM columns 0..127, 128..255), so that the rows keep
//            arriving while the tile before is finished;
//   warp 10  issues layers 2 and 3: H1 W2^T in columns 256..383, H2 W3^T (N
//            padded to 16) in 384..399;
//   warps 0-7 the epilogues: TMEM to registers (warp w reads lanes 32 (w % 4)
//            .. +31), bias and ReLU, and the next layer's BF16 operand into
//            shared memory (H2 over H1, whose MMAs have completed), no-swizzle
//            K-major core-matrix layout (8 rows x 16 bytes per core matrix).
// Everything between the roles is an mbarrier; every wait is bounded.
//
// What bounds it: reading the rows (768 bytes each).  A panel used to arrive
// as eight boxes of 16-byte rows, and one thread took copies, MMAs and
// epilogues in turn: 204 us for 262,144 rows (0.99 TB/s).  With whole 128-byte
// rows per box and the roles apart it takes 61 us with one thread issuing all
// three layers, and 50 us with layer 1 apart (4.0 TB/s); three panels (48 KB)
// in flight per SM is what the weights leave room for.
// --------------------------------------------------------------------------

constexpr int kRows = 128;                 // rows per tile (MMA M)
constexpr int kKc = 64;                    // columns of a panel of streamed features
constexpr int kNChunks = kInPad / kKc;     // 6
constexpr int kXStages = 3;                // panels in flight
constexpr int kN3 = 16;                    // layer-3 N (4 outputs, padded)
constexpr int kTmemCols = 512;             // 400 used; allocations are powers of two
constexpr int kMlpThreads = 352;
constexpr int kEpiWarps = 8;
constexpr int kStagers = kMlpThreads - 32; // threads that stage the weights: all but the copying warp's
constexpr int kPanel = kRows * kKc;        // elements of a panel (rows 128)

struct __align__(1024) TcSmem {
    bf16 W1[kNChunks][kPanel];             // rows 128, 64-column panels (128-byte swizzle)
    bf16 Xc[kXStages][kPanel];             // feature panels (TMA destinations, 128-byte swizzle)
    bf16 W2[kH * kH];                      // rows 128, K 128 (core-matrix layout)
    bf16 H[kRows * kH];                    // H1, then H2 (rows 128, K 128; core-matrix layout)
    bf16 W3[kN3 * kH];                     // rows 16, K 128 (rows >= kOut zero)
    float b1[kH], b2[kH], b3[kOutPad];
    uint64_t xfull[kXStages], xempty[kXStages];
    uint64_t d1[2], d2, d3;                // a layer's accumulator is complete
    uint64_t e1[2];                        // layer 1's accumulator is read (one arrival per epilogue warp)
    uint64_t h1, h2;                       // a layer's operand is written (likewise)
    uint32_t tmem;
};

// Element index of (row, k) in a core-matrix tile with `rows` rows.
__device__ __forceinline__ int core_idx(int row, int k, int rows)
{
    return (((k >> 3) * (rows >> 3) + (row >> 3)) << 6) + ((row & 7) << 3) + (k & 7);
}

// Descriptor of the K = 16 slice starting at column k0 of a core-matrix tile.
__device__ __forceinline__ uint64_t tile_desc(const bf16* base, int rows, int k0)
{
    const uint32_t lbo = (uint32_t)(rows >> 3) * 128u;
    return smem_desc(smem_addr(base) + (uint32_t)(k0 >> 3) * lbo, lbo, 128u);
}

// Row-major [rows][K] BF16 weights (global) -> core-matrix tile (shared), by
// thread `first` of `step`.
__device__ __forceinline__ void stage_weights(bf16* dst, const bf16* __restrict__ src, int rows,
                                              int src_rows, int K, int first, int step)
{
    const int n = rows * (K / 8);
#pragma unroll 4
    for (int e = first; e < n; e += step) {
        const int r = e / (K / 8), j = e % (K / 8);
        uint4 v = make_uint4(0u, 0u, 0u, 0u);
        if (r < src_rows) v = *reinterpret_cast<const uint4*>(src + (long long)r * K + j * 8);
        *reinterpret_cast<uint4*>(dst + core_idx(r, j * 8, rows)) = v;
    }
}

// Row-major [128][384] BF16 weights (global) -> swizzled 64-column panels.
__device__ __forceinline__ void stage_panels(bf16 (*dst)[kPanel], const bf16* __restrict__ src, int first,
                                             int step)
{
#pragma unroll 8
    for (int e = first; e < kH * (kInPad / 8); e += step) {
        const int r = e / (kInPad / 8), j = e % (kInPad / 8);
        *reinterpret_cast<uint4*>(dst[j >> 3] + r * kKc + (((j & 7) ^ (r & 7)) << 3)) =
            *reinterpret_cast<const uint4*>(src + (long long)r * kInPad + j * 8);
    }
}

// D (TMEM, 128 lanes x 128 columns from column `col`) + bias, ReLU -> BF16
// core-matrix tile `dst` (rows 128, K 128); warps 0-7, half the columns each.
__device__ __forceinline__ void epilogue_relu(uint32_t tmem, uint32_t col, const float* bias, bf16* dst)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int q = warp & 3, half = warp >> 2, row = 32 * q + lane;
#pragma unroll 1
    for (int j = 0; j < 2; ++j) {
        const int c0 = half * 64 + j * 32;
        float v[32];
        tmem_ld32(tmem + ((uint32_t)(32 * q) << 16) + col + (uint32_t)c0, v);
#pragma unroll
        for (int h = 0; h < 4; ++h) {
            uint32_t w[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int c = c0 + 8 * h + 2 * i;
                const __nv_bfloat162 pr = __floats2bfloat162_rn(fmaxf(v[8 * h + 2 * i] + bias[c], 0.f),
                                                                fmaxf(v[8 * h + 2 * i + 1] + bias[c + 1], 0.f));
                w[i] = *reinterpret_cast<const uint32_t*>(&pr);
            }
            *reinterpret_cast<uint4*>(dst + core_idx(row, c0 + 8 * h, kRows)) =
                make_uint4(w[0], w[1], w[2], w[3]);
        }
    }
}

// The block's smem is the whole 227 KB (one block per SM; the TMEM allocation
// can then never wait).
constexpr size_t kTcSmemBytes = 232448;
static_assert(sizeof(TcSmem) + 1024 <= kTcSmemBytes, "tensor-core tile does not fit in shared memory");

// Network outputs Y [rows][4] of the feature rows X [rows][384] (bf16, read by
// the tensor map xmap), for rows < (*count_dev if given, capped at M, else M).
// A timed-out wait sets kFlagTimeout in *flags (host_flags: page-locked host
// memory, written by a plain store).
__global__ void __launch_bounds__(kMlpThreads, 1) k_mlp_rows(const __grid_constant__ MlpWeights W,
                                                             const __grid_constant__ CUtensorMap xmap,
                                                             long long M, const unsigned* count_dev,
                                                             float* __restrict__ Y, unsigned* flags,
                                                             int host_flags)
{
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char* base = smem_raw + ((1024u - (smem_addr(smem_raw) & 1023u)) & 1023u);
    TcSmem& S = *reinterpret_cast<TcSmem*>(base);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (count_dev) grid_release();       // within a run; by itself it is the call's last kernel
    grid_wait();
    const long long nrows = count_dev ? min((long long)*count_dev, M) : M;
    const long long ntiles = (nrows + kRows - 1) / kRows;
    if ((long long)blockIdx.x >= ntiles) return;                  // block-uniform
    if (tid == 0) {
        for (int b = 0; b < kXStages; ++b) {
            mbar_init(&S.xfull[b], 1);
            mbar_init(&S.xempty[b], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&S.d1[b], 1);
            mbar_init(&S.e1[b], kEpiWarps);
        }
        mbar_init(&S.d2, 1);
        mbar_init(&S.d3, 1);
        mbar_init(&S.h1, kEpiWarps);
        mbar_init(&S.h2, kEpiWarps);
        mbar_fence_init();
    }
    if (warp == 0) {
        tmem_alloc(&S.tmem, kTmemCols);
        tmem_relinquish();
    }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    if (warp != kEpiWarps) {             // (the rows' copies start meanwhile)
        const int i = warp < kEpiWarps ? tid : tid - 32;
        stage_panels(S.W1, W.W1, i, kStagers);
        stage_weights(S.W2, W.W2, kH, kH, kH, i, kStagers);
        stage_weights(S.W3, W.W3, kN3, kOutPad, kH, i, kStagers);
        for (int k = i; k < kH; k += kStagers) {
            S.b1[k] = W.b1[k];
            S.b2[k] = W.b2[k];
        }
        if (i < kOutPad) S.b3[i] = W.b3[i];
        fence_async_shared();
        asm volatile("bar.sync 1, %0;" ::"n"(kStagers) : "memory");
    }
    const uint32_t tm = S.tmem;
    bool ok = true;
    if (warp == kEpiWarps) {
        // ---- the copies ----
        if (lane == 0) {
            uint32_t n = 0;                                       // panels requested
            for (long long t = blockIdx.x; t < ntiles && ok; t += gridDim.x)
                for (int c = 0; c < kNChunks && ok; ++c, ++n) {
                    const uint32_t s = n % kXStages;
                    if (n >= kXStages) ok = mbar_wait_bounded(&S.xempty[s], (n / kXStages - 1) & 1u);
                    if (!ok) break;
                    mbar_arrive_expect_tx(&S.xfull[s], kPanel * 2);
                    tma_load_2d(S.Xc[s], &xmap, c * kKc, (int)(t * kRows), &S.xfull[s]);
                }
            // the copies still in flight land before the block leaves
            for (uint32_t k = n > kXStages ? n - kXStages : 0; k < n; ++k)
                mbar_wait_bounded(&S.xfull[k % kXStages], (k / kXStages) & 1u);
        }
    } else if (warp == kEpiWarps + 1) {
        // ---- layer 1 ----
        if (lane == 0) {
            constexpr uint32_t kId = idesc_bf16_f32(kRows, kH);
            uint32_t n = 0, i = 0;                                // panels consumed, tiles begun
            for (long long t = blockIdx.x; t < ntiles && ok; t += gridDim.x, ++i) {
                const uint32_t b = i & 1u;
                if (i >= 2) ok = mbar_wait_bounded(&S.e1[b], (i / 2 - 1) & 1u);
                for (int c = 0; c < kNChunks && ok; ++c, ++n) {
                    const uint32_t s = n % kXStages;
                    ok = mbar_wait_bounded(&S.xfull[s], (n / kXStages) & 1u);
                    if (!ok) break;
                    tc_fence_after_sync();
                    const uint32_t xa = smem_addr(S.Xc[s]), wa = smem_addr(S.W1[c]);
#pragma unroll
                    for (int kk = 0; kk < kKc; kk += 16)
                        tc_mma_bf16(tm + b * kH, smem_desc_sw128(xa, kk * 2), smem_desc_sw128(wa, kk * 2), kId,
                                    (c | kk) != 0);
                    tc_commit(&S.xempty[s]);
                }
                tc_commit(&S.d1[b]);
            }
        }
    } else if (warp == kEpiWarps + 2) {
        // ---- layers 2 and 3 ----
        if (lane == 0) {
            constexpr uint32_t kId128 = idesc_bf16_f32(kRows, kH), kId16 = idesc_bf16_f32(kRows, kN3);
            uint32_t i = 0;
            for (long long t = blockIdx.x; t < ntiles && ok; t += gridDim.x, ++i) {
                ok = mbar_wait_bounded(&S.h1, i & 1u);
                if (!ok) break;
                tc_fence_after_sync();
#pragma unroll
                for (int kk = 0; kk < kH; kk += 16)
                    tc_mma_bf16(tm + 2 * kH, tile_desc(S.H, kRows, kk), tile_desc(S.W2, kH, kk), kId128, kk != 0);
                tc_commit(&S.d2);
                ok = mbar_wait_bounded(&S.h2, i & 1u);
                if (!ok) break;
                tc_fence_after_sync();
#pragma unroll
                for (int kk = 0; kk < kH; kk += 16)
                    tc_mma_bf16(tm + 3 * kH, tile_desc(S.H, kRows, kk), tile_desc(S.W3, kN3, kk), kId16, kk != 0);
                tc_commit(&S.d3);
            }
        }
    } else {
        // ---- the epilogues ----
        uint32_t i = 0;
        for (long long t = blockIdx.x; t < ntiles && ok; t += gridDim.x, ++i) {
            ok = __all_sync(0xffffffffu, mbar_wait_bounded(&S.d1[i & 1u], (i / 2) & 1u));
            if (!ok) break;
            tc_fence_after_sync();
            epilogue_relu(tm, (i & 1u) * kH, S.b1, S.H);
            fence_async_shared();
            tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) {
                mbar_arrive(&S.e1[i & 1u]);
                mbar_arrive(&S.h1);
            }
            ok = __all_sync(0xffffffffu, mbar_wait_bounded(&S.d2, i & 1u));
            if (!ok) break;
            tc_fence_after_sync();
            epilogue_relu(tm, 2u * kH, S.b2, S.H);                // H2 over H1 (its MMAs have completed)
            fence_async_shared();
            tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) mbar_arrive(&S.h2);
            ok = __all_sync(0xffffffffu, mbar_wait_bounded(&S.d3, i & 1u));
            if (!ok) break;
            tc_fence_after_sync();
            if (warp < 4) {
                float v[16];
                tmem_ld16(tm + ((uint32_t)(32 * warp) << 16) + 3 * kH, v);
                const long long row = t * kRows + 32 * warp + lane;
                if (row < nrows) {
                    float* y = Y + row * kOut;
#pragma unroll
                    for (int o = 0; o < kOut; ++o) y[o] = v[o] + S.b3[o];
                }
            }
            tc_fence_before_sync();
        }
    }
    if (!ok && lane == 0) {
        if (host_flags) *(volatile unsigned*)flags = kFlagTimeout;
        else atomicOr(flags, kFlagTimeout);
    }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    if (warp == 0) tmem_dealloc(tm, kTmemCols);
}

cudaError_t launch_mlp_rows(const MlpWeights& W, const bf16* X, long long M, const unsigned* count_dev,
                            float* Y, unsigned* flags, int host_flags, cudaStream_t s)
{
    if (M <= 0) return cudaSuccess;
    CUtensorMap xmap;
    if (!encode_bf16_2d(&xmap, X, kInPad, (unsigned long long)M, kInPad * 2, kKc, kRows, true))
        return cudaErrorInvalidValue;
    cudaError_t e = cudaFuncSetAttribute(k_mlp_rows, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)kTcSmemBytes);
    if (e != cudaSuccess) return e;
    const long long tiles = (M + kRows - 1) / kRows;
    const int grid = (int)std::max<long long>(1, std::min<long long>(tiles, device_sm_count()));
    if (count_dev)       // within a run: the kernels before it on the stream are the run's own
        launch_next(k_mlp_rows, grid, kMlpThreads, kTcSmemBytes, s, W, xmap, M, count_dev, Y, flags, host_flags);
    else
        k_mlp_rows<<<grid, kMlpThreads, kTcSmemBytes, s>>>(W, xmap, M, count_dev, Y, flags, host_flags);
    return cudaGetLastError();
}

cudaError_t launch_mlp_infer(const MlpWeights& W, const bf16* X, long long M, float* Y,
                             unsigned* host_flags, cudaStream_t s)
{
    return launch_mlp_rows(W, X, M, nullptr, Y, host_flags, 1, s);
}

// --------------------------------------------------------------------------
// Training: forward, loss and the backward pass of the rows in one kernel
//
// A block takes one tile of 128 rows through
//   Z1 = X W1^T + b1, H1 = relu(Z1),  Z2 = H1 W2^T + b2, H2 = relu(Z2),
//   Y = H2 W3^T + b3,  the Huber loss and dY,
//   dZ2 = (dY W3) * [Z2 > 0],  dH1 = dZ2 W2,  dZ1 = dH1 * [Z1 > 0]
// with the four products on the tensor cores (operands in shared memory,
// accumulators in TMEM: columns 0..127 Z1 and then dH1, 128..255 Z2, 256..271
// Y), the element-wise parts in the epilogue warps between them, and the ReLU
// masks in their registers.  Per tile it adds the column sums (bias gradients,
// dW3 = dY^T H2) to the gradients, and it writes what the weight-gradient
// product needs, with the batch as K: X, H1, dZ1 and dZ2 transposed ([column]
// [row], a lane per row, so that a warp's stores are 64 contiguous bytes).
// Warp 8 copies the panels of X, warp 9 issues the MMAs.  Every wait is
// bounded, and every warp passes every block barrier.
//
// What bounds it: the latency of one tile's chain (a training batch of 8,192
// rows is 64 tiles).  Before, the same work took 17 launches: a GEMM per
// product, bias, activation, loss, mask, column-sum and transpose passes
// over memory: about 190 us of kernels in a step of 8,192 rows, now 42 us here
// and 11 us in k_wgrad.
// --------------------------------------------------------------------------

struct __align__(1024) TrainSmem {
    bf16 W1[kNChunks][kPanel];             // W1 panels (128-byte swizzle); W2^T (core matrices) once Z1 is done
    bf16 Xc[kXStages][kPanel];             // X panels (128-byte swizzle); then dZ2 (core matrices)
    bf16 W2[kH * kH];                      // core matrices, as below
    bf16 H[kRows * kH];                    // H1, then H2
    bf16 W3[kN3 * kH];
    float W3f[kOut * kH];                  // the FP32 master of W3
    float dY[kRows][kOut];
    float gW3[kOut * kH], gb1[kH], gb2[kH], gb3[kOut];   // this tile's sums
    float b1[kH], b2[kH], b3[kOutPad];
    uint64_t xfull[kXStages], xempty[kXStages];   // (xempty: the MMAs and the eight transposing warps)
    uint64_t d1, d2, d3, d4, h1, h2, z2;
    uint32_t tmem;
};
static_assert(sizeof(TrainSmem) + 1024 <= kTcSmemBytes, "training tile does not fit in shared memory");
static_assert(sizeof(bf16) * kXStages * kPanel >= sizeof(bf16) * kRows * kH, "dZ2 takes the X panels' place");

struct TrainArgs {
    MlpWeights W;
    const bf16* W2T;                       // [kH][kH], W2 transposed
    const float* W3f;                      // [kOutPad][kH], FP32 master
    const float* T;                        // [M][kOut] targets
    long long M, Mp;                       // rows; row stride of the transposed outputs
    float inv_count;
    bf16 *XT, *H1T, *dZ1T, *dZ2T;          // [kInPad or kH][Mp]
    float *gb1, *gb2, *gW3, *gb3, *loss;
    unsigned* flags;
};

// Column sums over a warp's 32 rows: lane l gets the sum of v[l] over the
// lanes (31 exchanges for 32 columns).
__device__ __forceinline__ float warp_column_sum(float (&v)[32])
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int m = 16; m >= 1; m >>= 1) {
        const bool up = lane & m;
#pragma unroll
        for (int i = 0; i < m; ++i) {
            const float send = up ? v[i] : v[i + m], keep = up ? v[i + m] : v[i];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, m);
        }
    }
    return v[0];
}

constexpr int kTrainThreads = 320;

__global__ void __launch_bounds__(kTrainThreads, 1) k_train_rows(const __grid_constant__ TrainArgs A,
                                                                 const __grid_constant__ CUtensorMap xmap)
{
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char* base = smem_raw + ((1024u - (smem_addr(smem_raw) & 1023u)) & 1023u);
    TrainSmem& S = *reinterpret_cast<TrainSmem*>(base);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const long long row0 = (long long)blockIdx.x * kRows;
    if (tid == 0) {
        for (int b = 0; b < kXStages; ++b) {
            mbar_init(&S.xfull[b], 1);
            mbar_init(&S.xempty[b], 1 + kEpiWarps);
        }
        mbar_init(&S.d1, 1);
        mbar_init(&S.d2, 1);
        mbar_init(&S.d3, 1);
        mbar_init(&S.d4, 1);
        mbar_init(&S.h1, kEpiWarps);
        mbar_init(&S.h2, kEpiWarps);
        mbar_init(&S.z2, kEpiWarps);
        mbar_fence_init();
    }
    if (warp == 0) {
        tmem_alloc(&S.tmem, kTmemCols);
        tmem_relinquish();
    }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tm = S.tmem;
    bool ok = true;
    if (warp == kEpiWarps) {
        // ---- the copies (from here on, while the others stage the weights) ----
        if (lane == 0) {
            int c = 0;
            for (; c < kNChunks; ++c) {
                const int s = c % kXStages;
                if (c >= kXStages) ok = mbar_wait_bounded(&S.xempty[s], (c / kXStages - 1) & 1u);
                if (!ok) break;
                mbar_arrive_expect_tx(&S.xfull[s], kPanel * 2);
                tma_load_2d(S.Xc[s], &xmap, c * kKc, (int)row0, &S.xfull[s]);
            }
            // the copies still in flight land before the block leaves
            for (int k = max(0, c - kXStages); k < c; ++k) mbar_wait_bounded(&S.xfull[k % kXStages], (k / kXStages) & 1u);
        }
    } else {
        constexpr int n = kTrainThreads - 32;
        const int i0 = warp < kEpiWarps ? tid : tid - 32;
        stage_panels(S.W1, A.W.W1, i0, n);
        stage_weights(S.W2, A.W.W2, kH, kH, kH, i0, n);
        stage_weights(S.W3, A.W.W3, kN3, kOutPad, kH, i0, n);
        for (int k = i0; k < kOut * kH; k += n) {
            S.W3f[k] = A.W3f[k];
            S.gW3[k] = 0.f;
        }
        for (int k = i0; k < kH; k += n) {
            S.b1[k] = A.W.b1[k];
            S.b2[k] = A.W.b2[k];
            S.gb1[k] = S.gb2[k] = 0.f;
        }
        if (i0 < kOutPad) S.b3[i0] = A.W.b3[i0];
        if (i0 < kOut) S.gb3[i0] = 0.f;
        fence_async_shared();
        asm volatile("bar.sync 1, %0;" ::"n"(n) : "memory");
    }
    if (warp == kEpiWarps + 1) {
        // ---- the MMAs ----
        if (lane == 0) {
            constexpr uint32_t kId128 = idesc_bf16_f32(kRows, kH), kId16 = idesc_bf16_f32(kRows, kN3);
            for (int c = 0; c < kNChunks && ok; ++c) {
                const int s = c % kXStages;
                ok = mbar_wait_bounded(&S.xfull[s], (c / kXStages) & 1u);
                if (!ok) break;
                tc_fence_after_sync();
                const uint32_t xa = smem_addr(S.Xc[s]), wa = smem_addr(S.W1[c]);
#pragma unroll
                for (int kk = 0; kk < kKc; kk += 16)
                    tc_mma_bf16(tm, smem_desc_sw128(xa, kk * 2), smem_desc_sw128(wa, kk * 2), kId128, (c | kk) != 0);
                tc_commit(&S.xempty[s]);
            }
            tc_commit(&S.d1);
            auto layer = [&](uint64_t* ready, const bf16* a, const bf16* b, int brows, uint32_t col, uint32_t id,
                             uint64_t* done) {
                if (ok) ok = mbar_wait_bounded(ready, 0u);
                if (!ok) return;
                tc_fence_after_sync();
#pragma unroll
                for (int kk = 0; kk < kH; kk += 16)
                    tc_mma_bf16(tm + col, tile_desc(a, kRows, kk), tile_desc(b, brows, kk), id, kk != 0);
                tc_commit(done);
            };
            layer(&S.h1, S.H, S.W2, kH, kH, kId128, &S.d2);
            layer(&S.h2, S.H, S.W3, kN3, 2 * kH, kId16, &S.d3);
            layer(&S.z2, S.Xc[0], S.W1[0], kH, 0, kId128, &S.d4);
        }
    } else if (warp < kEpiWarps) {
        // ---- the element-wise parts: row 32 q + lane, columns 64 half .. + 63 ----
        const int q = warp & 3, half = warp >> 2, row = 32 * q + lane;
        const long long grow = row0 + row;
        const bool store = grow < A.Mp, live = grow < A.M;
        const uint32_t tl = tm + ((uint32_t)(32 * q) << 16);
        auto wait = [&](uint64_t* bar, uint32_t parity) {
            ok = __all_sync(0xffffffffu, ok && mbar_wait_bounded(bar, parity));
            return ok;
        };
        // X transposed, while the MMAs take the same panels
        for (int c = 0; c < kNChunks; ++c) {
            const int s = c % kXStages;
            if (!wait(&S.xfull[s], (c / kXStages) & 1u)) break;
            if (store) {
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int ch = half * 4 + j;
                    uint4 v = *reinterpret_cast<const uint4*>(S.Xc[s] + row * kKc + ((ch ^ (row & 7)) << 3));
                    const bf16* e = reinterpret_cast<const bf16*>(&v);
                    bf16* dst = A.XT + (long long)(c * kKc + ch * 8) * A.Mp + grow;
#pragma unroll
                    for (int u = 0; u < 8; ++u) dst[u * A.Mp] = e[u];
                }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&S.xempty[s]);
        }
        // an activation epilogue: bias, ReLU, BF16 into H, the mask of positive
        // values, and (H1) the transposed output
        auto activate = [&](uint32_t col, const float* bias, uint32_t (&mask)[2], bf16* outT) {
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const int c0 = half * 64 + j * 32;
                float v[32];
                tmem_ld32(tl + col + (uint32_t)c0, v);
                mask[j] = 0;
#pragma unroll
                for (int h = 0; h < 4; ++h) {
                    uint4 w;
                    bf16* o = reinterpret_cast<bf16*>(&w);
#pragma unroll
                    for (int u = 0; u < 8; ++u) {
                        const float z = v[8 * h + u] + bias[c0 + 8 * h + u];
                        mask[j] |= z > 0.f ? 1u << (8 * h + u) : 0u;
                        o[u] = __float2bfloat16(fmaxf(z, 0.f));
                        if (outT && store)
                            outT[(long long)(c0 + 8 * h + u) * A.Mp + grow] = live ? o[u] : __float2bfloat16(0.f);
                    }
                    *reinterpret_cast<uint4*>(S.H + core_idx(row, c0 + 8 * h, kRows)) = w;
                }
            }
            fence_async_shared();
            tc_fence_before_sync();
            __syncwarp();
        };
        uint32_t m1[2] = {0, 0}, m2[2] = {0, 0};
        if (wait(&S.d1, 0u)) {
            tc_fence_after_sync();
            activate(0u, S.b1, m1, A.H1T);
            if (lane == 0) mbar_arrive(&S.h1);
            // W1 has been used: W2^T takes its place (ordered by the arrival on z2)
            stage_weights(S.W1[0], A.W2T, kH, kH, kH, tid, kEpiWarps * 32);
        }
        if (wait(&S.d2, 0u)) {
            tc_fence_after_sync();
            activate(kH, S.b2, m2, nullptr);
            if (lane == 0) mbar_arrive(&S.h2);
        }
        if (wait(&S.d3, 0u) && warp < 4) {
            // loss and dY of this lane's row (Huber, delta 1; rows without a finite
            // target are passed over)
            tc_fence_after_sync();
            float y[16], t[kOut] = {0.f, 0.f, 0.f, 0.f}, acc = 0.f;
            tmem_ld16(tl + 2 * kH, y);
            bool valid = false;
            if (live) {
#pragma unroll
                for (int j = 0; j < kOut; ++j) t[j] = A.T[grow * kOut + j];
                valid = isfinite(t[kOut - 1]);
            }
            float d[kOut];
#pragma unroll
            for (int j = 0; j < kOut; ++j) {
                const float r = valid ? y[j] + S.b3[j] - t[j] : 0.f;
                const float a = fabsf(r);
                acc += a <= 1.f ? 0.5f * r * r : a - 0.5f;
                d[j] = live ? (a <= 1.f ? r : copysignf(1.f, r)) * A.inv_count : 0.f;
                S.dY[row][j] = d[j];
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                acc += __shfl_xor_sync(0xffffffffu, acc, o);
#pragma unroll
                for (int j = 0; j < kOut; ++j) d[j] += __shfl_xor_sync(0xffffffffu, d[j], o);
            }
            if (lane == 0) {
                atomicAdd(A.loss, acc * A.inv_count);
#pragma unroll
                for (int j = 0; j < kOut; ++j) atomicAdd(&S.gb3[j], d[j]);
            }
        }
        asm volatile("bar.sync 2, %0;" ::"n"(kEpiWarps * 32) : "memory");
        if (ok) {
            float dy[kOut];
#pragma unroll
            for (int j = 0; j < kOut; ++j) dy[j] = S.dY[row][j];
            bf16* dz = &S.Xc[0][0];
#pragma unroll 1
            for (int j2 = 0; j2 < 2; ++j2) {
                const int c0 = half * 64 + j2 * 32;
                const uint32_t mk = j2 ? m2[1] : m2[0];
                float h[32], v[32];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const uint4 w = *reinterpret_cast<const uint4*>(S.H + core_idx(row, c0 + 8 * k, kRows));
                    const bf16* e = reinterpret_cast<const bf16*>(&w);
#pragma unroll
                    for (int u = 0; u < 8; ++u) h[8 * k + u] = __bfloat162float(e[u]);
                }
                // dW3 = dY^T H2
#pragma unroll
                for (int j = 0; j < kOut; ++j) {
#pragma unroll
                    for (int c = 0; c < 32; ++c) v[c] = dy[j] * h[c];
                    const float s = warp_column_sum(v);
                    atomicAdd(&S.gW3[j * kH + c0 + lane], s);
                }
                // dZ2 = (dY W3) * [Z2 > 0]
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    uint4 w;
                    bf16* o = reinterpret_cast<bf16*>(&w);
#pragma unroll
                    for (int u = 0; u < 8; ++u) {
                        const int c = c0 + 8 * k + u;
                        float d = 0.f;
#pragma unroll
                        for (int j = 0; j < kOut; ++j) d = fmaf(dy[j], S.W3f[j * kH + c], d);
                        o[u] = __float2bfloat16((mk >> (8 * k + u)) & 1u ? d : 0.f);
                        v[8 * k + u] = __bfloat162float(o[u]);
                        if (store) A.dZ2T[(long long)c * A.Mp + grow] = o[u];
                    }
                    *reinterpret_cast<uint4*>(dz + core_idx(row, c0 + 8 * k, kRows)) = w;
                }
                atomicAdd(&S.gb2[c0 + lane], warp_column_sum(v));
            }
            fence_async_shared();
            tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) mbar_arrive(&S.z2);
        }
        if (wait(&S.d4, 0u)) {
            // dZ1 = dH1 * [Z1 > 0]
            tc_fence_after_sync();
#pragma unroll 1
            for (int j = 0; j < 2; ++j) {
                const int c0 = half * 64 + j * 32;
                const uint32_t mk = j ? m1[1] : m1[0];
                float v[32];
                tmem_ld32(tl + (uint32_t)c0, v);
#pragma unroll
                for (int c = 0; c < 32; ++c) {
                    const bf16 o = __float2bfloat16((mk >> c) & 1u ? v[c] : 0.f);
                    v[c] = __bfloat162float(o);
                    if (store) A.dZ1T[(long long)(c0 + c) * A.Mp + grow] = o;
                }
                atomicAdd(&S.gb1[c0 + lane], warp_column_sum(v));
            }
            tc_fence_before_sync();
        }
        asm volatile("bar.sync 2, %0;" ::"n"(kEpiWarps * 32) : "memory");
        if (ok) {
            for (int k = tid; k < kOut * kH; k += kEpiWarps * 32) atomicAdd(&A.gW3[k], S.gW3[k]);
            if (tid < kH) atomicAdd(&A.gb1[tid], S.gb1[tid]);
            else atomicAdd(&A.gb2[tid - kH], S.gb2[tid - kH]);
            if (tid < kOut) atomicAdd(&A.gb3[tid], S.gb3[tid]);
        }
    }
    if (!ok && lane == 0) atomicOr(A.flags, kFlagTimeout);
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    if (warp == 0) tmem_dealloc(tm, kTmemCols);
}

cudaError_t launch_train_rows(const TrainArgs& A, const bf16* X, cudaStream_t s)
{
    CUtensorMap xmap;
    if (!encode_bf16_2d(&xmap, X, kInPad, (unsigned long long)A.M, kInPad * 2, kKc, kRows, true))
        return cudaErrorInvalidValue;
    cudaError_t e = cudaFuncSetAttribute(k_train_rows, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)kTcSmemBytes);
    if (e != cudaSuccess) return e;
    k_train_rows<<<(unsigned)((A.M + kRows - 1) / kRows), kTrainThreads, kTcSmemBytes, s>>>(A, xmap);
    return cudaGetLastError();
}

// --------------------------------------------------------------------------
// Seeding of the queued voxels: features, network, exact seeds
// --------------------------------------------------------------------------

// Cost bucket of a queued voxel whose running squared gamma is g2: 1 + floor(2
// log2 of the table cells with key < gamma) (0 when there are none), the
// bucket k_shell gives.
__device__ __forceinline__ int cost_bucket(const Problem& P, float g2)
{
    return cost_bucket_of(P.bucket_key, sqrtf(g2));
}

// The seed rows of one pair (BATCH = false: P0.seed_list items) or of every
// pair of a batch group (the (pair, item) rows of bd): their number, capped
// at the row buffer, and the pair and queue item of row r.
template <bool BATCH>
struct SeedRows {
    const Problem* P0;
    const BatchDesc* bd;
    __device__ unsigned count() const
    {
        return BATCH ? min(*bd->seed_count, bd->seed_cap) : min(P0->ctr->seed_count, P0->seed_cap);
    }
    __device__ bf16* X() const { return BATCH ? bd->seed_X : P0->seed_X; }
    __device__ float* Y() const { return BATCH ? bd->seed_Y : P0->seed_Y; }
    __device__ const Problem& prob(unsigned r) const { return BATCH ? bd->probs[bd->seed_pair[r]] : *P0; }
    __device__ unsigned item(unsigned r) const { return BATCH ? bd->seed_item[r] : P0->seed_list[r]; }
};

// Features of every seed row into the row buffer, one warp per row.
template <int N, bool BATCH>
__global__ void __launch_bounds__(256) k_seed_features(const __grid_constant__ Problem P0,
                                                       const BatchDesc* __restrict__ bd)
{
    __shared__ float sh_e[8][FeatBox<N>::ELEMS], sh_r[8][FeatBox<N>::ELEMS];
    grid_release();
    grid_wait();
    const SeedRows<BATCH> rows{&P0, bd};
    const unsigned total = rows.count();
    bf16* X = rows.X();
    const int wi = threadIdx.x >> 5;
    const unsigned gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const unsigned nw = (gridDim.x * blockDim.x) >> 5;
    for (unsigned r = gw; r < total; r += nw) {               // warp-uniform
        const Problem& P = rows.prob(r);
        const unsigned v = P.tail_raw[rows.item(r)];
        const float dr = __ldg(P.ref + v);
        const float inv = 1.0f / (P.dd_frac * (P.local ? dr : resolve_dnorm(P)));
        row_features<N>(P, v, dr, inv, sh_e[wi], sh_r[wi], X + (long long)r * kInPad);
    }
}

// Exact seeds from the network's proposals: for every seed row, the faces of
// the 2^N cells around the proposed nearest point (two threads per row), a
// true distance to the evaluation surface, lower the voxel's running squared
// gamma; the voxel moves to the cost bucket of the tighter bound.
template <int N, bool BATCH>
__global__ void __launch_bounds__(256) k_seed_apply(const __grid_constant__ Problem P0,
                                                    const BatchDesc* __restrict__ bd)
{
    grid_release();
    grid_wait();
    const SeedRows<BATCH> rows{&P0, bd};
    const unsigned total = rows.count();
    const float* Y = rows.Y();
    __shared__ unsigned sh_hist[kNumBuckets];
    __shared__ unsigned sh_seed, sh_imp;
    if (threadIdx.x < kNumBuckets) sh_hist[threadIdx.x] = 0;
    if (threadIdx.x == 0) sh_seed = sh_imp = 0;
    __syncthreads();
    // a warp takes 16 rows at a time (two lanes per row), so that every lane
    // of the warp runs the same iterations (the shuffle below)
    const int lane = threadIdx.x & 31, half = lane & 1;
    const unsigned gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const unsigned nw = (gridDim.x * blockDim.x) >> 5;
    for (unsigned rb = gw * 16u; rb < total; rb += nw * 16u) {
        const unsigned r = rb + (unsigned)(lane >> 1);
        const bool live = r < total;
        float sd2 = kInf;
        unsigned v = 0, item = 0;
        const Problem& P = rows.prob(live ? r : 0u);
        if (live) {
            item = rows.item(r);
            v = P.tail_raw[item];
            const int x = (int)(v % (unsigned)P.nx);
            const unsigned r1 = v / (unsigned)P.nx;
            const int y = (int)(r1 % (unsigned)P.ny), z = (int)(r1 / (unsigned)P.ny);
            const float dr = __ldg(P.ref + v);
            const float inv = 1.0f / (P.dd_frac * (P.local ? dr : resolve_dnorm(P)));
            int o[3];
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                const float ov = a < N ? Y[(long long)r * kOut + a] / P.hn[a] : 0.f;
                o[a] = (int)floorf(fminf(fmaxf(ov, -256.f), 256.f));
            }
            constexpr int NCELL = 1 << N;
#pragma unroll 1
            for (int u = half; u < NCELL; u += 2) {
                const int cx = o[0] + (u & 1), cy = o[1] + ((u >> 1) & 1),
                          cz = N == 3 ? o[2] + ((u >> 2) & 1) : 0;
                float q[8];
                uint32_t okc;
                if (!load_cell<N>(P, x, y, z, cx, cy, cz, dr, inv, q, okc)) continue;
                CellGeom<float> gg;
                cell_geom<N, float>(cx, cy, cz, P.mt, gg);
                bool ill = false;
                const float cb = cell_min_d2<N, float>(q, gg, P.mt,
                                                       P.tau > 0.f ? 0.99f * rsqrtf(P.tau) : kInf,
                                                       kInf, ill);
                if (ill) ill = cell_gram_ill<N>(q, okc, P.mt.kappa, P.tau);
                if (!ill) sd2 = fminf(sd2, cb);            // ill-conditioned cells are not used as seeds
            }
        }
        sd2 = fminf(sd2, __shfl_xor_sync(0xffffffffu, sd2, 1));
        if (live && half == 0) {
            const float cur = P.out[v];                     // gamma^2 after the faces through v
            const float nb = fminf(cur, sd2);
            const bool better = nb < cur;
            if (better) P.out[v] = nb;
            const int bucket = cost_bucket(P, nb);
            const int was = P.tail_bucket[item];
            if (BATCH) {
                atomicAdd(&P.ctr->seeded, 1u);
                if (better) atomicAdd(&P.ctr->seed_improved, 1u);
                if (bucket != was) {                        // move the voxel between its pair's bins
                    P.tail_bucket[item] = (unsigned char)bucket;
                    atomicAdd(&P.ctr->hist[bucket], 1u);
                    atomicSub(&P.ctr->hist[was], 1u);
                }
            } else {
                atomicAdd(&sh_seed, 1u);
                if (better) atomicAdd(&sh_imp, 1u);
                if (bucket != was) {
                    P.tail_bucket[item] = (unsigned char)bucket;
                    atomicAdd(&sh_hist[bucket], 1u);
                    atomicSub(&sh_hist[was], 1u);          // wraps; the sum over the block is exact
                }
            }
        }
    }
    if constexpr (!BATCH) {
        __syncthreads();
        if (threadIdx.x < kNumBuckets && sh_hist[threadIdx.x])
            atomicAdd(&P0.ctr->hist[threadIdx.x], sh_hist[threadIdx.x]);
        if (threadIdx.x == 0) {
            if (sh_seed) atomicAdd(&P0.ctr->seeded, sh_seed);
            if (sh_imp) atomicAdd(&P0.ctr->seed_improved, sh_imp);
        }
    }
}

// Queue items of every pair of a batch group past the cost gate, as (pair,
// item) rows (blockIdx.y = pair).
__global__ void __launch_bounds__(256) k_seed_select_batch(const BatchDesc* __restrict__ bd,
                                                           int min_bucket)
{
    grid_release();
    grid_wait();
    const Problem& P = bd->probs[blockIdx.y];
    const unsigned total = min(P.ctr->tail_count, P.tail_cap);
    const int lane = threadIdx.x & 31;
    const unsigned stride = gridDim.x * blockDim.x;
    for (unsigned c0 = blockIdx.x * blockDim.x; c0 < total; c0 += stride) {
        const unsigned i = c0 + threadIdx.x;
        const bool take = i < total && (int)P.tail_bucket[i] >= min_bucket;
        const unsigned m = __ballot_sync(0xffffffffu, take);
        unsigned base = 0;
        if (lane == 0 && m) base = atomicAdd(bd->seed_count, (unsigned)__popc(m));
        base = __shfl_sync(0xffffffffu, base, 0);
        if (take) {
            const unsigned pos = base + __popc(m & ((1u << lane) - 1u));
            if (pos < bd->seed_cap) {                       // rows past the buffer go unseeded
                bd->seed_item[pos] = i;
                bd->seed_pair[pos] = (unsigned short)blockIdx.y;
            }
        }
    }
}

template <int N, bool BATCH>
static cudaError_t launch_seeding_n(const Problem& P, const BatchDesc* bd, const MlpWeights& W,
                                    const bf16* X, float* Y, unsigned cap, const unsigned* count,
                                    unsigned* flags, cudaStream_t s)
{
    const int sms = device_sm_count();
    launch_next(k_seed_features<N, BATCH>, sms * 16, 256, 0, s, P, bd);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    if ((e = launch_mlp_rows(W, X, cap, count, Y, flags, 0, s)) != cudaSuccess) return e;
    launch_next(k_seed_apply<N, BATCH>, sms * 8, 256, 0, s, P, bd);
    return cudaGetLastError();
}

cudaError_t launch_seeding(const Problem& P, const MlpWeights& W, int min_bucket, cudaStream_t s)
{
    if (!P.seed_list || !P.seed_X || !P.seed_Y || P.seed_cap == 0) return cudaErrorInvalidValue;
    launch_next(k_seed_select, device_sm_count() * 4, 256, 0, s, P, min_bucket);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    return P.ndim == 3
               ? launch_seeding_n<3, false>(P, nullptr, W, P.seed_X, P.seed_Y, P.seed_cap,
                                            &P.ctr->seed_count, &P.ctr->flags, s)
               : launch_seeding_n<2, false>(P, nullptr, W, P.seed_X, P.seed_Y, P.seed_cap,
                                            &P.ctr->seed_count, &P.ctr->flags, s);
}

cudaError_t launch_batch_seeding(const BatchGroup& g, const MlpWeights& W, int min_bucket,
                                 cudaStream_t s)
{
    if (g.npairs <= 0 || g.seed_cap == 0) return cudaSuccess;
    const int bx = std::max(1, device_sm_count() * 2 / std::max(1, g.npairs)) + 1;
    launch_next(k_seed_select_batch, dim3(bx, g.npairs), 256, 0, s, g.desc, min_bucket);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    Problem dummy{};
    return g.ndim == 3 ? launch_seeding_n<3, true>(dummy, g.desc, W, g.seed_X, g.seed_Y, g.seed_cap,
                                                   g.seed_count, g.flags, s)
                       : launch_seeding_n<2, true>(dummy, g.desc, W, g.seed_X, g.seed_Y, g.seed_cap,
                                                   g.seed_count, g.flags, s);
}

cudaError_t launch_features(const Problem& P, const unsigned* vox, long long n, bf16* X,
                            cudaStream_t s)
{
    const int grid = (int)std::min<long long>((n + 7) / 8, (long long)device_sm_count() * 16);
    if (P.ndim == 3) k_features<3><<<std::max(grid, 1), 256, 0, s>>>(P, vox, n, X);
    else k_features<2><<<std::max(grid, 1), 256, 0, s>>>(P, vox, n, X);
    return cudaGetLastError();
}

cudaError_t launch_labels(const Problem& P, const float* gmap, const unsigned* vox, long long n,
                          float* T, cudaStream_t s)
{
    const int grid = (int)std::min<long long>((n + 3) / 4, (long long)device_sm_count() * 16);
    if (P.ndim == 3) k_labels<3><<<std::max(grid, 1), 128, 0, s>>>(P, gmap, vox, n, T);
    else k_labels<2><<<std::max(grid, 1), 128, 0, s>>>(P, gmap, vox, n, T);
    return cudaGetLastError();
}

}  // namespace gk

// ==========================================================================
// Model object and its C ABI
// ==========================================================================

using gk::bf16;

struct gamma_model_s {
    int device = 0;
    float* p = nullptr;           // fp32 master parameters (layout below)
    float* gr = nullptr;          // gradients
    float* m1 = nullptr;          // Adam first moment
    float* m2 = nullptr;          // Adam second moment
    unsigned char* mask = nullptr;  // 1 for trainable entries (padding stays zero)
    bf16 *W1h = nullptr, *W2h = nullptr, *W2Th = nullptr, *W3h = nullptr;
    long long step = 0;
    unsigned long long seed = 0;
    // training workspace: X, H1, dZ1 and dZ2 of a batch transposed (the
    // operands of the weight-gradient product), row stride wsMp = wsM rounded
    // up to 8 (16-byte rows for TMA)
    long long wsM = 0, wsMp = 0;
    bf16 *XT = nullptr, *H1T = nullptr, *dZ1T = nullptr, *dZ2T = nullptr;
    gk::WgradMaps maps{};         // their tensor maps for batches of mapsM rows
    long long mapsM = 0;
    float* loss = nullptr;        // behind the gradients (gr), and dflags behind it: one reset, one read
    unsigned* dflags = nullptr;   // error flags of the training kernels
    unsigned* hflags = nullptr;   // ... of gamma_model_infer: page-locked, mapped host memory
    unsigned* hflags_dev = nullptr;   // its device address
};

namespace {

// Parameter layout (floats): W1 [128][384], b1 [128], W2 [128][128], b2 [128],
// W3 [8][128], b3 [8].
constexpr long long kOffW1 = 0;
constexpr long long kOffB1 = kOffW1 + gk::kH * gk::kInPad;
constexpr long long kOffW2 = kOffB1 + gk::kH;
constexpr long long kOffB2 = kOffW2 + gk::kH * gk::kH;
constexpr long long kOffW3 = kOffB2 + gk::kH;
constexpr long long kOffB3 = kOffW3 + gk::kOutPad * gk::kH;
constexpr long long kNParams = kOffB3 + gk::kOutPad;

int cuda_rc(cudaError_t e) { return e == cudaSuccess ? GAMMA_OK : (e == cudaErrorMemoryAllocation ? GAMMA_ERR_OOM : GAMMA_ERR_CUDA); }

#define MCK(call)                                  \
    do {                                           \
        int rc_ = cuda_rc(call);                   \
        if (rc_) return rc_;                       \
    } while (0)

void free_ws(gamma_model_s* m)
{
    cudaFree(m->XT);               // one allocation
    m->XT = m->H1T = m->dZ1T = m->dZ2T = nullptr;
    m->wsM = m->wsMp = m->mapsM = 0;
}

int ensure_ws(gamma_model_s* m, long long M)
{
    const long long Mp = (M + 7) / 8 * 8;
    if (M > m->wsM) {
        free_ws(m);
        MCK(cudaMalloc(&m->XT, sizeof(bf16) * (size_t)Mp * (gk::kInPad + 3 * gk::kH)));
        m->H1T = m->XT + Mp * gk::kInPad;
        m->dZ1T = m->H1T + Mp * gk::kH;
        m->dZ2T = m->dZ1T + Mp * gk::kH;
        m->wsM = M;
        m->wsMp = Mp;
    }
    if (m->mapsM != M) {
        m->mapsM = 0;
        if (!gk::encode_wgrad_maps(&m->maps, m->dZ1T, m->XT, m->dZ2T, m->H1T, M, m->wsMp)) return GAMMA_ERR_CUDA;
        m->mapsM = M;
    }
    return GAMMA_OK;
}

// Host-side parameter initialisation: He-normal weights from a splitmix64 /
// Box-Muller stream, zero biases and padding.
void init_params(std::vector<float>& h, unsigned long long seed)
{
    h.assign(kNParams, 0.f);
    unsigned long long st = seed ? seed : 0x9e3779b97f4a7c15ull;
    auto next = [&]() {
        st += 0x9e3779b97f4a7c15ull;
        unsigned long long z = st;
        z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
        z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
        return z ^ (z >> 31);
    };
    auto unif = [&]() { return ((next() >> 11) + 0.5) * (1.0 / 9007199254740992.0); };
    auto normal = [&]() { return std::sqrt(-2.0 * std::log(unif())) * std::cos(6.283185307179586 * unif()); };
    for (int r = 0; r < gk::kH; ++r)
        for (int c = 0; c < gk::kIn; ++c) h[kOffW1 + r * gk::kInPad + c] = (float)(normal() * std::sqrt(2.0 / gk::kIn));
    for (int i = 0; i < gk::kH * gk::kH; ++i) h[kOffW2 + i] = (float)(normal() * std::sqrt(2.0 / gk::kH));
    for (int r = 0; r < gk::kOut; ++r)
        for (int c = 0; c < gk::kH; ++c) h[kOffW3 + r * gk::kH + c] = (float)(normal() * std::sqrt(1.0 / gk::kH));
}

std::vector<unsigned char> param_mask()
{
    std::vector<unsigned char> k(kNParams, 1);
    for (int r = 0; r < gk::kH; ++r)
        for (int c = gk::kIn; c < gk::kInPad; ++c) k[kOffW1 + r * gk::kInPad + c] = 0;
    for (int r = gk::kOut; r < gk::kOutPad; ++r)
        for (int c = 0; c < gk::kH; ++c) k[kOffW3 + r * gk::kH + c] = 0;
    for (int r = gk::kOut; r < gk::kOutPad; ++r) k[kOffB3 + r] = 0;
    return k;
}

gk::WeightCopies weight_copies(const gamma_model_s* m)
{
    return gk::WeightCopies{m->W1h, m->W2h, m->W2Th, m->W3h, (int)kOffW2, (int)kOffW3};
}

int refresh_bf16(gamma_model_s* m, cudaStream_t s)
{
    gk::k_cast_weights<<<(int)(kNParams + 255) / 256, 256, 0, s>>>((int)kNParams, m->p, weight_copies(m));
    return cuda_rc(cudaGetLastError());
}

// Loss and gradients of a minibatch into m->gr (zeroed first, with the loss and
// the flags behind it): the rows' passes in one kernel, then both weight
// gradients in one product with the batch as K, split over several blocks per
// tile that add into them.
int backward_train(gamma_model_s* m, const bf16* X, const float* T, long long M, cudaStream_t s)
{
    MCK(cudaMemsetAsync(m->gr, 0, sizeof(float) * kNParams + 2 * sizeof(unsigned), s));
    gk::TrainArgs A{};
    gk::model_weights(m, &A.W);
    A.W2T = m->W2Th;
    A.W3f = m->p + kOffW3;
    A.T = T;
    A.M = M;
    A.Mp = m->wsMp;
    A.inv_count = 1.f / (float)M;
    A.XT = m->XT;
    A.H1T = m->H1T;
    A.dZ1T = m->dZ1T;
    A.dZ2T = m->dZ2T;
    A.gb1 = m->gr + kOffB1;
    A.gb2 = m->gr + kOffB2;
    A.gW3 = m->gr + kOffW3;
    A.gb3 = m->gr + kOffB3;
    A.loss = m->loss;
    A.flags = m->dflags;
    MCK(gk::launch_train_rows(A, X, s));
    MCK(gk::launch_wgrad(m->maps, M, m->gr + kOffW1, m->gr + kOffW2, m->dflags, s));
    return GAMMA_OK;
}

// Loss (optional) of the last backward pass: synchronises.
int read_loss(gamma_model_s* m, float* loss_out, cudaStream_t s)
{
    if (!loss_out) return GAMMA_OK;
    unsigned w[2];                                 // loss, flags
    MCK(cudaMemcpyAsync(w, m->loss, sizeof(w), cudaMemcpyDeviceToHost, s));
    MCK(cudaStreamSynchronize(s));
    std::memcpy(loss_out, &w[0], sizeof(float));
    return (w[1] & gk::kFlagTimeout) ? GAMMA_ERR_TIMEOUT : GAMMA_OK;
}

}  // namespace

namespace gk {

bool model_weights(const gamma_model_s* m, MlpWeights* w)
{
    if (!m) return false;
    w->W1 = m->W1h;
    w->W2 = m->W2h;
    w->W3 = m->W3h;
    w->b1 = m->p + kOffB1;
    w->b2 = m->p + kOffB2;
    w->b3 = m->p + kOffB3;
    return true;
}

}  // namespace gk

extern "C" {

int gamma_model_create(gamma_model* out, uint64_t seed)
{
    if (!out) return GAMMA_ERR_INVALID_ARG;
    *out = nullptr;
    gamma_model_s* m = new (std::nothrow) gamma_model_s();
    if (!m) return GAMMA_ERR_OOM;
    auto fail = [&](int rc) { gamma_model_destroy(m); return rc; };
    if (cudaGetDevice(&m->device) != cudaSuccess) return fail(GAMMA_ERR_CUDA);
    int rc;
    if ((rc = cuda_rc(cudaMalloc(&m->p, sizeof(float) * kNParams)))) return fail(rc);
    if ((rc = cuda_rc(cudaMalloc(&m->gr, sizeof(float) * kNParams + 2 * sizeof(unsigned))))) return fail(rc);
    m->loss = m->gr + kNParams;
    m->dflags = reinterpret_cast<unsigned*>(m->loss + 1);
    if ((rc = cuda_rc(cudaMemset(m->gr, 0, sizeof(float) * kNParams + 2 * sizeof(unsigned))))) return fail(rc);
    if ((rc = cuda_rc(cudaMalloc(&m->m1, sizeof(float) * kNParams)))) return fail(rc);
    if ((rc = cuda_rc(cudaMalloc(&m->m2, sizeof(float) * kNParams)))) return fail(rc);
    if ((rc = cuda_rc(cudaMalloc(&m->mask, kNParams)))) return fail(rc);
    if ((rc = cuda_rc(cudaMalloc(&m->W1h, sizeof(bf16) * gk::kH * gk::kInPad)))) return fail(rc);
    if ((rc = cuda_rc(cudaMalloc(&m->W2h, sizeof(bf16) * gk::kH * gk::kH)))) return fail(rc);
    if ((rc = cuda_rc(cudaMalloc(&m->W2Th, sizeof(bf16) * gk::kH * gk::kH)))) return fail(rc);
    if ((rc = cuda_rc(cudaMalloc(&m->W3h, sizeof(bf16) * gk::kOutPad * gk::kH)))) return fail(rc);
    if ((rc = cuda_rc(cudaHostAlloc(&m->hflags, sizeof(unsigned), cudaHostAllocMapped)))) return fail(rc);
    if ((rc = cuda_rc(cudaHostGetDevicePointer((void**)&m->hflags_dev, m->hflags, 0)))) return fail(rc);
    std::vector<float> h;
    init_params(h, seed);
    m->seed = seed;
    const std::vector<unsigned char> k = param_mask();
    if ((rc = cuda_rc(cudaMemcpy(m->p, h.data(), sizeof(float) * kNParams, cudaMemcpyHostToDevice)))) return fail(rc);
    if ((rc = cuda_rc(cudaMemcpy(m->mask, k.data(), kNParams, cudaMemcpyHostToDevice)))) return fail(rc);
    if ((rc = cuda_rc(cudaMemset(m->m1, 0, sizeof(float) * kNParams)))) return fail(rc);
    if ((rc = cuda_rc(cudaMemset(m->m2, 0, sizeof(float) * kNParams)))) return fail(rc);
    if ((rc = refresh_bf16(m, 0))) return fail(rc);
    if ((rc = cuda_rc(cudaDeviceSynchronize()))) return fail(rc);
    *out = m;
    return GAMMA_OK;
}

void gamma_model_destroy(gamma_model m)
{
    if (!m) return;
    cudaFree(m->p); cudaFree(m->gr); cudaFree(m->m1); cudaFree(m->m2); cudaFree(m->mask);
    cudaFree(m->W1h); cudaFree(m->W2h); cudaFree(m->W2Th); cudaFree(m->W3h);
    if (m->hflags) cudaFreeHost(m->hflags);
    free_ws(m);
    delete m;
}

int64_t gamma_model_num_params(void) { return kNParams; }

int gamma_model_get_params(gamma_model m, float* host, int64_t n, int which)
{
    if (!m || !host || n != kNParams || which < 0 || which > 3) return GAMMA_ERR_INVALID_ARG;
    const float* src = which == 0 ? m->p : which == 1 ? m->gr : which == 2 ? m->m1 : m->m2;
    MCK(cudaDeviceSynchronize());
    MCK(cudaMemcpy(host, src, sizeof(float) * kNParams, cudaMemcpyDeviceToHost));
    return GAMMA_OK;
}

int gamma_model_set_params(gamma_model m, const float* host, int64_t n)
{
    if (!m || !host || n != kNParams) return GAMMA_ERR_INVALID_ARG;
    MCK(cudaMemcpy(m->p, host, sizeof(float) * kNParams, cudaMemcpyHostToDevice));
    if (int rc = refresh_bf16(m, 0)) return rc;
    MCK(cudaDeviceSynchronize());
    return GAMMA_OK;
}

int gamma_model_forward(gamma_model m, const void* X_bf16_dev, int64_t M, float* Y_dev,
                        void* cuda_stream)
{
    if (!m || !X_bf16_dev || !Y_dev || M <= 0) return GAMMA_ERR_INVALID_ARG;
    cudaStream_t s = (cudaStream_t)cuda_stream;
    if (reinterpret_cast<uintptr_t>(X_bf16_dev) % 16 != 0) return GAMMA_ERR_INVALID_ARG;
    gk::MlpWeights W;
    gk::model_weights(m, &W);
    MCK(gk::launch_mlp_rows(W, (const bf16*)X_bf16_dev, M, nullptr, Y_dev, m->dflags, 0, s));
    return GAMMA_OK;
}

int gamma_model_infer(gamma_model m, const void* X_bf16_dev, int64_t M, float* Y_dev,
                      void* cuda_stream)
{
    if (!m || !X_bf16_dev || !Y_dev || M <= 0) return GAMMA_ERR_INVALID_ARG;
    if (reinterpret_cast<uintptr_t>(X_bf16_dev) % 16 != 0) return GAMMA_ERR_INVALID_ARG;
    cudaStream_t s = (cudaStream_t)cuda_stream;
    gk::MlpWeights W;
    gk::model_weights(m, &W);
    // the kernel reports a timeout in mapped host memory: no reset or copy
    // around it (the call ends with the stream's synchronisation anyway)
    volatile unsigned* flag = m->hflags;
    *flag = 0;
    MCK(gk::launch_mlp_infer(W, (const bf16*)X_bf16_dev, M, Y_dev, m->hflags_dev, s));
    MCK(cudaStreamSynchronize(s));
    return (*flag & gk::kFlagTimeout) ? GAMMA_ERR_TIMEOUT : GAMMA_OK;
}

int gamma_model_backward(gamma_model m, const void* X_bf16_dev, const float* T_dev, int64_t M,
                         float* loss_out, void* cuda_stream)
{
    if (!m || !X_bf16_dev || !T_dev || M <= 0) return GAMMA_ERR_INVALID_ARG;
    cudaStream_t s = (cudaStream_t)cuda_stream;
    if (reinterpret_cast<uintptr_t>(X_bf16_dev) % 16 != 0) return GAMMA_ERR_INVALID_ARG;
    if (int rc = ensure_ws(m, M)) return rc;
    if (int rc = backward_train(m, (const bf16*)X_bf16_dev, T_dev, M, s)) return rc;
    return read_loss(m, loss_out, s);
}

int gamma_model_train_step(gamma_model m, const void* X_bf16_dev, const float* T_dev, int64_t M,
                           float lr, float* loss_out, void* cuda_stream)
{
    if (!m || !(lr >= 0.f)) return GAMMA_ERR_INVALID_ARG;
    cudaStream_t s = (cudaStream_t)cuda_stream;
    if (int rc = gamma_model_backward(m, X_bf16_dev, T_dev, M, nullptr, cuda_stream)) return rc;
    m->step += 1;
    const float b1 = 0.9f, b2 = 0.999f;
    const float c1 = 1.f - std::pow(b1, (float)m->step), c2 = 1.f - std::pow(b2, (float)m->step);
    gk::k_adam<<<(int)(kNParams + 255) / 256, 256, 0, s>>>((int)kNParams, m->p, m->gr, m->m1, m->m2, m->mask,
                                                           weight_copies(m), lr, b1, b2, 1e-8f, c1, c2);
    MCK(cudaGetLastError());
    return read_loss(m, loss_out, s);
}

// File format: 8-byte magic "GAMMAMLP", int32 version 1, int32 kIn, kInPad,
// kH, kOut, kOutPad, int64 Adam step, uint64 seed, then kNParams floats each of
// parameters, Adam first and second moments (little-endian).
int gamma_model_save(gamma_model m, const char* path)
{
    if (!m || !path) return GAMMA_ERR_INVALID_ARG;
    std::vector<float> p(kNParams), a(kNParams), b(kNParams);
    if (int rc = gamma_model_get_params(m, p.data(), kNParams, 0)) return rc;
    if (int rc = gamma_model_get_params(m, a.data(), kNParams, 2)) return rc;
    if (int rc = gamma_model_get_params(m, b.data(), kNParams, 3)) return rc;
    FILE* f = std::fopen(path, "wb");
    if (!f) return GAMMA_ERR_INVALID_ARG;
    const int32_t hdr[7] = {1, gk::kIn, gk::kInPad, gk::kH, gk::kOut, gk::kOutPad, 0};
    const int64_t step = m->step;
    const uint64_t seed = m->seed;
    bool ok = std::fwrite("GAMMAMLP", 1, 8, f) == 8 && std::fwrite(hdr, 4, 6, f) == 6 &&
              std::fwrite(&step, 8, 1, f) == 1 && std::fwrite(&seed, 8, 1, f) == 1 &&
              std::fwrite(p.data(), 4, kNParams, f) == (size_t)kNParams &&
              std::fwrite(a.data(), 4, kNParams, f) == (size_t)kNParams &&
              std::fwrite(b.data(), 4, kNParams, f) == (size_t)kNParams;
    ok = (std::fclose(f) == 0) && ok;
    return ok ? GAMMA_OK : GAMMA_ERR_INVALID_ARG;
}

int gamma_model_load(gamma_model m, const char* path)
{
    if (!m || !path) return GAMMA_ERR_INVALID_ARG;
    FILE* f = std::fopen(path, "rb");
    if (!f) return GAMMA_ERR_MODEL;
    char magic[8];
    int32_t hdr[6];
    int64_t step = 0;
    uint64_t seed = 0;
    std::vector<float> p(kNParams), a(kNParams), b(kNParams);
    bool ok = std::fread(magic, 1, 8, f) == 8 && std::memcmp(magic, "GAMMAMLP", 8) == 0 &&
              std::fread(hdr, 4, 6, f) == 6 && hdr[0] == 1 && hdr[1] == gk::kIn &&
              hdr[2] == gk::kInPad && hdr[3] == gk::kH && hdr[4] == gk::kOut &&
              hdr[5] == gk::kOutPad && std::fread(&step, 8, 1, f) == 1 &&
              std::fread(&seed, 8, 1, f) == 1 &&
              std::fread(p.data(), 4, kNParams, f) == (size_t)kNParams &&
              std::fread(a.data(), 4, kNParams, f) == (size_t)kNParams &&
              std::fread(b.data(), 4, kNParams, f) == (size_t)kNParams;
    std::fclose(f);
    if (!ok) return GAMMA_ERR_MODEL;
    for (float x : p)
        if (!std::isfinite(x)) return GAMMA_ERR_MODEL;
    MCK(cudaMemcpy(m->p, p.data(), sizeof(float) * kNParams, cudaMemcpyHostToDevice));
    MCK(cudaMemcpy(m->m1, a.data(), sizeof(float) * kNParams, cudaMemcpyHostToDevice));
    MCK(cudaMemcpy(m->m2, b.data(), sizeof(float) * kNParams, cudaMemcpyHostToDevice));
    m->step = step;
    m->seed = seed;
    if (int rc = refresh_bf16(m, 0)) return rc;
    MCK(cudaDeviceSynchronize());
    return GAMMA_OK;
}

}  // extern "C"
