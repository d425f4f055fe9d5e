// CUDA kernels of the gamma search (sm_103a).
//
// One run over a dose pair is six stream-ordered launches:
//   k_prepare     max of the reference dose (the global dose norm) and its
//                 finite check (the shell checks the evaluation dose, every
//                 value of which is the centre of one tile voxel)  (Algorithm
//                 A2 step 2)
//   k_shell_w     per reference voxel: criteria, low-dose cutoff, gamma0 =
//                 DD/dD (A1 step 4a) and every face through the voxel's node
//                 (reduced closed form), from a TMA-staged tile; voxels whose
//                 running gamma still exceeds the distance to any other face
//                 are queued with a cost bucket
//   k_plane_seed  a tight bound for every queued voxel from one cell near its
//                 nearest surface point
//   k_scatter     order the queue by estimated cost, most expensive first (the
//                 role the paper's DD sort plays, Section 2.2 and Table 2)
//   k_tail_cq     persistent: warps walk the sorted cell table for batches of
//                 queued voxels with the exact early exit of A1 step 4b-ii
//                 (key >= gamma), the dose gap and a plane bound, and evaluate
//                 what is left 32 cells at a time
//   k_tail_fix    the voxels with a near-singular cell or past a cut table
// The other walks (options walk = 0, 1, 2) take k_tail, k_walk or k_walk_rows
// in place of the seeds and the last two.
// No kernel waits on another block or allocates memory.
#include <cuda.h>
#include <cuda_runtime.h>
#include <math.h>

#include <algorithm>
#include <cstring>

#include "gamma_cell.cuh"
#include "gamma_internal.h"
#include "gamma_launch.cuh"
#include "gamma_near.cuh"
#include "gamma_plane.cuh"
#include "gamma_tma.cuh"

namespace gk {

// --------------------------------------------------------------------------
// k_prepare: dose norm and finite check
// --------------------------------------------------------------------------

// part: bit 0 = maximum and finite check of the reference dose, bit 1 =
// finite check of the evaluation dose (a part left out reads as zeros).
template <bool BATCH>
__global__ void __launch_bounds__(256)
    k_prepare(const __grid_constant__ Problem P0, const BatchDesc* __restrict__ bd, int part)
{
    grid_release();
    grid_wait();
    const Problem& P = BATCH ? bd->probs[blockIdx.y] : P0;
    if constexpr (BATCH) {
        if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) {
            *bd->shell_next = 0u;
            if (bd->seed_count) {
                *bd->seed_count = 0u;
                *bd->seed_head = 0u;
            }
        }
    }
    float m = -kInf;
    bool bad = false;
    const long long stride = (long long)gridDim.x * blockDim.x;
    const long long first = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const float* ref = (part & 1) ? P.ref : nullptr;
    const float* ev = (part & 2) ? P.ev : nullptr;
    long long done = 0;
    if ((((uintptr_t)P.ref | (uintptr_t)P.ev) & 15u) == 0) {      // 16-byte vector reads
        const long long n4 = P.nvox / 4;
        const float4 zero4 = make_float4(0.f, 0.f, 0.f, 0.f);
        const float4* r4p = (const float4*)ref;
        const float4* e4p = (const float4*)ev;
        auto r4 = [&](long long i) { return r4p ? __ldg(r4p + i) : zero4; };
        auto e4 = [&](long long i) { return e4p ? __ldg(e4p + i) : zero4; };
        auto take = [&](const float4 r, const float4 e) {
            bad |= !(isfinite(r.x) && isfinite(r.y) && isfinite(r.z) && isfinite(r.w) &&
                     isfinite(e.x) && isfinite(e.y) && isfinite(e.z) && isfinite(e.w));
            m = fmaxf(m, fmaxf(fmaxf(r.x, r.y), fmaxf(r.z, r.w)));
        };
        long long i = first;
        for (; i + stride < n4; i += 2 * stride) {          // four 16-byte reads in flight
            const float4 ra = r4(i), ea = e4(i);
            const float4 rb = r4(i + stride), eb = e4(i + stride);
            take(ra, ea);
            take(rb, eb);
        }
        if (i < n4) take(r4(i), e4(i));
        done = n4 * 4;
    }
    for (long long i = done + first; i < P.nvox; i += stride) {
        const float r = ref ? __ldg(ref + i) : 0.f, e = ev ? __ldg(ev + i) : 0.f;
        bad |= !(isfinite(r) && isfinite(e));
        m = fmaxf(m, r);
    }
    // one atomic per block: same-address atomics serialise in L2
    __shared__ float sh_m[8];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(kFull, m, o));
    if ((threadIdx.x & 31) == 0) sh_m[threadIdx.x >> 5] = m;
    bad = __syncthreads_or(bad);
    if (threadIdx.x == 0) {
        for (int w = 1; w < (int)(blockDim.x >> 5); ++w) m = fmaxf(m, sh_m[w]);
        if (part & 1) atomicMax(&P.ctr->dnorm_enc, fenc(m));
        if (bad) atomicOr(&P.ctr->flags, kFlagNonFinite);
    }
}

// --------------------------------------------------------------------------
// k_shell: gamma0 and the key-0 cells, one block per tile of voxels
// --------------------------------------------------------------------------

// Tile of voxels per block (x fastest; a warp is one x row) and its halo box
// in shared memory.  The box starts 4 voxels left of the tile so that the TMA
// x coordinate stays a multiple of 4 floats (16 bytes).
template <int N>
struct ShellTile {
    static constexpr int TX = 32, TY = N == 3 ? 4 : 8, TZ = N == 3 ? 2 : 1;
    static constexpr int BX = 40, BY = TY + 2, BZ = N == 3 ? TZ + 2 : 1;
    static constexpr int ELEMS = BX * BY * BZ;
    // each staging buffer starts on a 128-byte boundary (TMA destination rule)
    static constexpr int STRIDE = (ELEMS + 31) / 32 * 32;
    static_assert(STRIDE * 4 % 128 == 0, "TMA destination must stay 128-byte aligned");
};

template <int N, int MINB, bool BATCH>
__global__ void __launch_bounds__(256, MINB)
    k_shell(const __grid_constant__ Problem P0, const __grid_constant__ CUtensorMap tmap0,
            int use_tma0, int t_first, int ntiles, unsigned* tile_next,
            const __grid_constant__ SlabGate gate, const BatchDesc* __restrict__ bd)
{
    using T = ShellTile<N>;
    __shared__ __align__(128) float tile[2][T::STRIDE];
    __shared__ __align__(8) uint64_t bar[2];
    __shared__ unsigned int sh_hist[kNumBuckets];
    __shared__ unsigned long long sh_eval, sh_pass;
    __shared__ unsigned int sh_rmax;
    __shared__ __align__(16) Problem sh_P;     // the current pair (batched launches)
    __shared__ int sh_next[2];                 // the block's next tile, per staging buffer
    __shared__ unsigned sh_tb[2];              // 1 + largest cost bucket queued in the tile (0: none)

    const int lane = threadIdx.x & 31;
    const int lx = lane, ly = (threadIdx.x >> 5) % T::TY, lz = (threadIdx.x >> 5) / T::TY;

    if (threadIdx.x < kNumBuckets) sh_hist[threadIdx.x] = 0;
    if (threadIdx.x == 0) {
        sh_eval = 0;
        sh_pass = 0;
        sh_rmax = 0;
        sh_tb[0] = sh_tb[1] = 0;
        mbar_init(&bar[0], 1);
        mbar_init(&bar[1], 1);
        mbar_fence_init();
    }
    __syncthreads();

    // global tile -> (pair, tile of that pair)
    auto locate = [&](int t, int& pr, int& lt) {
        if constexpr (!BATCH) {
            pr = 0;
            lt = t;
        } else {
            int lo = 0, hi = bd->npairs - 1;
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if (bd->tile_start[mid] <= t) lo = mid; else hi = mid - 1;
            }
            pr = lo;
            lt = t - bd->tile_start[lo];
        }
    };
    auto pair_tma = [&](int pr) { return BATCH ? bd->use_tma[pr] : use_tma0; };
    auto tile_origin = [&](int nx, int ny, int lt, int& x0, int& y0, int& z0) {
        const int ntx = (nx + T::TX - 1) / T::TX, nty = (ny + T::TY - 1) / T::TY;
        x0 = (lt % ntx) * T::TX;
        y0 = ((lt / ntx) % nty) * T::TY;
        z0 = (lt / ntx / nty) * T::TZ;
    };
    bool gate_failed = false;            // thread 0: a slab wait gave up
    auto issue = [&](int t, int b) {
        if (t >= ntiles) return;
        int pr, lt;
        locate(t, pr, lt);
        if (!pair_tma(pr)) return;
        const Problem& Q = BATCH ? bd->probs[pr] : P0;
        const CUtensorMap* map = BATCH ? &bd->maps[pr] : &tmap0;
        int x0, y0, z0;
        tile_origin(Q.nx, Q.ny, lt, x0, y0, z0);
        if (!BATCH && gate.flag && !gate_failed) {
            // the box reads slices z0 - 1 .. z0 + TZ, from at most two slabs
            const int zlo = max(z0 - 1, 0), zhi = min(z0 + T::TZ, Q.nz - 1);
            if (!flag_wait_bounded(gate.flag + zlo / gate.depth, gate.epoch) ||
                !flag_wait_bounded(gate.flag + zhi / gate.depth, gate.epoch)) {
                atomicOr(&Q.ctr->flags, kFlagTimeout);     // the run reports a timeout
                gate_failed = true;                        // and this block waits no more
            }
            fence_async_global();
        }
        mbar_arrive_expect_tx(&bar[b], T::ELEMS * (uint32_t)sizeof(float));
        if (N == 3) tma_load_3d(tile[b], map, x0 - 4, y0 - 1, z0 - 1, &bar[b]);
        else tma_load_2d(tile[b], map, x0 - 4, y0 - 1, &bar[b]);
    };
    if (threadIdx.x == 0) issue(t_first + blockIdx.x, 0);
    uint32_t parity = 0;                 // bit b: phase of bar[b] to wait for
    unsigned my_eval = 0, my_pass = 0;
    float my_rmax = 0.f;
    bool bad_ev = false;                 // a non-finite evaluation dose was seen
    int buf = 0;
    int cur = -1;                        // pair whose counters my_* accumulate

    // per-block counters -> the pair's global counters
    auto flush = [&](const Problem& Q) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            my_eval += __shfl_xor_sync(kFull, my_eval, o);
            my_pass += __shfl_xor_sync(kFull, my_pass, o);
            my_rmax = fmaxf(my_rmax, __shfl_xor_sync(kFull, my_rmax, o));
        }
        if (__any_sync(kFull, bad_ev) && lane == 0) atomicOr(&Q.ctr->flags, kFlagNonFinite);
        bad_ev = false;
        if (lane == 0) {
            if (my_eval) atomicAdd(&sh_eval, (unsigned long long)my_eval);
            if (my_pass) atomicAdd(&sh_pass, (unsigned long long)my_pass);
            atomicMax(&sh_rmax, fenc(my_rmax));
        }
        my_eval = my_pass = 0;
        my_rmax = 0.f;
        __syncthreads();
        if (threadIdx.x < kNumBuckets && sh_hist[threadIdx.x]) {
            atomicAdd(&Q.ctr->hist[threadIdx.x], sh_hist[threadIdx.x]);
            sh_hist[threadIdx.x] = 0;
        }
        if (threadIdx.x == 0) {
            if (sh_eval) atomicAdd(&Q.ctr->n_eval, sh_eval);
            if (sh_pass) atomicAdd(&Q.ctr->n_pass, sh_pass);
            atomicMax(&Q.ctr->rmax_enc, sh_rmax);
            sh_eval = 0;
            sh_pass = 0;
            sh_rmax = 0;
        }
        __syncthreads();
    };

    // Tiles after the first come from a work counter when one is given (the
    // block that finishes first takes the next tile), else in grid stride.
    for (int t = t_first + blockIdx.x; t < ntiles; buf ^= 1) {
        int pr, lt;
        locate(t, pr, lt);
        if constexpr (BATCH) {
            if (pr != cur) {                       // block-uniform
                if (cur >= 0) flush(sh_P);
                const int* src = (const int*)&bd->probs[pr];
                int* dst = (int*)&sh_P;
                for (int i = threadIdx.x; i < (int)(sizeof(Problem) / 4); i += blockDim.x)
                    dst[i] = src[i];
                __syncthreads();
                cur = pr;
            }
        }
        const Problem& P = BATCH ? sh_P : P0;
        const bool use_tma = pair_tma(pr) != 0;
        const float dnorm = resolve_dnorm(P);
        const float thr = cutoff_threshold(P.local, P.cutoff_frac, dnorm);
        // every face not through the voxel is at spatial distance >= the
        // first table key, or >= the cover radius when the table was cut
        const float k0 = P.ntable > 0 ? P.table[0].key : kInf;
        const float qlim = fminf(k0 * k0, P.r_cover * P.r_cover);
        int x0, y0, z0;
        tile_origin(P.nx, P.ny, lt, x0, y0, z0);
        float* tl = tile[buf];
        // ---- stage: prefetch the next tile, wait for this one ----
        // Every thread waits on the tile's mbarrier itself; a wait that gives
        // up is reported at the end-of-tile barrier, where the block leaves
        // together (the smem reads in between stay in bounds).
        if (threadIdx.x == 0) {
            const int nt = tile_next ? t_first + (int)gridDim.x + (int)atomicAdd(tile_next, 1u)
                                     : t + (int)gridDim.x;
            sh_next[buf] = nt;                 // read by every thread after this tile's barrier
            issue(nt, buf ^ 1);
        }
        bool timed_out = false;
        if (use_tma) {
            timed_out = !mbar_wait_bounded(&bar[buf], (parity >> buf) & 1u);
            parity ^= 1u << buf;
        } else {
            for (int i = threadIdx.x; i < T::ELEMS; i += blockDim.x) {
                const int bx = i % T::BX, by = (i / T::BX) % T::BY, bz = i / (T::BX * T::BY);
                const int gx = x0 - 4 + bx, gy = y0 - 1 + by, gz = (N == 3 ? z0 - 1 : 0) + bz;
                const bool in = (unsigned)gx < (unsigned)P.nx && (unsigned)gy < (unsigned)P.ny &&
                                (N == 2 || (unsigned)gz < (unsigned)P.nz);
                tl[i] = in ? __ldg(P.ev + ((long long)gz * P.ny + gy) * P.nx + gx) : kNaN;
            }
            __syncthreads();
        }

        // ---- gamma0 and the faces that contain the voxel ----
        const int x = x0 + lx, y = y0 + ly, z = z0 + lz;
        const bool inside = x < P.nx && y < P.ny && z < P.nz;
        const long long v = inside ? ((long long)z * P.ny + y) * P.nx + x : 0;
        const int tix0 = ((N == 3 ? lz + 1 : 0) * T::BY + (ly + 1)) * T::BX + (lx + 4);
        float dr = 0.f, best = 0.f;
        bool act = false;
        if (inside) {
            dr = __ldg(P.ref + v);
            act = is_evaluated(P, dr, thr);
            if (!act) P.out[v] = __int_as_float(0x7fc00000);
            bad_ev |= !isfinite(tl[tix0]);           // every evaluation dose is some tile's centre
        }
        const int tix = tix0;
        if (act) {
            const float dD = P.dd_frac * (P.local ? dr : dnorm);
            const float q0 = (tl[tix] - dr) / dD;
            best = q0 * q0;
            my_rmax = fmaxf(my_rmax, fabsf(q0));
            if (best > 0.f) best = near_gamma2<N, T::BX, T::BX * T::BY>(tl, tix, dr, dD, P.mt.kappa);
        }

        // ---- finish or queue ----
        bool tail = false;
        int bucket = 0;
        if (act) {
            tail = best > qlim;
            if (tail) {
                P.out[v] = best;                       // gamma^2, finished by k_tail
                // 1 + floor(2 log2 of the table cells with key < gamma)
                bucket = cost_bucket_of(P.bucket_key, sqrtf(best));
            } else {
                const float gam = sqrtf(best);
                P.out[v] = gam;
                ++my_eval;
                my_pass += gam <= 1.f;                 // decided on the value written
            }
        }
        const unsigned tm = __ballot_sync(kFull, tail);
        if (!BATCH && P.tile_mask) {
            // the tile's queue for the tile-staged walk: one bit per voxel
            if (lane == 0) P.tile_mask[(size_t)lt * 8 + (threadIdx.x >> 5)] = tm;
            if (tm) {
                unsigned bm = tail ? (unsigned)bucket + 1u : 0u;
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) bm = max(bm, __shfl_xor_sync(kFull, bm, o));
                if (lane == 0) atomicMax(&sh_tb[buf], bm);
            }
        }
        if (!BATCH && P.row_items && tm) {
            // this warp row's item for the row-staged walk
            unsigned bm = tail ? (unsigned)bucket : 0u;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) bm = max(bm, __shfl_xor_sync(kFull, bm, o));
            if (lane == 0) {
                const unsigned ip = atomicAdd(&P.ctr->row_count, 1u);
                P.row_items[ip] = ((unsigned long long)((unsigned)lt * 8u + (threadIdx.x >> 5)) << 32) | tm;
                P.row_bkt[ip] = (unsigned char)bm;
                atomicAdd(&P.ctr->row_hist[bm], 1u);
            }
        }
        if (tm) {
            unsigned pos0 = 0;
            if (lane == 0) pos0 = atomicAdd(&P.ctr->tail_count, (unsigned)__popc(tm));
            pos0 = __shfl_sync(kFull, pos0, 0);
            if (tail) {
                const unsigned pos = pos0 + __popc(tm & ((1u << lane) - 1u));
                if (pos < P.tail_cap) {
                    P.tail_raw[pos] = (unsigned)v;
                    P.tail_bucket[pos] = (unsigned char)bucket;
                    atomicAdd(&sh_hist[bucket], 1u);
                } else {
                    atomicOr(&P.ctr->flags, kFlagTailFull);
                }
            }
        }
        // tile[buf] is free for reuse once every thread has passed this point
        if (__syncthreads_or(timed_out)) {
            if (threadIdx.x == 0) {
                atomicOr(&P.ctr->flags, kFlagTimeout);
                // let this block's own copies land before it leaves
                mbar_wait_bounded(&bar[buf], (parity >> buf) & 1u);
                mbar_wait_bounded(&bar[buf ^ 1], (parity >> (buf ^ 1)) & 1u);
            }
            break;
        }
        if (!BATCH && P.tile_mask && threadIdx.x == 0) {
            const unsigned b1 = sh_tb[buf];
            if (b1) {
                const unsigned pos = atomicAdd(&P.ctr->tile_count, 1u);
                P.tile_list[pos] = (unsigned)lt;
                P.tile_bkt[pos] = (unsigned char)(b1 - 1u);
                atomicAdd(&P.ctr->tile_hist[b1 - 1u], 1u);
            }
            sh_tb[buf] = 0;            // the next tile of this buffer comes after the next barrier
        }
        t = sh_next[buf];
    }
    if (!BATCH || cur >= 0) flush(BATCH ? sh_P : P0);
}

// --------------------------------------------------------------------------
// k_shell_w: the same per-voxel work, one warp per tile, no block barriers
// --------------------------------------------------------------------------

// In k_shell the eight warps of a block share one staged tile and meet at a
// block barrier per tile, so a tile takes as long as its slowest warp row.
// Here each warp stages its own smaller tile (32 x 2 x 2 voxels in 3D, 32 x 4
// in 2D, with a one-voxel halo) into a double buffer of its own, with its own
// TMA copies and mbarriers (or plain loads when the grid takes no TMA map),
// and takes its next tile from the work counter by itself: warps never wait
// for one another until the end of the kernel.  Batched launches number the
// tiles of all pairs of a group in one range; a warp keeps a copy of its
// current pair's Problem in shared memory.  The next tile's number, pair, box
// and reference doses are all requested a tile ahead (warps stalled on memory
// half as often: 0.8 of 7 cycles per instruction; 454 to 418 us on a batch of
// eight planes and eight volumes, 656 to 640 us with the plane seeds on a
// 320x320x240 map).
template <int N>
struct WarpTile {
    static constexpr int TX = 32, TY = N == 3 ? 2 : 4, TZ = N == 3 ? 2 : 1;
    static constexpr int BX = 40, BY = TY + 2, BZ = N == 3 ? TZ + 2 : 1;
    static constexpr int ELEMS = BX * BY * BZ;
    static constexpr int STRIDE = (ELEMS + 31) / 32 * 32;   // 128-byte aligned buffers
    static_assert(STRIDE * 4 % 128 == 0, "TMA destination must stay 128-byte aligned");
};

template <int N, int MINB, bool BATCH>
__global__ void __launch_bounds__(256, MINB)
    k_shell_w(const __grid_constant__ Problem P0, const __grid_constant__ CUtensorMap tmap0,
              int use_tma0, int t_first, int ntiles, unsigned* tile_next,
              const __grid_constant__ SlabGate gate, const BatchDesc* __restrict__ bd)
{
    using T = WarpTile<N>;
    __shared__ __align__(128) float tiles[8][2][T::STRIDE];
    __shared__ float refs[8][2][T::TX * T::TY * T::TZ];     // the tiles' reference doses
    __shared__ __align__(8) uint64_t bar[8][2];
    __shared__ __align__(16) Problem sh_P[BATCH ? 8 : 1];   // batched: each warp's current pair
    __shared__ unsigned int sh_hist[kNumBuckets];
    __shared__ unsigned long long sh_eval, sh_pass;
    __shared__ unsigned int sh_rmax, sh_bad;
    // each warp's queued voxels (and cost buckets) not yet in the run's queue:
    // one atomic on the queue counter per kShellQ of them, not one per row
    constexpr int kShellQ = BATCH ? 64 : 128;     // (the batched kernel keeps 8 Problems too)
    __shared__ unsigned qv[8][kShellQ];
    __shared__ unsigned char qb[8][kShellQ];

    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (threadIdx.x < kNumBuckets) sh_hist[threadIdx.x] = 0;
    if (threadIdx.x == 0) {
        sh_eval = sh_pass = 0;
        sh_rmax = sh_bad = 0;
    }
    if (lane == 0) {
        mbar_init(&bar[w][0], 1);
        mbar_init(&bar[w][1], 1);
        mbar_fence_init();
    }
    __syncthreads();
    grid_release();
    grid_wait();

    // global tile -> (pair, tile of that pair)
    auto locate = [&](int t, int& pr, int& lt) {
        if constexpr (!BATCH) {
            pr = 0;
            lt = t;
        } else {
            int lo = 0, hi = bd->npairs - 1;
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if (bd->tile_start[mid] <= t) lo = mid; else hi = mid - 1;
            }
            pr = lo;
            lt = t - bd->tile_start[lo];
        }
    };
    auto origin = [&](int nx, int ny, int lt, int& x0, int& y0, int& z0) {
        const int ntx = (nx + T::TX - 1) / T::TX, nty = (ny + T::TY - 1) / T::TY;
        x0 = (lt % ntx) * T::TX;
        y0 = ((lt / ntx) % nty) * T::TY;
        z0 = (lt / ntx / nty) * T::TZ;
    };
    bool gate_failed = false;                 // lane 0: a slab wait gave up
    // the copies of a tile (lt of pair pr) into buffer b, by the whole warp, a
    // whole tile ahead of its use: its box of evaluation doses by one TMA copy
    // issued by lane 0, or, for a grid without a TMA map (its rows are not
    // 16-byte aligned), by 4-byte asynchronous copies of every lane; its
    // reference doses by such copies too, each lane its own.  One cp.async
    // group per call, so that the group of the tile to compute is the second
    // most recent one.  (Slab gates come only with a TMA map.)
    constexpr int ROWS = T::TY * T::TZ;
    auto issue = [&](int t, int pr, int lt, int tma, int b) {
        if (t < ntiles) {
            const Problem& Q = BATCH ? bd->probs[pr] : P0;
            int x0, y0, z0;
            origin(Q.nx, Q.ny, lt, x0, y0, z0);
            const int nx = Q.nx, ny = Q.ny, nz = Q.nz;
            if (tma) {
                if constexpr (BATCH) {
                    // the buffer may hold an earlier pair's box, written by the lanes
                    fence_async_shared();
                    __syncwarp();
                }
                if (lane == 0) {
                    const CUtensorMap* map = BATCH ? &bd->maps[pr] : &tmap0;
                    if (!BATCH && gate.flag && !gate_failed) {
                        // the box reads slices z0 - 1 .. z0 + TZ, from at most two slabs
                        const int zlo = max(z0 - 1, 0), zhi = min(z0 + T::TZ, nz - 1);
                        if (!flag_wait_bounded(gate.flag + zlo / gate.depth, gate.epoch) ||
                            !flag_wait_bounded(gate.flag + zhi / gate.depth, gate.epoch)) {
                            atomicOr(&Q.ctr->flags, kFlagTimeout);     // the run reports a timeout
                            gate_failed = true;                        // and this warp waits no more
                        }
                        fence_async_global();
                    }
                    mbar_arrive_expect_tx(&bar[w][b], T::ELEMS * (uint32_t)sizeof(float));
                    if (N == 3) tma_load_3d(tiles[w][b], map, x0 - 4, y0 - 1, z0 - 1, &bar[w][b]);
                    else tma_load_2d(tiles[w][b], map, x0 - 4, y0 - 1, &bar[w][b]);
                }
                // the other lanes wait here for lane 0's slab waits: polling the box's
                // barrier meanwhile would slow lane 0's own polls down
                if (!BATCH && gate.flag) __syncwarp();
            } else {
                const float* ev = Q.ev;
                float* dst = tiles[w][b];
                for (int i = lane; i < T::ELEMS; i += 32) {
                    const int bx = i % T::BX, by = (i / T::BX) % T::BY, bz = i / (T::BX * T::BY);
                    const int gx = x0 - 4 + bx, gy = y0 - 1 + by, gz = (N == 3 ? z0 - 1 : 0) + bz;
                    const bool in = (unsigned)gx < (unsigned)nx && (unsigned)gy < (unsigned)ny &&
                                    (N == 2 || (unsigned)gz < (unsigned)nz);
                    if (in) cp_async_f32(dst + i, ev + ((long long)gz * ny + gy) * nx + gx);
                    else dst[i] = kNaN;             // a node outside the grid
                }
            }
            const int x = x0 + lane;
            const float* src = Q.ref + ((long long)z0 * ny + y0) * nx + x;
#pragma unroll
            for (int r = 0; r < ROWS; ++r) {
                const int ly = r % T::TY, lz = r / T::TY;
                if (x < nx && y0 + ly < ny && z0 + lz < nz)
                    cp_async_f32(&refs[w][b][r * 32 + lane], src + ((long long)lz * ny + ly) * nx);
            }
        }
        cp_async_commit();
    };
    auto pair_tma = [&](int t, int pr) { return BATCH ? (t < ntiles ? bd->use_tma[pr] : 0) : use_tma0; };
    const int nwarps = (int)gridDim.x * 8;
    // the first two tiles of every warp, then the work counter, read a tile ahead
    int t = t_first + (int)blockIdx.x * 8 + w, nt = t + nwarps;
    int pr = 0, lt = 0;                       // the current tile's pair, and its number in the pair
    if (t < ntiles) locate(t, pr, lt);
    int tma = pair_tma(t, pr);
    issue(t, pr, lt, tma, 0);

    unsigned my_eval = 0, my_pass = 0;
    float my_rmax = 0.f;
    bool bad_ev = false, timed_out = false;
    uint32_t parity = 0;                      // bit b: phase of bar[w][b] to wait for
    int b = 0;
    int cur = -1;                             // batched: the pair in sh_P[w] and counted in my_*
    // the current pair's constants: dose norm, cutoff, and the bound below
    // which a voxel is final (every face not through the voxel is at spatial
    // distance >= the first table key, or >= the cover radius when the table
    // was cut)
    float dnorm = 0.f, thr = 0.f, qlim = 0.f;
    auto constants = [&](const Problem& Q) {
        dnorm = resolve_dnorm(Q);
        thr = cutoff_threshold(Q.local, Q.cutoff_frac, dnorm);
        const float k0 = Q.ntable > 0 ? Q.table[0].key : kInf;
        qlim = fminf(k0 * k0, Q.r_cover * Q.r_cover);
    };
    if constexpr (!BATCH) constants(P0);

    // a warp's counts -> its pair's counters (batched: when its pair changes)
    auto flush_counts = [&](const Problem& Q) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            my_eval += __shfl_xor_sync(kFull, my_eval, o);
            my_pass += __shfl_xor_sync(kFull, my_pass, o);
            my_rmax = fmaxf(my_rmax, __shfl_xor_sync(kFull, my_rmax, o));
        }
        if (__any_sync(kFull, bad_ev) && lane == 0) atomicOr(&Q.ctr->flags, kFlagNonFinite);
        if (lane == 0) {
            if (my_eval) atomicAdd(&Q.ctr->n_eval, (unsigned long long)my_eval);
            if (my_pass) atomicAdd(&Q.ctr->n_pass, (unsigned long long)my_pass);
            if (my_rmax > 0.f) atomicMax(&Q.ctr->rmax_enc, fenc(Q.local ? my_rmax : my_rmax / (Q.dd_frac * dnorm)));
        }
        my_eval = my_pass = 0;
        my_rmax = 0.f;
        bad_ev = false;
    };

    int qn = 0;                               // entries in qv[w] (warp-uniform)
    auto flush_queue = [&](const Problem& Q) {
        if (qn == 0) return;
        unsigned base = 0;
        if (lane == 0) base = atomicAdd(&Q.ctr->tail_count, (unsigned)qn);
        base = __shfl_sync(kFull, base, 0);
        for (int i0 = 0; i0 < qn; i0 += 32) {
            const int i = i0 + lane;
            bool counted = false;
            int bk = 0;
            if (i < qn) {
                const unsigned pos = base + (unsigned)i;
                bk = qb[w][i];
                if (pos < Q.tail_cap) {
                    Q.tail_raw[pos] = qv[w][i];
                    Q.tail_bucket[pos] = (unsigned char)bk;
                    counted = true;
                } else {
                    atomicOr(&Q.ctr->flags, kFlagTailFull);
                }
            }
            if constexpr (BATCH) {
                // the pair's histogram, one atomic per distinct bucket of the 32
                const unsigned peers = __match_any_sync(kFull, counted ? bk : -1);
                if (counted && lane == __ffs(peers) - 1)
                    atomicAdd(&Q.ctr->hist[bk], (unsigned)__popc(peers));
            } else {
                if (counted) atomicAdd(&sh_hist[bk], 1u);
            }
        }
        __syncwarp();
        qn = 0;
    };

    while (t < ntiles) {
        unsigned nn = 0;                       // the tile after next
        if (lane == 0) nn = atomicAdd(tile_next, 1u);
        int npr = 0, nlt = 0;
        if (nt < ntiles) locate(nt, npr, nlt);
        const int ntma = pair_tma(nt, npr);
        issue(nt, npr, nlt, ntma, b ^ 1);
        if constexpr (BATCH) {
            if (pr != cur) {                   // warp-uniform
                if (cur >= 0) {
                    flush_queue(sh_P[w]);
                    flush_counts(sh_P[w]);
                }
                __syncwarp();
                const int* src = (const int*)&bd->probs[pr];
                int* dst = (int*)&sh_P[w];
                for (int i = lane; i < (int)(sizeof(Problem) / 4); i += 32) dst[i] = src[i];
                __syncwarp();
                cur = pr;
                constants(sh_P[w]);
            }
        }
        const Problem& P = BATCH ? sh_P[w] : P0;
        float* tl = tiles[w][b];
        int x0, y0, z0;
        origin(P.nx, P.ny, lt, x0, y0, z0);
        cp_async_wait<1>();                    // this tile's copies (the next tile's may be in flight)
        if (tma) {
            if (!mbar_wait_bounded(&bar[w][b], (parity >> b) & 1u)) {
                timed_out = true;              // (warp-uniform: every lane polls the same phase)
                break;
            }
            parity ^= 1u << b;
        } else {
            __syncwarp();
        }
#pragma unroll 1
        for (int r = 0; r < ROWS; r += 2) {        // rows y and y + 1 together
            const int ly = r % T::TY, lz = r / T::TY;
            const int x = x0 + lane, y = y0 + ly, z = z0 + lz;
            const int tix = ((N == 3 ? lz + 1 : 0) * T::BY + (ly + 1)) * T::BX + (lane + 4);
            const float dr[2] = {refs[w][b][r * 32 + lane], refs[w][b][r * 32 + 32 + lane]};
            const bool in0 = x < P.nx && y < P.ny && z < P.nz, in1 = in0 && y + 1 < P.ny;
            const bool act[2] = {in0 && is_evaluated(P, dr[0], thr), in1 && is_evaluated(P, dr[1], thr)};
            float* const out = P.out + (in0 ? ((long long)z * P.ny + y) * P.nx + x : 0);
            if (in0) {
                if (!act[0]) out[0] = kNaN;
                bad_ev |= !isfinite(tl[tix]);       // every evaluation dose is some tile's centre
            }
            if (in1) {
                if (!act[1]) out[P.nx] = kNaN;
                bad_ev |= !isfinite(tl[tix + T::BX]);
            }
            float best[2] = {0.f, 0.f};
            // gamma0 = |g| / dD.  Where the doses agree gamma is 0 without the faces: equal
            // doses of 160x160x120 voxels take 41 us per map, with the faces 66 us.
            const float g0 = fabsf(tl[tix] - dr[0]), g1 = fabsf(tl[tix + T::BX] - dr[1]);
            if ((act[0] && g0 != 0.f) || (act[1] && g1 != 0.f)) {
                const float dD0 = P.dd_frac * (P.local ? dr[0] : dnorm), dD1 = P.dd_frac * (P.local ? dr[1] : dnorm);
                // with one dD for all voxels the division of gamma0 waits for the maximum
                if (P.local) my_rmax = max3(my_rmax, act[0] ? g0 / dD0 : 0.f, act[1] ? g1 / dD1 : 0.f);
                else my_rmax = max3(my_rmax, act[0] ? g0 : 0.f, act[1] ? g1 : 0.f);
                near_gamma2_pair<N, T::BX, T::BX * T::BY>(tl, tix, dr[0], dr[1], dD0, dD1, P.mt.kappa, best[0],
                                                          best[1]);
            }
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                bool tail = false;
                int bucket = 0;
                if (act[k]) {
                    tail = best[k] > qlim;
                    if (tail) {
                        out[k ? P.nx : 0] = best[k];       // gamma^2, finished by the table walk
                        // 1 + floor(2 log2 of the table cells with key < gamma)
                        bucket = cost_bucket_of(P.bucket_key, sqrtf(best[k]));
                    } else {
                        const float gam = sqrtf(best[k]);
                        out[k ? P.nx : 0] = gam;
                        ++my_eval;
                        my_pass += gam <= 1.f;             // decided on the value written
                    }
                }
                const unsigned tm = __ballot_sync(kFull, tail);
                if (tm) {
                    if (qn + 32 > kShellQ) flush_queue(P);
                    if (tail) {
                        const int i = qn + __popc(tm & ((1u << lane) - 1u));
                        qv[w][i] = (unsigned)(((long long)z * P.ny + y + k) * P.nx + x);
                        qb[w][i] = (unsigned char)bucket;
                    }
                    qn += __popc(tm);
                    __syncwarp();
                }
            }
        }
        __syncwarp();                          // tiles[w][b] is free for the copy after next
        t = nt;
        pr = npr;
        lt = nlt;
        tma = ntma;
        nt = t_first + 2 * nwarps + (int)__shfl_sync(kFull, nn, 0);
        b ^= 1;
    }
    cp_async_wait<0>();                        // no copy into this block's memory outlives it
    if (timed_out) {
        if (lane == 0) {
            if constexpr (BATCH) atomicOr(&bd->probs[cur < 0 ? 0 : cur].ctr->flags, kFlagTimeout);
            else atomicOr(&P0.ctr->flags, kFlagTimeout);
            // let this warp's own copies land before the block leaves
            mbar_wait_bounded(&bar[w][0], parity & 1u);
            mbar_wait_bounded(&bar[w][1], (parity >> 1) & 1u);
        }
        __syncwarp();
    }
    if constexpr (BATCH) {
        if (cur >= 0) {
            flush_queue(sh_P[w]);
            flush_counts(sh_P[w]);
        }
    } else {
        flush_queue(P0);
        // per block, then one atomic each: same-address atomics serialise in L2
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            my_eval += __shfl_xor_sync(kFull, my_eval, o);
            my_pass += __shfl_xor_sync(kFull, my_pass, o);
            my_rmax = fmaxf(my_rmax, __shfl_xor_sync(kFull, my_rmax, o));
        }
        const bool bad = __any_sync(kFull, bad_ev);
        if (lane == 0) {
            if (my_eval) atomicAdd(&sh_eval, (unsigned long long)my_eval);
            if (my_pass) atomicAdd(&sh_pass, (unsigned long long)my_pass);
            if (!P0.local && my_rmax > 0.f) my_rmax /= P0.dd_frac * dnorm;
            atomicMax(&sh_rmax, fenc(my_rmax));
            if (bad) sh_bad = 1;
        }
        __syncthreads();
        if (threadIdx.x < kNumBuckets && sh_hist[threadIdx.x])
            atomicAdd(&P0.ctr->hist[threadIdx.x], sh_hist[threadIdx.x]);
        if (threadIdx.x == 0) {
            if (sh_eval) atomicAdd(&P0.ctr->n_eval, sh_eval);
            if (sh_pass) atomicAdd(&P0.ctr->n_pass, sh_pass);
            atomicMax(&P0.ctr->rmax_enc, sh_rmax);
            if (sh_bad) atomicOr(&P0.ctr->flags, kFlagNonFinite);
        }
    }
}

// Table cells a queued voxel of cost bucket b is estimated to key: the middle
// of the bucket.
__device__ __forceinline__ float bucket_cells(int b) { return b > 0 ? exp2f((2 * b - 1) * 0.25f) : 0.5f; }

// The estimated cells of a whole queue, lane b of a full warp holding the count
// of bucket b.
__device__ __forceinline__ float queue_cells(unsigned count)
{
    float c = (float)count * bucket_cells(threadIdx.x & 31);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(kFull, c, o);
    return c;
}

// Whether the walk of a queue with this many estimated cells takes the cells'
// dose ranges from an array, which the ordering kernel then writes (it decides,
// and tells the walk with Counters::range_on): one read
// per tested cell instead of eight and their minimum and maximum, for a pass
// over the grid that reads 4 and writes 8 bytes per voxel.  The line lies where
// the pass (2.8 us per million voxels) meets what it saves (1.3 to 2.2 us per
// million cells), with a margin: 320x320x240 voxels, 395 M cells: 68 us for
// 520 us; 1.05 G cells: 2.35 ms.
constexpr float kRangeCells = 3.f;                 // tested cells per grid voxel
__device__ __forceinline__ bool wants_range(const Problem& P, float cells)
{
    return P.range && P.plane_raw && cells > kRangeCells * (float)P.nvox;
}

// A dose range, by an ordinary load: the kernel before writes them, and this one
// may have been set up meanwhile, so they are not read-only for its lifetime.
// (Constant once the walk runs, so the compiler may move it like a read-only one.)
__device__ __forceinline__ float2 load_range(const float2* p)
{
    float2 r;
    asm("ld.global.v2.f32 {%0, %1}, [%2];" : "=f"(r.x), "=f"(r.y) : "l"(p));
    return r;
}

// The queue's parts chosen from the queue itself (option group_bucket < 0):
// a queued voxel of cost bucket b is estimated to key c(b) = 2^((2b - 1) / 4)
// table cells (the middle of the bucket), the walk's W = sum of c over the
// queue, spread over its L lanes, ideally takes T = W / L steps per lane.  A
// voxel walks alone unless that takes longer than s T; it walks 4 lanes
// above s T, 8 above 4 s T and a whole warp above 8 s T, so that no voxel's
// own walk sets the kernel's length while the lanes stay busy.  Called by a
// full warp, lane b holding the count of bucket b; every lane gets the
// three thresholds.
__device__ __forceinline__ void auto_part_buckets(unsigned count, unsigned lanes, float scale, int& b4,
                                                  int& b8, int& b32)
{
    const int lane = threadIdx.x & 31;
    const float c = lane > 0 ? exp2f((2 * lane - 1) * 0.25f) : 0.f;
    float w = (float)count * c;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) w += __shfl_xor_sync(kFull, w, o);
    const float t = scale * w / (float)max(lanes, 1u);
    auto first_above = [&](float lim) {
        const unsigned m = __ballot_sync(kFull, lane > 0 && c > lim);
        return m ? __ffs(m) - 1 : kNumBuckets;
    };
    b4 = first_above(t);
    b8 = first_above(4.f * t);
    b32 = first_above(8.f * t);
}

// --------------------------------------------------------------------------
// Queue ordering: bucket offsets (most expensive first) and scatter
// --------------------------------------------------------------------------

// Scatter queued voxels into bucket order.  Every block derives the bucket
// starts from the histogram itself (32 values), then reserves one range per
// bucket per block-chunk with a single atomic on a per-bucket cursor.
__global__ void __launch_bounds__(256) k_scatter(const __grid_constant__ Problem P)
{
    __shared__ unsigned start[kNumBuckets], cnt[kNumBuckets], base[kNumBuckets];
    __shared__ float s_cells;
    grid_release();
    grid_wait();
    if (threadIdx.x < kNumBuckets) {
        const unsigned own = P.ctr->hist[threadIdx.x];
        unsigned sum = own;                    // of this bucket and the costlier ones
#pragma unroll
        for (int o = 1; o < kNumBuckets; o <<= 1) {
            const unsigned u = __shfl_down_sync(kFull, sum, o);
            if (threadIdx.x + o < kNumBuckets) sum += u;
        }
        start[threadIdx.x] = sum - own;
        const float cells = queue_cells(own);
        if (threadIdx.x == 0) s_cells = cells;
    }
    __syncthreads();
    const unsigned total = min(P.ctr->tail_count, P.tail_cap);
    for (unsigned c0 = blockIdx.x * blockDim.x; c0 < total; c0 += gridDim.x * blockDim.x) {
        if (threadIdx.x < kNumBuckets) cnt[threadIdx.x] = 0;
        __syncthreads();
        const unsigned i = c0 + threadIdx.x;
        int b = -1;
        unsigned rank = 0;
        if (i < total) {
            b = P.tail_bucket[i];
            rank = atomicAdd(&cnt[b], 1u);
        }
        __syncthreads();
        if (threadIdx.x < kNumBuckets && cnt[threadIdx.x])
            base[threadIdx.x] = start[threadIdx.x] + atomicAdd(&P.ctr->cursor[threadIdx.x], cnt[threadIdx.x]);
        __syncthreads();
        if (b >= 0) {
            P.tail_sorted[base[b] + rank] = P.tail_raw[i];
            if (P.plane_raw) P.plane_sorted[base[b] + rank] = P.plane_raw[i];
        }
        __syncthreads();
    }
    if (!wants_range(P, s_cells)) return;
    if (blockIdx.x == 0 && threadIdx.x == 0) P.ctr->range_on = 1u;
    // the dose range of every cell whose vertices all lie in the grid: a warp
    // takes a segment of 31 cells along x and marches along z, each node read once
    const int lane = threadIdx.x & 31;
    const int nx = P.nx, ny = P.ny, nz = P.nz, sz = nx * ny;
    const int segs = (nx + 30) / 31;
    constexpr int kRun = 16;                       // cells along z per turn
    const int runs = P.ndim == 3 ? (nz + kRun - 1) / kRun : 1;
    const long long work = (long long)segs * ny * runs;
    for (long long wk = (long long)blockIdx.x * 8 + (threadIdx.x >> 5); wk < work; wk += (long long)gridDim.x * 8) {
        const int sg = (int)(wk % segs), y = (int)(wk / segs % ny), rn = (int)(wk / segs / ny);
        const int x = sg * 31 + lane, z0 = rn * kRun;
        if (y + 1 >= ny) continue;                 // warp-uniform
        const bool inx = x < nx;
        float lo = 0.f, hi = 0.f;                  // of the nodes (x, x + 1) x (y, y + 1) one plane below
        for (int z = z0; z <= (P.ndim == 3 ? min(z0 + kRun, nz - 1) : 0); ++z) {
            const float* q = P.ev + ((long long)z * sz + (long long)y * nx + x);
            const float a = inx ? __ldg(q) : 0.f, c = inx ? __ldg(q + nx) : 0.f;
            float l = fminf(a, c), h = fmaxf(a, c);
            l = fminf(l, __shfl_down_sync(kFull, l, 1));
            h = fmaxf(h, __shfl_down_sync(kFull, h, 1));
            if (lane < 31 && x + 1 < nx && (P.ndim == 2 || z > z0))
                P.range[(long long)(P.ndim == 3 ? z - 1 : 0) * sz + (long long)y * nx + x] =
                    P.ndim == 3 ? make_float2(fminf(l, lo), fmaxf(h, hi)) : make_float2(l, h);
            lo = l;
            hi = h;
        }
    }
}

// The tiles with queued voxels in order of their largest cost bucket, most
// expensive first (same scheme as k_scatter).
__global__ void __launch_bounds__(256) k_scatter_tiles(const __grid_constant__ Problem P)
{
    __shared__ unsigned start[kNumBuckets], cnt[kNumBuckets], base[kNumBuckets];
    if (threadIdx.x == 0) {
        unsigned acc = 0;
        for (int b = kNumBuckets - 1; b >= 0; --b) {
            start[b] = acc;
            acc += P.ctr->tile_hist[b];
        }
    }
    const unsigned total = P.ctr->tile_count;
    for (unsigned c0 = blockIdx.x * blockDim.x; c0 < total; c0 += gridDim.x * blockDim.x) {
        if (threadIdx.x < kNumBuckets) cnt[threadIdx.x] = 0;
        __syncthreads();
        const unsigned i = c0 + threadIdx.x;
        int b = -1;
        unsigned rank = 0;
        if (i < total) {
            b = P.tile_bkt[i];
            rank = atomicAdd(&cnt[b], 1u);
        }
        __syncthreads();
        if (threadIdx.x < kNumBuckets && cnt[threadIdx.x])
            base[threadIdx.x] = start[threadIdx.x] + atomicAdd(&P.ctr->tile_cursor[threadIdx.x], cnt[threadIdx.x]);
        __syncthreads();
        if (b >= 0) P.tile_sorted[base[b] + rank] = P.tile_list[i];
        __syncthreads();
    }
}

// The warp rows with queued voxels in order of their largest cost bucket,
// most expensive first (same scheme as k_scatter).
__global__ void __launch_bounds__(256) k_scatter_rows(const __grid_constant__ Problem P)
{
    __shared__ unsigned start[kNumBuckets], cnt[kNumBuckets], base[kNumBuckets];
    if (threadIdx.x == 0) {
        unsigned acc = 0;
        for (int b = kNumBuckets - 1; b >= 0; --b) {
            start[b] = acc;
            acc += P.ctr->row_hist[b];
        }
    }
    const unsigned total = P.ctr->row_count;
    for (unsigned c0 = blockIdx.x * blockDim.x; c0 < total; c0 += gridDim.x * blockDim.x) {
        if (threadIdx.x < kNumBuckets) cnt[threadIdx.x] = 0;
        __syncthreads();
        const unsigned i = c0 + threadIdx.x;
        int b = -1;
        unsigned rank = 0;
        if (i < total) {
            b = P.row_bkt[i];
            rank = atomicAdd(&cnt[b], 1u);
        }
        __syncthreads();
        if (threadIdx.x < kNumBuckets && cnt[threadIdx.x])
            base[threadIdx.x] = start[threadIdx.x] + atomicAdd(&P.ctr->row_cursor[threadIdx.x], cnt[threadIdx.x]);
        __syncthreads();
        if (b >= 0) P.row_sorted[base[b] + rank] = P.row_items[i];
        __syncthreads();
    }
}

// Global order of a batch group's queued voxels, in four parts by cost
// bucket: b >= group32_bucket, then b >= group8_bucket, then b >=
// group_bucket, then the rest (the thresholds made non-increasing); within a
// part pair by pair (so that the walks in flight share one pair's doses in
// L2), most expensive bucket first within a pair.  All thresholds 0 give one
// pair-major order.  Each pair's cursor[b] starts at its range in that order;
// item_start holds those starts, the total and the ends of the first three
// parts, and the walk's work counters restart.  One block.
__global__ void __launch_bounds__(256) k_bucket_scan_batch(const BatchDesc* __restrict__ bd)
{
    __shared__ unsigned tot[4];
    __shared__ unsigned sc[4][256];
    __shared__ unsigned hsum[kNumBuckets];
    __shared__ int sh_b[3];
    grid_release();
    grid_wait();
    const int np = bd->npairs, tid = threadIdx.x;
    if (bd->group_bucket < 0) {
        // parts chosen from the group's queue (auto_part_buckets over every pair's histogram)
        if (tid < kNumBuckets) hsum[tid] = 0;
        __syncthreads();
        for (int i = tid; i < np * kNumBuckets; i += blockDim.x) {
            const unsigned v = bd->probs[i / kNumBuckets].ctr->hist[i % kNumBuckets];
            if (v) atomicAdd(&hsum[i % kNumBuckets], v);
        }
        __syncthreads();
        if (tid < 32) {
            int a4, a8, a32;
            auto_part_buckets(hsum[tid], bd->walk_lanes, bd->auto_scale, a4, a8, a32);
            if (tid == 0) {
                sh_b[0] = a4;
                sh_b[1] = a8;
                sh_b[2] = a32;
            }
        }
        __syncthreads();
    }
    const bool autop = bd->group_bucket < 0;
    const int b32 = autop ? sh_b[2] : bd->group32_bucket, b8 = min(autop ? sh_b[1] : bd->group8_bucket, b32),
              b4 = min(autop ? sh_b[0] : bd->group_bucket, b8);
    auto part_of = [&](int b) { return b >= b32 ? 0 : (b >= b8 ? 1 : (b >= b4 ? 2 : 3)); };
    auto sums = [&](int p, unsigned (&u)[4]) {
        u[0] = u[1] = u[2] = u[3] = 0;
        if (p >= np) return;
        const Counters* c = bd->probs[p].ctr;
        for (int b = 0; b < kNumBuckets; ++b) u[part_of(b)] += c->hist[b];
    };
    if (tid < 4) tot[tid] = 0;
    __syncthreads();
    for (int p = tid; p < np; p += blockDim.x) {
        unsigned u[4];
        sums(p, u);
        for (int r = 0; r < 4; ++r)
            if (u[r]) atomicAdd(&tot[r], u[r]);
    }
    __syncthreads();
    unsigned rb[4], carry[4] = {0, 0, 0, 0};
    rb[0] = 0;
    for (int r = 1; r < 4; ++r) rb[r] = rb[r - 1] + tot[r - 1];
    for (int c0 = 0; c0 < np; c0 += blockDim.x) {
        const int p = c0 + tid;
        unsigned u[4];
        sums(p, u);
        for (int r = 0; r < 4; ++r) sc[r][tid] = u[r];
        __syncthreads();
        for (int o = 1; o < (int)blockDim.x; o <<= 1) {      // inclusive scans, per part
            unsigned v[4];
            for (int r = 0; r < 4; ++r) v[r] = tid >= o ? sc[r][tid - o] : 0u;
            __syncthreads();
            for (int r = 0; r < 4; ++r) sc[r][tid] += v[r];
            __syncthreads();
        }
        if (p < np) {
            Counters* c = bd->probs[p].ctr;
            unsigned start[4];
            for (int r = 0; r < 4; ++r) start[r] = rb[r] + carry[r] + sc[r][tid] - u[r];
            for (int b = kNumBuckets - 1; b >= 0; --b) {
                const int r = part_of(b);
                bd->item_start[p * kNumBuckets + (kNumBuckets - 1 - b)] = start[r];
                c->cursor[b] = start[r];
                start[r] += c->hist[b];
            }
        }
        for (int r = 0; r < 4; ++r) carry[r] += sc[r][blockDim.x - 1];
        __syncthreads();
    }
    if (tid == 0) {
        const int nb = np * kNumBuckets;
        bd->item_start[nb] = rb[3] + tot[3];
        bd->item_start[nb + 1] = rb[1];
        bd->item_start[nb + 2] = rb[2];
        bd->item_start[nb + 3] = rb[3];
        *bd->head = 0;
        if (bd->part_head) {
            for (int r = 0; r < 4; ++r) bd->part_head[r] = 0;
            *bd->fix_count = 0;
        }
    }
}

// Scatter the pairs of a batch group into the group order (the block's pair:
// BatchGroup::blocks): per chunk of 256 queued voxels one atomic per cost bucket
// on the pair's cursor (as k_scatter), not one per voxel.
__global__ void __launch_bounds__(256) k_scatter_batch(const BatchDesc* __restrict__ bd,
                                                       const QueueBlock* __restrict__ blocks)
{
    __shared__ unsigned cnt[kNumBuckets], base[kNumBuckets];
    grid_release();
    grid_wait();
    const QueueBlock blk = blocks[blockIdx.x];
    const unsigned first = (blk.share & 0xffffu) * 256u;
    if (first >= blk.ctr->tail_count) return;                 // block-uniform
    const Problem& P = bd->probs[blk.pair];
    const unsigned total = min(P.ctr->tail_count, P.tail_cap);
    for (unsigned c0 = first; c0 < total; c0 += (blk.share >> 16) * 256u) {
        if (threadIdx.x < kNumBuckets) cnt[threadIdx.x] = 0;
        __syncthreads();
        const unsigned i = c0 + threadIdx.x;
        int b = -1;
        unsigned rank = 0;
        if (i < total) {
            b = P.tail_bucket[i];
            rank = atomicAdd(&cnt[b], 1u);
        }
        __syncthreads();
        if (threadIdx.x < kNumBuckets && cnt[threadIdx.x])
            base[threadIdx.x] = atomicAdd(&P.ctr->cursor[threadIdx.x], cnt[threadIdx.x]);
        __syncthreads();
        if (b >= 0) {
            const unsigned pos = base[b] + rank;
            bd->items_v[pos] = P.tail_raw[i];
            bd->items_p[pos] = (unsigned short)blk.pair;
            if (P.plane_raw) bd->items_s[pos] = P.plane_raw[i];
        }
        __syncthreads();
    }
}

// --------------------------------------------------------------------------
// k_tail: persistent, G lanes per voxel, walk of the sorted cell table
// --------------------------------------------------------------------------

struct TailStats {
    unsigned long long visited = 0, pruned = 0, keyed = 0;
};

template <int N>
__device__ __forceinline__ float visit_cell(const Problem& P, int x, int y, int z, int cx, int cy,
                                            int cz, float key, float dr, float inv, float dnorm,
                                            float best, TailStats& st)
{
    const int px = x + cx, py = y + cy, pz = z + cz;
    if ((unsigned)px >= (unsigned)P.nx || (unsigned)py >= (unsigned)P.ny ||
        (N == 3 && (unsigned)pz >= (unsigned)P.nz))
        return best;
    const bool ex = px + 1 < P.nx, ey = py + 1 < P.ny, ez = N == 3 && pz + 1 < P.nz;
    const long long sy = P.nx, sz = (long long)P.nx * P.ny;
    const long long p = (long long)pz * sz + (long long)py * sy + px;
    float q[8];
    uint32_t ok = 0;
    float qmin = kInf, qmax = -kInf;
#pragma unroll
    for (int u = 0; u < 8; ++u) {
        q[u] = kNaN;
        if (u < (1 << N)) {
            const bool present = (!(u & 1) || ex) && (!(u & 2) || ey) && (!(u & 4) || ez);
            if (present) {
                const long long o = p + ((u & 1) ? 1 : 0) + ((u & 2) ? sy : 0) + ((u & 4) ? sz : 0);
                q[u] = (__ldg(P.ev + o) - dr) * inv;
                qmin = fminf(qmin, q[u]);
                qmax = fmaxf(qmax, q[u]);
                ok |= 1u << u;
            }
        }
    }
    // every point of the cell's faces has spatial distance >= key and a dose
    // coordinate in [qmin, qmax]
    const float gap = qmin > 0.f ? qmin : (qmax < 0.f ? -qmax : 0.f);
    if (fmaf(gap, gap, key * key) >= best) {
        if (P.stats) ++st.pruned;
        return best;
    }
    if (P.stats) ++st.visited;
    const float cb = cell_all_faces<N, true>(P, q[0], q[1], q[2], q[3], q[4], q[5], q[6], q[7], ok, cx, cy,
                                       cz, p, dr, dnorm);
    return fminf(best, cb);
}

template <int G>
__device__ __forceinline__ float group_min(float v, unsigned gmask)
{
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) v = fminf(v, __shfl_xor_sync(gmask, v, o));
    return v;
}

// The walk ran past a truncated table with the running bound still above
// the cover radius: scan every cell of the remaining search box, G lanes
// together (rare; keeps the result exact).
template <int N, int G>
__device__ __forceinline__ float tail_box_scan(const Problem& P, int x, int y, int z, float dr,
                                            float inv, float dnorm, float best, int gl,
                                            unsigned gmask, TailStats& st)
{
    const float rc2 = P.r_cover * P.r_cover;
    const float g = sqrtf(best);
    const int ax = (int)ceilf(g / P.hn[0]) + 1;
    const int ay = (int)ceilf(g / P.hn[1]) + 1;
    const int az = N == 3 ? (int)ceilf(g / P.hn[2]) + 1 : 0;
    const int x0 = max(-ax - 1, -x), x1 = min(ax, P.nx - 1 - x);
    const int y0 = max(-ay - 1, -y), y1 = min(ay, P.ny - 1 - y);
    const int z0 = N == 3 ? max(-az - 1, -z) : 0, z1 = N == 3 ? min(az, P.nz - 1 - z) : 0;
    const long long bx = x1 - x0 + 1, by = y1 - y0 + 1, bz = z1 - z0 + 1;
    const long long tot = bx * by * bz;
    const float lim = rc2 * 0.99999f;
    float lb = best;
    for (long long b = gl; b < tot; b += G) {
        const int cx = x0 + (int)(b % bx);
        const long long rr = b / bx;
        const int cy = y0 + (int)(rr % by);
        const int cz = z0 + (int)(rr / by);
        const float axd = (float)max(max(cx, -cx - 1), 0) * P.hn[0];
        const float ayd = (float)max(max(cy, -cy - 1), 0) * P.hn[1];
        const float azd = N == 3 ? (float)max(max(cz, -cz - 1), 0) * P.hn[2] : 0.f;
        float k2 = axd * axd + ayd * ayd + azd * azd;
        if (k2 == 0.f)       // key-0 cell: only its faces off the voxel remain
            k2 = P.key0_far2[(cx & 1) | ((cy & 1) << 1) | ((cz & 1) << 2)];
        if (k2 < lim || k2 >= lb) continue;
        lb = visit_cell<N>(P, x, y, z, cx, cy, cz, sqrtf(k2), dr, inv, dnorm, lb, st);
    }
    return group_min<G>(lb, gmask);
}

template <int N, int G, int MINB, bool BATCH>
__global__ void __launch_bounds__(256, MINB)
    k_tail(const __grid_constant__ Problem P0, const BatchDesc* __restrict__ bd)
{
    const int lane = threadIdx.x & 31;
    const int gl = lane & (G - 1);
    const int gbase = lane & ~(G - 1);
    const unsigned gmask = G == 32 ? kFull : (((1u << G) - 1u) << gbase);
    const unsigned total = BATCH ? bd->item_start[kNumBuckets * bd->npairs]
                                 : min(P0.ctr->tail_count, P0.tail_cap);
    unsigned* head = BATCH ? bd->head : &P0.ctr->head;
    unsigned int my_eval = 0, my_pass = 0, my_over = 0;
    int my_pair = -1;          // batched: pair whose counts my_* hold
    TailStats st;
    // batched launches: hand this lane's counts to their pair
    auto flush_pair = [&]() {
        if (my_pair >= 0 && gl == 0) {
            Counters* c = bd->probs[my_pair].ctr;
            if (my_eval) atomicAdd(&c->n_eval, (unsigned long long)my_eval);
            if (my_pass) atomicAdd(&c->n_pass, (unsigned long long)my_pass);
            if (my_over) atomicAdd(&c->overflow_count, my_over);
        }
        my_eval = my_pass = my_over = 0;
    };

    for (;;) {
        unsigned item = 0;
        if (gl == 0) item = atomicAdd(head, 1u);
        item = __shfl_sync(gmask, item, gbase);
        if (item >= total) break;
        int pr = 0;
        unsigned v;
        if constexpr (BATCH) {
            v = bd->items_v[item];
            pr = bd->items_p[item];
            if (pr != my_pair) {                 // uniform over the group
                flush_pair();
                my_pair = pr;
            }
        } else {
            v = P0.sort_tail ? P0.tail_sorted[item] : P0.tail_raw[item];
        }
        const Problem& P = BATCH ? bd->probs[pr] : P0;
        const float dnorm = resolve_dnorm(P);
        const float rc2 = P.r_cover * P.r_cover;
        const int x = (int)(v % (unsigned)P.nx);
        const unsigned r1 = v / (unsigned)P.nx;
        const int y = (int)(r1 % (unsigned)P.ny);
        const int z = (int)(r1 / (unsigned)P.ny);
        const float dr = __ldg(P.ref + v);
        const float dD = P.dd_frac * (P.local ? dr : dnorm);
        const float inv = 1.0f / dD;
        float best = P.out[v];                       // gamma^2 over the faces through v
        int t = 0;
        while (t < P.ntable) {
            const int idx = t + gl;
            float key = kInf;
            uint32_t off = 0;
            if (idx < P.ntable) {
                const TableEntry e = P.table[idx];
                key = e.key;
                off = e.off;
            }
            const float k0 = __shfl_sync(gmask, key, gbase);
            if (k0 * k0 >= best) break;                   // A1 step 4b-ii, exact
            float cb = best;
            if (key * key < best) {
                if (P.stats) ++st.keyed;
                cb = visit_cell<N>(P, x, y, z, unpack10(off, 0), unpack10(off, 10),
                                   unpack10(off, 20), key, dr, inv, dnorm, best, st);
            }
            best = group_min<G>(cb, gmask);
            t += G;
        }
        if (t >= P.ntable && best > rc2) {
            if (gl == 0) ++my_over;
            best = tail_box_scan<N, G>(P, x, y, z, dr, inv, dnorm, best, gl, gmask, st);
        }
        if (gl == 0) {
            const float gam = sqrtf(best);
            P.out[v] = gam;
            ++my_eval;
            my_pass += gam <= 1.f;
        }
    }
    if constexpr (BATCH) flush_pair();
    if constexpr (!BATCH) {      // single-pair totals (batched ones went out per pair run)
        const Problem& P = P0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            my_eval += __shfl_xor_sync(kFull, my_eval, o);
            my_pass += __shfl_xor_sync(kFull, my_pass, o);
            my_over += __shfl_xor_sync(kFull, my_over, o);
            if (P.stats) {
                st.visited += __shfl_xor_sync(kFull, st.visited, o);
                st.pruned += __shfl_xor_sync(kFull, st.pruned, o);
                st.keyed += __shfl_xor_sync(kFull, st.keyed, o);
            }
        }
        if (lane == 0) {
            if (my_eval) atomicAdd(&P.ctr->n_eval, (unsigned long long)my_eval);
            if (my_pass) atomicAdd(&P.ctr->n_pass, (unsigned long long)my_pass);
            if (my_over) atomicAdd(&P.ctr->overflow_count, my_over);
            if (P.stats) {
                atomicAdd(&P.ctr->cells_visited, st.visited);
                atomicAdd(&P.ctr->cells_pruned, st.pruned);
                atomicAdd(&P.ctr->cells_keyed, st.keyed);
            }
        }
    }
}

// --------------------------------------------------------------------------
// Plane seeds: a queued voxel's bound before its table walk
// --------------------------------------------------------------------------

constexpr unsigned kNoSeed = 0xffffffffu;         // no table offset packs to this (two bits stay zero)
constexpr int kPlaneSteps = 3;

// The bound of a queued voxel from its own neighbourhood: kPlaneSteps steps
// that each replace the surface by the affine part of one cell, starting with
// the voxel's own, and move to the cell that holds the foot point on it; then
// every face of the last cell.  On the smooth doses of a plan the last cell
// holds the nearest point itself for 70 to 99 % of the queued voxels, so the
// walk starts from the final gamma: it keys no cell past it, plane_bound
// leaves few of the others to evaluate, and the cost buckets (recomputed
// here) are those of the walk that follows.  The bound is a true distance to
// the surface, so the result does not depend on it.  One thread per voxel;
// the cells differ per lane but every lane evaluates exactly one.  Bound by
// the latency of the dependent dose loads: 136 k voxels of a 160x160x120 map
// take 13.2 us, 648 k of a 200x200x150 map 35 us, 5.9 M of a 320x320x240 map
// 261 us, and spare the walk half of its time there.  Batched volumes, whose
// form needs 97 registers, take 64 (84 bytes spilled) in blocks of 128 for 32
// instead of 16 warps per SM: a batch's eight volumes 55.6 to 42 us.  For one
// pair the same (16 bytes spilled) was 10.4, 31 and 234 us, but a map of 99 k
// queued voxels, one wave of blocks either way, lost 1 us in 89.  What decides
// is the length of the queue, which the host does not know when it launches:
// a batch's is long as a rule.
__host__ __device__ constexpr int seed_threads(int n, bool batch) { return n == 3 && batch ? 128 : 256; }

template <int N, bool BATCH>
__global__ void __launch_bounds__(seed_threads(N, BATCH), seed_threads(N, BATCH) == 128 ? 8 : 0)
    k_plane_seed(const __grid_constant__ Problem P0, const BatchDesc* __restrict__ bd,
                 const QueueBlock* __restrict__ blocks)
{
    __shared__ unsigned sh_hist[kNumBuckets];
    grid_release();
    grid_wait();
    // this block's first item, and the items from one turn of the pair's blocks to the next
    unsigned first = blockIdx.x * blockDim.x, step = gridDim.x * blockDim.x, pr = 0;
    if constexpr (BATCH) {
        constexpr unsigned kSub = 256u / seed_threads(N, true);
        const QueueBlock blk = blocks[blockIdx.x / kSub];
        pr = blk.pair;
        first = (blk.share & 0xffffu) * 256u + blockIdx.x % kSub * blockDim.x;
        step = (blk.share >> 16) * 256u;
        if (first >= blk.ctr->tail_count) return;             // block-uniform
    }
    const Problem& P = BATCH ? bd->probs[pr] : P0;
    const unsigned total = min(P.ctr->tail_count, P.tail_cap);
    if (first >= total) return;                               // block-uniform
    if (threadIdx.x < kNumBuckets) sh_hist[threadIdx.x] = 0;
    __syncthreads();
    const float dnorm = resolve_dnorm(P);
    const float hn2[3] = {P.mt.hn2[0], P.mt.hn2[1], P.mt.hn2[2]};
    const float kap[3] = {P.mt.kappa[1], P.mt.kappa[2], P.mt.kappa[4]};
    const int nx = P.nx, ny = P.ny, nz = P.nz, sz = nx * ny;
    for (unsigned i = first + threadIdx.x; i < total; i += step) {
        const unsigned v = P.tail_raw[i];
        const int x = (int)(v % (unsigned)nx);
        const unsigned r1 = v / (unsigned)nx;
        const int y = (int)(r1 % (unsigned)ny), z = (int)(r1 / (unsigned)ny);
        const float dr = __ldg(P.ref + v);
        const float inv = 1.0f / (P.dd_frac * (P.local ? dr : dnorm));
        const float best = P.out[v];
        // cells whose every vertex lies in the grid, at most the bound (and
        // the packed offset's range) away
        int lo[3], hi[3], c[3] = {0, 0, 0};
        const int xyz[3] = {x, y, z}, dim[3] = {nx, ny, nz};
        float e[8];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            lo[a] = a < N ? max(-xyz[a], -511) : 0;
            hi[a] = a < N ? min(dim[a] - 2 - xyz[a], 510) : 0;
            c[a] = max(lo[a], min(hi[a], 0));
        }
        const float rmax = sqrtf(best);
#pragma unroll 1
        for (int it = 0;; ++it) {
            const float* q = P.ev + ((int)v + c[0] + c[1] * nx + c[2] * sz);
#pragma unroll
            for (int u = 0; u < (1 << N); ++u)
                e[u] = __ldg(q + (u & 1) + ((u & 2) ? nx : 0) + ((u & 4) ? sz : 0));
            if (it == kPlaneSteps) break;
            const CellPlane<N> p = cell_plane<N>(e);
            float L = p.m - dr, D = 0.f, gk[3];
#pragma unroll
            for (int a = 0; a < N; ++a) {
                L = fmaf(-p.G[a], (float)c[a] + 0.5f, L);
                gk[a] = p.G[a] * kap[a];
                D = fmaf(p.G[a], gk[a], D);
            }
            const float inv2 = inv * inv;
            const float r = __fdividef(L * inv2, fmaf(D, inv2, 1.f));
            bool same = true;
#pragma unroll
            for (int a = 0; a < N; ++a) {
                const float lim = rmax * rsqrtf(hn2[a]);
                const float s = fminf(fmaxf(-r * gk[a], -lim), lim);
                const int t = max(lo[a], min(hi[a], __float2int_rd(s)));
                same = same && t == c[a];
                c[a] = t;
            }
            if (same) break;                                  // e holds this cell's doses
        }
        float q[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) q[u] = u < (1 << N) ? rel_dose(e[u], dr, inv) : kNaN;
        OwnVertex<N> own;
        own.take(q, c[0], c[1], c[2], P.mt.kappa, ill_dmax(P));
        CellGeom<float> g;
        cell_geom<N, float>(c[0], c[1], c[2], P.mt, g);
        bool ill = false;
        const float cb = cell_min_d2<N, float>(q, g, P.mt, ill_dmax(P), kInf, ill);
        if (ill || own.steep) {
            own.put(q);
            ill = cell_gram_ill<N>(q, (1u << (1 << N)) - 1u, P.mt.kappa, P.tau);
        }
        // a near-singular cell is left to the walk (and its FP64 redo)
        P.plane_raw[i] = ill ? kNoSeed : pack10(c[0], c[1], c[2]);
        if (!ill && cb < best) {
            P.out[v] = cb + 0.f;                              // -0 -> +0
            const int was = P.tail_bucket[i], now = cost_bucket_of(P.bucket_key, sqrtf(fmaxf(cb, 0.f)));
            if (now != was) {
                P.tail_bucket[i] = (unsigned char)now;
                atomicAdd(&sh_hist[now], 1u);
                atomicSub(&sh_hist[was], 1u);                 // wraps; the sum over the block is exact
            }
        }
    }
    __syncthreads();
    if (threadIdx.x < kNumBuckets && sh_hist[threadIdx.x])
        atomicAdd(&P.ctr->hist[threadIdx.x], sh_hist[threadIdx.x]);
}

// --------------------------------------------------------------------------
// k_tail_cq: the table walk, surviving cells evaluated 32 at a time by the warp
// --------------------------------------------------------------------------

// A warp takes a batch of up to 32 queued voxels of about the same cost, sets
// them up one per lane, and walks the table for 32 / g of them at a time, g
// lanes each (a round): lane l of a voxel looks at entries t + l and t + g + l, and the round
// ends when no lane's key is below its voxel's bound (the exact stop of A1
// step 4b-ii).  A cell below the bound is tested in three tiers, each of which
// leaves a fraction of the cells, so each runs with a full warp on the cells
// that the tier before has collected in a ring buffer:
//   1. the dose gap of its vertices with the key, in the round itself;
//   2. plane_bound, 32 cells at a time;
//   3. its faces, 32 cells at a time, which lower the owner's bound in shared
//      memory (atomicMin on the bits of a non-negative float).
// From the plane seed on the bound is nearly final, so a test against a bound
// that is not yet the lowest keeps few cells more, and it never drops one:
// each cell is evaluated with the arithmetic of k_tail and the map is the one
// k_tail writes.  The cell the plane seed evaluated is passed over.  The rings
// are emptied once per batch, not per round, so that few passes run part full.
//
// The queue is ordered by cost bucket, most expensive first: the voxels of
// the costliest buckets walk 32, 8 or 4 lanes each (options group32_bucket,
// group8_bucket, group_bucket), the rest one lane each.  The rare paths (a
// cell whose Gram matrix is near singular, a bound past a truncated table) are
// not taken here: such a voxel goes to fix_list with its bound, and k_tail_fix
// finishes it, so that this kernel's registers stay those of the FP32
// evaluation.
//
// What bounds it: issue (56 % at 25 % occupancy), about a third each in the
// three tiers; the dose loads hit L1 at 92 %.  Before, one walker per lane or
// group collected the cells past the dose gap alone and evaluated all of them
// (21.8 per queued voxel of a 320x320x240 map at 3 %/3 mm, 36.5 at 1 %/1 mm
// local; now 3.5 and 8.3): 10.5 ms there and 23.6 ms, now 2.95 ms and 7.11 ms
// (twelve warps in each of two blocks per SM); 428 us and 185 us on a
// 200x200x150 map at 2 %/2 mm.  Two entries per lane and step and the cells'
// dose ranges (wants_range) are the last 0.5 ms and 2.3 ms of these.
constexpr int kCqRing = 128;              // cells in each ring of a warp (up to 31 + 64 wait)

struct CqWarp {
    unsigned ring[2][kCqRing]; // pending cells of tiers 2 and 3: table entry << 5 | slot of the voxel
    unsigned best[32];         // per slot: running squared gamma (float bits),
    unsigned vox[32];          // voxel, reference dose, 1 / Delta D, grid position,
    float dr[32], inv[32];
    int xyz[3][32];
    unsigned skip[32];         // the plane seed's cell
    unsigned short pair[32];   // batched: its pair
    unsigned fixm;             // slots whose voxel goes to the finishing pass
};

// Lanes per voxel of the four parts of the queue.
constexpr int kCqParts = 4;
__device__ __forceinline__ int cq_part_lanes(int part)
{
    return part == 0 ? 32 : (part == 1 ? 8 : (part == 2 ? 4 : 1));
}

template <int N, int MINB, bool BATCH>
__global__ void __launch_bounds__(cq_threads(MINB), MINB)
    k_tail_cq(const __grid_constant__ Problem P0, const BatchDesc* __restrict__ bd)
{
    __shared__ CqWarp cqw[cq_threads(MINB) / 32];
    __shared__ unsigned s_end[kCqParts];   // the parts of the queue end at these items
    __shared__ unsigned long long s_stat[4];   // option "stats": visited, pruned, keyed, lane slots
    __shared__ unsigned s_cnt[2];          // single pair: voxels finished and passed
    __shared__ unsigned s_start[kNumBuckets];  // ... first item of each cost bucket (the costliest is 0)
    __shared__ float s_cells;              // ... estimated table cells of the whole queue
    CqWarp& W = cqw[threadIdx.x >> 5];
    volatile CqWarp& V = cqw[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31;
    const unsigned lt_mask = (1u << lane) - 1u;
    grid_release();
    grid_wait();
    if (threadIdx.x < 32) {
        if constexpr (BATCH) {
            // the group's queue: the parts of every pair, costliest part first
            // (k_bucket_scan_batch)
            if (lane == 0) {
                const int nb = kNumBuckets * bd->npairs;
                s_end[0] = bd->item_start[nb + 1];
                s_end[1] = bd->item_start[nb + 2];
                s_end[2] = bd->item_start[nb + 3];
                s_end[3] = bd->item_start[nb];
            }
        } else {
            // the cost-ordered queue: items of bucket >= cq_group32_bucket
            // first, then those of bucket >= cq_group8_bucket, then >=
            // cq_group_bucket, then the rest
            const Problem& P = P0;
            const unsigned total = min(P.ctr->tail_count, P.tail_cap);
            const unsigned hb = P.sort_tail ? P.ctr->hist[lane] : 0u;
            int b32 = P.cq_group32_bucket, b8 = min(P.cq_group8_bucket, b32), b4 = min(P.cq_group_bucket, b8);
            if (P.cq_group_bucket < 0)
                auto_part_buckets(hb, gridDim.x * blockDim.x, P.cq_auto_scale, b4, b8, b32);
            unsigned h32 = lane >= b32 ? hb : 0u, h8 = lane >= b8 ? hb : 0u, h4 = lane >= b4 ? hb : 0u;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                h32 += __shfl_xor_sync(kFull, h32, o);
                h8 += __shfl_xor_sync(kFull, h8, o);
                h4 += __shfl_xor_sync(kFull, h4, o);
            }
            unsigned above = hb;               // items of this bucket and costlier ones
            const float cells = queue_cells(hb);
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned u = __shfl_down_sync(kFull, above, o);
                if (lane + o < 32) above += u;
            }
            s_start[lane] = above - hb;
            if (lane == 0) {
                s_end[0] = min(h32, total);
                s_end[1] = min(h8, total);
                s_end[2] = min(h4, total);
                s_end[3] = total;
                s_cnt[0] = s_cnt[1] = 0;
                s_cells = cells;
            }
            if (lane < 4) s_stat[lane] = 0;
        }
    }
    if (lane == 0) W.fixm = 0;
    __syncthreads();
    unsigned* const heads = BATCH ? bd->part_head : P0.ctr->head_part;
    const float dnorm0 = BATCH ? 0.f : resolve_dnorm(P0);
    const bool stats = !BATCH && P0.stats;
    const unsigned nwarps = gridDim.x * (blockDim.x >> 5);
    const bool use_range = !BATCH && P0.range && P0.ctr->range_on;

    for (int part = 0; part < kCqParts; ++part) {
        const unsigned lo = part ? s_end[part - 1] : 0u, hi = s_end[part];
        if (lo >= hi) continue;
        // lanes per voxel: the part's, and more where it is too short to fill
        // the warps (the walk is then bound by its steps' latency)
        int g = cq_part_lanes(part);
        while (g < 32 && (unsigned long long)(hi - lo) * (unsigned)g * 2u <= 32ull * nwarps) g *= 2;
        const unsigned nv = 32u / (unsigned)g;     // voxels per round
        const int gl = lane & (g - 1);
        unsigned at = lo;                          // where the queue stood when this warp last looked
        for (;;) {
            // voxels per batch: as many rounds as keep it below half of a
            // warp's share of the queue's estimated cells, from the cost bucket
            // at the last known position (costs only fall from there); in a
            // batch group, whose parts mix pairs and costs, two rounds
            unsigned nb = nv;
            if constexpr (BATCH) {
                nb = min(32u, 2u * nv);
            } else if (P0.sort_tail) {
                const unsigned m = __ballot_sync(kFull, s_start[lane] <= at && (lane == 0 || s_start[lane - 1] > at));
                const float share = s_cells / (2.f * (float)nwarps * bucket_cells(m ? 31 - __clz(m) : 0));
                nb = min(32u, max(nv, (unsigned)fminf(share, 32.f) / nv * nv));
            }
            unsigned base = 0;
            if (lane == 0) base = atomicAdd(&heads[part], nb);
            base = __shfl_sync(kFull, base, 0) + lo;
            if (base >= hi) break;                 // warp-uniform
            at = base;
            const unsigned nlive = min(nb, hi - base);
            // ---- the batch's voxels, one per lane ----
            if ((unsigned)lane < nlive) {
                const unsigned item = base + (unsigned)lane;
                unsigned v, skip;
                int pr = 0;
                if constexpr (BATCH) {
                    v = bd->items_v[item];
                    pr = bd->items_p[item];
                    skip = bd->items_s[item];
                } else {
                    v = P0.sort_tail ? P0.tail_sorted[item] : P0.tail_raw[item];
                    skip = P0.sort_tail ? P0.plane_sorted[item] : P0.plane_raw[item];
                }
                const Problem& Q = BATCH ? bd->probs[pr] : P0;
                const float dr = __ldg(Q.ref + v);
                V.best[lane] = __float_as_uint(Q.out[v]);      // squared gamma, an upper bound
                V.vox[lane] = v;
                V.skip[lane] = skip;
                V.xyz[0][lane] = (int)(v % (unsigned)Q.nx);
                const unsigned r1 = v / (unsigned)Q.nx;
                V.xyz[1][lane] = (int)(r1 % (unsigned)Q.ny);
                V.xyz[2][lane] = (int)(r1 / (unsigned)Q.ny);
                V.dr[lane] = dr;
                V.inv[lane] = 1.0f / (Q.dd_frac * (Q.local ? dr : (BATCH ? resolve_dnorm(Q) : dnorm0)));
                if (BATCH) V.pair[lane] = (unsigned short)pr;
            }
            __syncwarp();
            unsigned head1 = 0, cnt1 = 0, head2 = 0, cnt2 = 0;   // the rings: [head, head + cnt)
            unsigned r0 = 0;                       // first slot of the next round
            int slot = 0, t = -1;                  // this lane's voxel and table entry (t < 0: no round)
            for (;;) {
                const bool rest = t < 0 && r0 >= nlive;        // every round is done: empty the rings
                if (cnt2 >= 32u || (rest && cnt1 == 0u && cnt2 > 0u)) {
                    // ---- tier 3: the faces of the oldest pending cells ----
                    const unsigned n = min(cnt2, 32u);
                    if ((unsigned)lane < n) {
                        const unsigned w = V.ring[1][(head2 + (unsigned)lane) & (kCqRing - 1)];
                        const int own = (int)(w & 31u);
                        const Problem& O = BATCH ? bd->probs[V.pair[own]] : P0;
                        const WalkEntry oe = O.walk[w >> 5];
                        const float odr = V.dr[own], oinv = V.inv[own];
                        const int onx = O.nx, osz = onx * O.ny;
                        const int cx = unpack10(oe.off, 0), cy = unpack10(oe.off, 10), cz = unpack10(oe.off, 20);
                        const bool ex = V.xyz[0][own] + cx + 1 < onx, ey = V.xyz[1][own] + cy + 1 < O.ny,
                                   ez = N == 3 && V.xyz[2][own] + cz + 1 < O.nz;
                        const float* q = O.ev + ((int)V.vox[own] + oe.lin);
                        float cq[8];
                        uint32_t ok = 0;
#pragma unroll
                        for (int u = 0; u < 8; ++u) {
                            cq[u] = kNaN;
                            if (u < (1 << N) && (!(u & 1) || ex) && (!(u & 2) || ey) && (!(u & 4) || ez)) {
                                cq[u] = rel_dose(__ldg(q + (u & 1) + ((u & 2) ? onx : 0) + ((u & 4) ? osz : 0)), odr, oinv);
                                ok |= 1u << u;
                            }
                        }
                        auto evaluate = [&](const Metric& mt, float dmax, float tau) {
                            OwnVertex<N> self;
                            self.take(cq, cx, cy, cz, mt.kappa, dmax);
                            CellGeom<float> cg;
                            cell_geom<N, float>(cx, cy, cz, mt, cg);
                            bool ill = false;
                            const float cb = cell_min_d2<N, float>(cq, cg, mt, dmax, kInf, ill);
                            if (ill || self.steep) {
                                self.put(cq);
                                ill = cell_gram_ill<N>(cq, ok, mt.kappa, tau);
                            }
                            if (ill)
                                atomicOr(&W.fixm, 1u << own);                  // k_tail_fix redoes it
                            else
                                atomicMin(&W.best[own], __float_as_uint(cb + 0.f));   // -0 -> +0
                        };
                        if constexpr (BATCH) {
                            // the owner's pair's metric: three 16-byte loads
                            const float4* m4 = bd->metric4 + 3 * (int)V.pair[own];
                            const float4 a = __ldg(m4), b = __ldg(m4 + 1), c = __ldg(m4 + 2);
                            Metric mt;
                            mt.hn2[0] = a.x; mt.hn2[1] = a.y; mt.hn2[2] = a.z;
                            mt.kappa[0] = 0.f;
                            mt.kappa[1] = b.x; mt.kappa[2] = b.y; mt.kappa[3] = b.z; mt.kappa[4] = b.w;
                            mt.kappa[5] = c.x; mt.kappa[6] = c.y; mt.kappa[7] = c.z;
                            evaluate(mt, a.w > 0.f ? 0.99f * rsqrtf(a.w) : kInf, a.w);   // bound as ill_dmax
                        } else {
                            evaluate(P0.mt, ill_dmax(P0), P0.tau);
                        }
                    }
                    head2 += n;
                    cnt2 -= n;
                    if (stats && lane == 0) atomicAdd(&s_stat[0], (unsigned long long)n);
                    __syncwarp();
                    continue;
                }
                if (cnt1 >= 32u || (rest && cnt1 > 0u)) {
                    // ---- tier 2: plane_bound of the oldest cells past the dose gap ----
                    const unsigned n = min(cnt1, 32u);
                    bool cand = false;
                    unsigned w = 0;
                    if ((unsigned)lane < n) {
                        w = V.ring[0][(head1 + (unsigned)lane) & (kCqRing - 1)];
                        const int own = (int)(w & 31u);
                        const Problem& O = BATCH ? bd->probs[V.pair[own]] : P0;
                        const WalkEntry oe = O.walk[w >> 5];
                        const int onx = O.nx, osz = onx * O.ny;
                        const float* q = O.ev + ((int)V.vox[own] + oe.lin);
                        float d[8];
#pragma unroll
                        for (int u = 0; u < (1 << N); ++u)
                            d[u] = __ldg(q + (u & 1) + ((u & 2) ? onx : 0) + ((u & 4) ? osz : 0));
                        const float c[3] = {(float)unpack10(oe.off, 0), (float)unpack10(oe.off, 10),
                                            (float)unpack10(oe.off, 20)};
                        float hn2[3], kap[3];
                        if constexpr (BATCH) {
                            const float4* m4 = bd->metric4 + 3 * (int)V.pair[own];
                            const float4 ma = __ldg(m4), mb = __ldg(m4 + 1);
                            hn2[0] = ma.x; hn2[1] = ma.y; hn2[2] = ma.z;
                            kap[0] = mb.x; kap[1] = mb.y; kap[2] = mb.w;
                        } else {
                            hn2[0] = P0.mt.hn2[0]; hn2[1] = P0.mt.hn2[1]; hn2[2] = P0.mt.hn2[2];
                            kap[0] = P0.mt.kappa[1]; kap[1] = P0.mt.kappa[2]; kap[2] = P0.mt.kappa[4];
                        }
                        const float ob = __uint_as_float(V.best[own]);
                        cand = oe.off != V.skip[own] &&
                               !(plane_bound<N>(d, c, V.dr[own], V.inv[own], hn2, kap) >= ob * kPlaneSlack);
                    }
                    head1 += n;
                    cnt1 -= n;
                    const unsigned cm = __ballot_sync(kFull, cand);
                    if (cand) V.ring[1][(head2 + cnt2 + (unsigned)__popc(cm & lt_mask)) & (kCqRing - 1)] = w;
                    cnt2 += (unsigned)__popc(cm);
                    if (stats && lane == 0) atomicAdd(&s_stat[1], (unsigned long long)(n - (unsigned)__popc(cm)));
                    __syncwarp();
                    continue;
                }
                if (t < 0) {
                    if (r0 >= nlive) break;                    // the batch is done
                    slot = (int)r0 + lane / g;                 // the next round: nv voxels, g lanes each
                    r0 += nv;
                    t = gl;
                }
                // the lane's voxel (from shared memory after every pass of
                // the other tiers, which so need not keep it in registers)
                const bool live = (unsigned)slot < nlive;
                const int sl = live ? slot : 0;
                const Problem& Q = BATCH ? bd->probs[V.pair[sl]] : P0;
                const int x = V.xyz[0][sl], y = V.xyz[1][sl], z = V.xyz[2][sl];
                const int nx = Q.nx, sz = nx * Q.ny;
                int reach = min(min(x, nx - 1 - x), min(y, Q.ny - 1 - y));   // cells of this margin lie in the grid
                if (N == 3) reach = min(reach, min(z, Q.nz - 1 - z));
                const float* const ev = Q.ev + V.vox[sl];
                const WalkEntry* const tab = Q.walk;
                // the cells' dose ranges, where they are worth a pass over the grid
                const float2* const range = BATCH || !use_range ? nullptr : P0.range + V.vox[sl];
                const float dr = V.dr[sl], inv = V.inv[sl];
                const float best = live ? __uint_as_float(V.best[sl]) : -1.f;   // < 0: nothing is below it
                WalkEntry en0 = tab[t], en1 = tab[t + g];
                // ---- tier 1: two table entries per lane and step ----
                auto test = [&](const WalkEntry& e, bool& edge) -> bool {
                    edge = false;                  // a cell with vertices outside the grid
                    if (!(e.key2 < best)) return false;
                    const float* q = ev + e.lin;
                    float dlo, dhi;
                    bool in = true;
                    if (e.margin <= reach) {
                        if (range) {
                            const float2 r = load_range(range + e.lin);
                            dlo = r.x;
                            dhi = r.y;
                        } else {
                            float d[8];
#pragma unroll
                            for (int u = 0; u < (1 << N); ++u)
                                d[u] = __ldg(q + (u & 1) + ((u & 2) ? nx : 0) + ((u & 4) ? sz : 0));
                            dlo = fminf(min3(d[0], d[1], d[2]), d[3]);
                            dhi = fmaxf(max3(d[0], d[1], d[2]), d[3]);
                            if constexpr (N == 3) {
                                dlo = min3(min3(dlo, d[4], d[5]), d[6], d[7]);
                                dhi = max3(max3(dhi, d[4], d[5]), d[6], d[7]);
                            }
                        }
                    } else {
                        // near the grid's faces: a cell outside it does not exist, one with
                        // vertices outside keeps the faces that lie inside
                        const int px = x + unpack10(e.off, 0), py = y + unpack10(e.off, 10), pz = z + unpack10(e.off, 20);
                        in = (unsigned)px < (unsigned)nx && (unsigned)py < (unsigned)Q.ny &&
                             (N == 2 || (unsigned)pz < (unsigned)Q.nz);
                        const bool ex = px + 1 < nx, ey = py + 1 < Q.ny, ez = N == 3 && pz + 1 < Q.nz;
                        edge = !(ex && ey && (N == 2 || ez));
                        dlo = kInf;
                        dhi = -kInf;
                        if (in) {
#pragma unroll
                            for (int u = 0; u < (1 << N); ++u) {
                                if ((!(u & 1) || ex) && (!(u & 2) || ey) && (!(u & 4) || ez)) {
                                    const float f = __ldg(q + (u & 1) + ((u & 2) ? nx : 0) + ((u & 4) ? sz : 0));
                                    dlo = fminf(dlo, f);
                                    dhi = fmaxf(dhi, f);
                                }
                            }
                        }
                    }
                    const float gap = max3(dlo - dr, dr - dhi, 0.f) * inv;
                    return in && fmaf(gap, gap, e.key2) < best;
                };
                // a whole cell goes to tier 2, one at the grid's edge to tier 3
                auto push = [&](bool cand, bool edge, unsigned ent) {
                    const unsigned cm = __ballot_sync(kFull, cand && !edge);
                    if (cand && !edge)
                        V.ring[0][(head1 + cnt1 + (unsigned)__popc(cm & lt_mask)) & (kCqRing - 1)] = ent << 5 | (unsigned)slot;
                    cnt1 += (unsigned)__popc(cm);
                    const unsigned em = __ballot_sync(kFull, cand && edge);
                    if (em) {
                        if (cand && edge)
                            V.ring[1][(head2 + cnt2 + (unsigned)__popc(em & lt_mask)) & (kCqRing - 1)] = ent << 5 | (unsigned)slot;
                        cnt2 += (unsigned)__popc(em);
                    }
                };
                do {
                    const WalkEntry e0 = en0, e1 = en1;
                    if (!__any_sync(kFull, e0.key2 < best)) {  // (of a lane's two keys the smaller)
                        t = -1;
                        break;
                    }
                    const unsigned ent = (unsigned)t;
                    // A lane whose key is past its bound stays where it is: in a batch
                    // the lanes' voxels may belong to pairs with tables of different
                    // lengths, and one that went on with the others would leave its own.
                    // (Of one pair the round ends within 2 g entries of the table's end.)
                    if (!BATCH || e0.key2 < best) t += 2 * g;
                    en0 = tab[t];                  // the table is padded with unreachable keys
                    en1 = tab[t + g];
                    bool g0, g1;
                    const bool c0 = test(e0, g0), c1 = test(e1, g1);
                    push(c0, g0, ent);
                    push(c1, g1, ent + (unsigned)g);
                    if (stats) {
                        const unsigned k0 = __ballot_sync(kFull, e0.key2 < best), k1 = __ballot_sync(kFull, e1.key2 < best);
                        const unsigned p0 = __ballot_sync(kFull, e0.key2 < best && !c0),
                                       p1 = __ballot_sync(kFull, e1.key2 < best && !c1);
                        if (lane == 0) {
                            atomicAdd(&s_stat[1], (unsigned long long)(__popc(p0) + __popc(p1)));
                            atomicAdd(&s_stat[2], (unsigned long long)(__popc(k0) + __popc(k1)));
                            atomicAdd(&s_stat[3], 64ull);
                        }
                    }
                } while (max(cnt1, cnt2) < 32u);
                __syncwarp();
            }
            // ---- final values, one voxel per lane ----
            const unsigned fixm = V.fixm;
            bool pass = false, fin = false;
            int pr = 0;
            if ((unsigned)lane < nlive) {
                if (BATCH) pr = V.pair[lane];
                const Problem& Q = BATCH ? bd->probs[pr] : P0;
                const unsigned v = V.vox[lane];
                const float b = __uint_as_float(V.best[lane]);
                if (((fixm >> lane) & 1u) || b > Q.r_cover * Q.r_cover) {
                    Q.out[v] = b;                              // squared gamma: k_tail_fix completes it
                    if constexpr (BATCH) {
                        const unsigned k = atomicAdd(bd->fix_count, 1u);
                        bd->fix_v[k] = v;
                        bd->fix_p[k] = (unsigned short)pr;
                    } else {
                        Q.fix_list[atomicAdd(&Q.ctr->fix_count, 1u)] = v;
                    }
                } else {
                    const float gam = sqrtf(b);
                    Q.out[v] = gam;
                    fin = true;
                    pass = gam <= 1.f;
                }
            }
            const unsigned fm = __ballot_sync(kFull, fin), pm = __ballot_sync(kFull, pass);
            if constexpr (BATCH) {
                if (fin) {                         // one atomic per pair of the batch (almost always one)
                    const unsigned peers = __match_any_sync(fm, pr);
                    if (lane == __ffs(peers) - 1) {
                        Counters* c = bd->probs[pr].ctr;
                        atomicAdd(&c->n_eval, (unsigned long long)__popc(peers));
                        if (pm & peers) atomicAdd(&c->n_pass, (unsigned long long)__popc(pm & peers));
                    }
                }
            } else if (lane == 0) {
                atomicAdd(&s_cnt[0], (unsigned)__popc(fm));
                atomicAdd(&s_cnt[1], (unsigned)__popc(pm));
            }
            __syncwarp();
            if (lane == 0 && fixm) W.fixm = 0;
            __syncwarp();
        }
    }
    if constexpr (!BATCH) {
        __syncthreads();
        if (threadIdx.x == 0) {
            if (s_cnt[0]) atomicAdd(&P0.ctr->n_eval, (unsigned long long)s_cnt[0]);
            if (s_cnt[1]) atomicAdd(&P0.ctr->n_pass, (unsigned long long)s_cnt[1]);
            if (stats) {
                atomicAdd(&P0.ctr->cells_visited, s_stat[0]);
                atomicAdd(&P0.ctr->cells_pruned, s_stat[1]);
                atomicAdd(&P0.ctr->cells_keyed, s_stat[2]);
                atomicAdd(&P0.ctr->lane_steps, s_stat[3]);
            }
        }
    }
}

// Finishing pass of k_tail_cq: one warp per voxel of the fix list, whose
// bound (gamma^2, an upper bound of the result) is in out.  The walk of
// k_tail (32 lanes, FP64 redo of near-singular cells) from that bound, then
// the box scan when it runs past the table.
template <int N, bool BATCH>
__global__ void __launch_bounds__(256) k_tail_fix(const __grid_constant__ Problem P0,
                                                  const BatchDesc* __restrict__ bd)
{
    grid_wait();                       // (the run's last kernel: nothing is released early)
    const int lane = threadIdx.x & 31;
    const unsigned nfix = BATCH ? *bd->fix_count : P0.ctr->fix_count;
    unsigned my_eval = 0, my_pass = 0, my_over = 0;
    TailStats st;
    for (unsigned i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < nfix;
         i += (gridDim.x * blockDim.x) >> 5) {
        const Problem& P = BATCH ? bd->probs[bd->fix_p[i]] : P0;
        const unsigned v = BATCH ? bd->fix_v[i] : P.fix_list[i];
        const float dnorm = resolve_dnorm(P);
        const int x = (int)(v % (unsigned)P.nx);
        const unsigned r1 = v / (unsigned)P.nx;
        const int y = (int)(r1 % (unsigned)P.ny), z = (int)(r1 / (unsigned)P.ny);
        const float dr = __ldg(P.ref + v);
        const float inv = 1.0f / (P.dd_frac * (P.local ? dr : dnorm));
        float best = P.out[v];
        int t = 0;
        while (t < P.ntable) {
            const int idx = t + lane;
            float key = kInf;
            uint32_t off = 0;
            if (idx < P.ntable) {
                const TableEntry e = P.table[idx];
                key = e.key;
                off = e.off;
            }
            const float k0 = __shfl_sync(kFull, key, 0);
            if (k0 * k0 >= best) break;
            float cb = best;
            if (key * key < best) {
                if (P.stats) ++st.keyed;
                cb = visit_cell<N>(P, x, y, z, unpack10(off, 0), unpack10(off, 10), unpack10(off, 20),
                                   key, dr, inv, dnorm, best, st);
            }
            best = group_min<32>(cb, kFull);
            t += 32;
        }
        const bool over = t >= P.ntable && best > P.r_cover * P.r_cover;
        if (over) best = tail_box_scan<N, 32>(P, x, y, z, dr, inv, dnorm, best, lane, kFull, st);
        if (lane == 0) {
            const float gam = sqrtf(best);
            P.out[v] = gam;
            if constexpr (BATCH) {
                atomicAdd(&P.ctr->n_eval, 1ull);
                if (gam <= 1.f) atomicAdd(&P.ctr->n_pass, 1ull);
                if (over) atomicAdd(&P.ctr->overflow_count, 1u);
            } else {
                ++my_eval;
                my_pass += gam <= 1.f;
                my_over += over;
            }
        }
    }
    if constexpr (!BATCH) {
        const Problem& P = P0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            my_eval += __shfl_xor_sync(kFull, my_eval, o);
            my_pass += __shfl_xor_sync(kFull, my_pass, o);
            my_over += __shfl_xor_sync(kFull, my_over, o);
            if (P.stats) {
                st.visited += __shfl_xor_sync(kFull, st.visited, o);
                st.pruned += __shfl_xor_sync(kFull, st.pruned, o);
                st.keyed += __shfl_xor_sync(kFull, st.keyed, o);
            }
        }
        if (lane == 0) {
            if (my_eval) atomicAdd(&P.ctr->n_eval, (unsigned long long)my_eval);
            if (my_pass) atomicAdd(&P.ctr->n_pass, (unsigned long long)my_pass);
            if (my_over) atomicAdd(&P.ctr->overflow_count, my_over);
            if (P.stats) {
                atomicAdd(&P.ctr->cells_visited, st.visited);
                atomicAdd(&P.ctr->cells_pruned, st.pruned);
                atomicAdd(&P.ctr->cells_keyed, st.keyed);
            }
        }
    }
}

// --------------------------------------------------------------------------
// k_walk: tile-staged walk of the queued voxels, one shell tile per block
// --------------------------------------------------------------------------

// Halo box of a walk tile in shared memory: the shell tile plus H voxels on
// every side (the x start stays a multiple of 4 floats for the TMA copy).
// Every cell whose corner lies within H - 1 voxels of a tile voxel (cells
// with box distance up to (H - 1) h) reads its eight doses from the box;
// cells further out read global memory.
template <int N>
struct WalkBox {
    using T = ShellTile<N>;
    static constexpr int H = 4;
    static constexpr int BX = T::TX + 2 * H, BY = T::TY + 2 * H, BZ = N == 3 ? T::TZ + 2 * H : 1;
    static constexpr int ELEMS = BX * BY * BZ;
    static constexpr int STRIDE = (ELEMS + 31) / 32 * 32;
    static_assert(STRIDE * 4 % 128 == 0, "TMA destination must stay 128-byte aligned");
    static_assert(H % 4 == 0, "the box's x start must stay 16-byte aligned");
};

constexpr int kWalkTableCache = 1024;        // first table entries kept in shared memory

// visit_cell with the eight doses from the staged box B when the whole cell
// lies inside it (b0x, b0y, b0z: grid coordinates of the box's first element).
template <int N, class B = WalkBox<N>>
__device__ __forceinline__ float visit_cell_box(const Problem& P, const float* __restrict__ bx,
                                                int b0x, int b0y, int b0z, int x, int y, int z,
                                                int cx, int cy, int cz, float key, float dr,
                                                float inv, float dnorm, float best, TailStats& st)
{
    const int px = x + cx, py = y + cy, pz = z + cz;
    if ((unsigned)px >= (unsigned)P.nx || (unsigned)py >= (unsigned)P.ny ||
        (N == 3 && (unsigned)pz >= (unsigned)P.nz))
        return best;
    const bool ex = px + 1 < P.nx, ey = py + 1 < P.ny, ez = N == 3 && pz + 1 < P.nz;
    const int lx = px - b0x, ly = py - b0y, lz = N == 3 ? pz - b0z : 0;
    const bool inbox = (unsigned)lx <= (unsigned)(B::BX - 2) && (unsigned)ly <= (unsigned)(B::BY - 2) &&
                       (N == 2 || (unsigned)lz <= (unsigned)(B::BZ - 2));
    const long long sy = P.nx, sz = (long long)P.nx * P.ny;
    const long long p = (long long)pz * sz + (long long)py * sy + px;
    const int lp = (lz * B::BY + ly) * B::BX + lx;
    float q[8];
    uint32_t ok = 0;
    float qmin = kInf, qmax = -kInf;
#pragma unroll
    for (int u = 0; u < 8; ++u) {
        q[u] = kNaN;
        if (u < (1 << N)) {
            const bool present = (!(u & 1) || ex) && (!(u & 2) || ey) && (!(u & 4) || ez);
            if (present) {
                const int lo = ((u & 1) ? 1 : 0) + ((u & 2) ? B::BX : 0) + ((u & 4) ? B::BX * B::BY : 0);
                const long long o = p + ((u & 1) ? 1 : 0) + ((u & 2) ? sy : 0) + ((u & 4) ? sz : 0);
                const float d = inbox ? bx[lp + lo] : __ldg(P.ev + o);
                q[u] = (d - dr) * inv;
                qmin = fminf(qmin, q[u]);
                qmax = fmaxf(qmax, q[u]);
                ok |= 1u << u;
            }
        }
    }
    const float gap = qmin > 0.f ? qmin : (qmax < 0.f ? -qmax : 0.f);
    if (fmaf(gap, gap, key * key) >= best) {
        if (P.stats) ++st.pruned;
        return best;
    }
    if (P.stats) ++st.visited;
    const float cb = cell_all_faces<N, true>(P, q[0], q[1], q[2], q[3], q[4], q[5], q[6], q[7], ok, cx, cy,
                                       cz, p, dr, dnorm);
    return fminf(best, cb);
}

// Minimum over the G lanes of a group (G a power of two <= 32, lanes gbase ..
// gbase + G - 1 of the warp, mask gmask).
__device__ __forceinline__ float group_min_rt(float v, int G, unsigned gmask)
{
    for (int o = G >> 1; o > 0; o >>= 1) v = fminf(v, __shfl_xor_sync(gmask, v, o));
    return v;
}

// One block per tile with queued voxels, in cost order: the halo box of the
// tile arrives by TMA (double-buffered, the next tile's copy in flight while
// this one is walked); the tile's queued voxels are read from its bit mask;
// G lanes per voxel (G chosen per tile from the number of queued voxels so
// that the block's 256 threads are used) walk the sorted cell table G cells
// at a time with the exact stop of Algorithm A1 step 4b-ii and the dose-gap
// bound, reading cell doses from the box.
template <int N, int MINB>
__global__ void __launch_bounds__(256, MINB)
    k_walk(const __grid_constant__ Problem P, const __grid_constant__ CUtensorMap wmap, int use_tma)
{
    using T = ShellTile<N>;
    using B = WalkBox<N>;
    __shared__ __align__(128) float box[2][B::STRIDE];
    __shared__ __align__(8) uint64_t bar[2];
    __shared__ TableEntry sh_table[kWalkTableCache];
    __shared__ unsigned short sh_q[T::TX * T::TY * T::TZ];
    __shared__ int sh_nq;
    __shared__ int sh_next[2];

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const unsigned ntiles = P.ctr->tile_count;
    const unsigned* order = P.sort_tail ? P.tile_sorted : P.tile_list;
    const int ncache = min(P.ntable, kWalkTableCache);
    for (int i = tid; i < ncache; i += blockDim.x) sh_table[i] = P.table[i];
    if (tid == 0) {
        mbar_init(&bar[0], 1);
        mbar_init(&bar[1], 1);
        mbar_fence_init();
    }
    __syncthreads();
    const float dnorm = resolve_dnorm(P);
    const float rc2 = P.r_cover * P.r_cover;
    const int ntx = (P.nx + T::TX - 1) / T::TX, nty = (P.ny + T::TY - 1) / T::TY;
    auto origin = [&](unsigned lt, int& x0, int& y0, int& z0) {
        x0 = (int)(lt % (unsigned)ntx) * T::TX;
        y0 = (int)((lt / (unsigned)ntx) % (unsigned)nty) * T::TY;
        z0 = N == 3 ? (int)(lt / (unsigned)ntx / (unsigned)nty) * T::TZ : 0;
    };
    auto issue = [&](unsigned i, int b) {
        if (i >= ntiles || !use_tma) return;
        int x0, y0, z0;
        origin(order[i], x0, y0, z0);
        mbar_arrive_expect_tx(&bar[b], B::ELEMS * (uint32_t)sizeof(float));
        if (N == 3) tma_load_3d(box[b], &wmap, x0 - B::H, y0 - B::H, z0 - B::H, &bar[b]);
        else tma_load_2d(box[b], &wmap, x0 - B::H, y0 - B::H, &bar[b]);
    };
    unsigned my_eval = 0, my_pass = 0, my_over = 0;
    TailStats st;
    uint32_t parity = 0;
    int buf = 0;
    unsigned i = blockIdx.x;
    if (tid == 0) issue(i, 0);
    for (; i < ntiles; buf ^= 1) {
        const unsigned lt = order[i];
        int x0, y0, z0;
        origin(lt, x0, y0, z0);
        const int b0x = x0 - B::H, b0y = y0 - B::H, b0z = N == 3 ? z0 - B::H : 0;
        if (tid == 0) {
            const unsigned nt = gridDim.x + atomicAdd(&P.ctr->tile_head, 1u);
            sh_next[buf] = (int)min(nt, ntiles);
            issue(nt, buf ^ 1);
        }
        // the tile's queued voxels, in voxel order (warp 0)
        if (warp == 0) {
            const unsigned w = lane < 8 ? P.tile_mask[(size_t)lt * 8 + lane] : 0u;
            const int c = __popc(w);
            int incl = c;
#pragma unroll
            for (int o = 1; o < 8; o <<= 1) {
                const int t = __shfl_up_sync(kFull, incl, o);
                if (lane >= o) incl += t;
            }
            int pos = incl - c;
            for (unsigned m = w; m; m &= m - 1) sh_q[pos++] = (unsigned short)(lane * 32 + __ffs(m) - 1);
            if (lane == 7) sh_nq = incl;
        }
        float* bx = box[buf];
        bool timed_out = false;
        if (use_tma) {
            timed_out = !mbar_wait_bounded(&bar[buf], (parity >> buf) & 1u);
            parity ^= 1u << buf;
        } else {
            for (int e = tid; e < B::ELEMS; e += blockDim.x) {
                const int ex_ = e % B::BX, ey_ = (e / B::BX) % B::BY, ez_ = e / (B::BX * B::BY);
                const int gx = b0x + ex_, gy = b0y + ey_, gz = b0z + ez_;
                const bool in = (unsigned)gx < (unsigned)P.nx && (unsigned)gy < (unsigned)P.ny &&
                                (N == 2 || (unsigned)gz < (unsigned)P.nz);
                bx[e] = in ? __ldg(P.ev + ((long long)gz * P.ny + gy) * P.nx + gx) : 0.f;
            }
        }
        __syncthreads();
        const int nq = sh_nq;
        int G = 32;
        while (G > 2 && nq * G > (int)blockDim.x) G >>= 1;
        const int slots = (int)blockDim.x / G;
        const int gl = tid & (G - 1);
        const int gbase = lane & ~(G - 1);
        const unsigned gmask = G == 32 ? kFull : (((1u << G) - 1u) << gbase);
        for (int k = tid / G; k < nq && !timed_out; k += slots) {
            const int q = sh_q[k];
            const int x = x0 + (q & 31), y = y0 + (q >> 5) % T::TY, z = z0 + (q >> 5) / T::TY;
            const unsigned v = (unsigned)(((long long)z * P.ny + y) * P.nx + x);
            const float dr = __ldg(P.ref + v);
            const float dD = P.dd_frac * (P.local ? dr : dnorm);
            const float inv = 1.0f / dD;
            float best = P.out[v];                       // gamma^2 over the faces through v
            int t = 0;
            while (t < P.ntable) {
                const int idx = t + gl;
                float key = kInf;
                uint32_t off = 0;
                if (idx < P.ntable) {
                    const TableEntry e = idx < kWalkTableCache ? sh_table[idx] : P.table[idx];
                    key = e.key;
                    off = e.off;
                }
                const float k0 = __shfl_sync(gmask, key, gbase);
                if (k0 * k0 >= best) break;               // A1 step 4b-ii, exact
                float cb = best;
                if (key * key < best) {
                    if (P.stats) ++st.keyed;
                    cb = visit_cell_box<N>(P, bx, b0x, b0y, b0z, x, y, z, unpack10(off, 0),
                                           unpack10(off, 10), unpack10(off, 20), key, dr, inv, dnorm,
                                           best, st);
                }
                best = group_min_rt(cb, G, gmask);
                t += G;
            }
            if (t >= P.ntable && best > rc2) {
                // past a truncated table: the exact scan of the remaining box
                if (gl == 0) ++my_over;
                const float g = sqrtf(best);
                const int ax = (int)ceilf(g / P.hn[0]) + 1;
                const int ay = (int)ceilf(g / P.hn[1]) + 1;
                const int az = N == 3 ? (int)ceilf(g / P.hn[2]) + 1 : 0;
                const int xa = max(-ax - 1, -x), xb = min(ax, P.nx - 1 - x);
                const int ya = max(-ay - 1, -y), yb = min(ay, P.ny - 1 - y);
                const int za = N == 3 ? max(-az - 1, -z) : 0, zb = N == 3 ? min(az, P.nz - 1 - z) : 0;
                const long long wx = xb - xa + 1, wy = yb - ya + 1, wz = zb - za + 1;
                const long long tot = wx * wy * wz;
                const float lim = rc2 * 0.99999f;
                float lb = best;
                for (long long b = gl; b < tot; b += G) {
                    const int cx = xa + (int)(b % wx);
                    const long long rr = b / wx;
                    const int cy = ya + (int)(rr % wy);
                    const int cz = za + (int)(rr / wy);
                    const float axd = (float)max(max(cx, -cx - 1), 0) * P.hn[0];
                    const float ayd = (float)max(max(cy, -cy - 1), 0) * P.hn[1];
                    const float azd = N == 3 ? (float)max(max(cz, -cz - 1), 0) * P.hn[2] : 0.f;
                    float k2 = axd * axd + ayd * ayd + azd * azd;
                    if (k2 == 0.f)
                        k2 = P.key0_far2[(cx & 1) | ((cy & 1) << 1) | ((cz & 1) << 2)];
                    if (k2 < lim || k2 >= lb) continue;
                    lb = visit_cell_box<N>(P, bx, b0x, b0y, b0z, x, y, z, cx, cy, cz, sqrtf(k2), dr,
                                           inv, dnorm, lb, st);
                }
                best = group_min_rt(lb, G, gmask);
            }
            if (gl == 0) {
                const float gam = sqrtf(best);
                P.out[v] = gam;
                ++my_eval;
                my_pass += gam <= 1.f;
            }
        }
        // box[buf] and sh_q are free for reuse once every thread is here
        if (__syncthreads_or(timed_out)) {
            if (tid == 0) {
                atomicOr(&P.ctr->flags, kFlagTimeout);
                mbar_wait_bounded(&bar[buf], (parity >> buf) & 1u);
                mbar_wait_bounded(&bar[buf ^ 1], (parity >> (buf ^ 1)) & 1u);
            }
            break;
        }
        i = (unsigned)sh_next[buf];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        my_eval += __shfl_xor_sync(kFull, my_eval, o);
        my_pass += __shfl_xor_sync(kFull, my_pass, o);
        my_over += __shfl_xor_sync(kFull, my_over, o);
        if (P.stats) {
            st.visited += __shfl_xor_sync(kFull, st.visited, o);
            st.pruned += __shfl_xor_sync(kFull, st.pruned, o);
            st.keyed += __shfl_xor_sync(kFull, st.keyed, o);
        }
    }
    if (lane == 0) {
        if (my_eval) atomicAdd(&P.ctr->n_eval, (unsigned long long)my_eval);
        if (my_pass) atomicAdd(&P.ctr->n_pass, (unsigned long long)my_pass);
        if (my_over) atomicAdd(&P.ctr->overflow_count, my_over);
        if (P.stats) {
            atomicAdd(&P.ctr->cells_visited, st.visited);
            atomicAdd(&P.ctr->cells_pruned, st.pruned);
            atomicAdd(&P.ctr->cells_keyed, st.keyed);
        }
    }
}

// --------------------------------------------------------------------------
// k_walk_rows: row-staged walk, one shell warp row per warp at a time
// --------------------------------------------------------------------------

// Halo box of one shell warp row (32 voxels along x): 4 voxels on each side in
// x (the x start stays a multiple of 4 floats for the TMA copy) and RH in y
// and z.  Cells whose corner lies within 3 voxels in x and RH - 1 in y and z
// of the row's voxels read their doses from the box; others global memory.
template <int N>
struct RowBox {
    static constexpr int RH = 3;
    static constexpr int BX = 32 + 8, BY = 2 * RH + 1, BZ = N == 3 ? 2 * RH + 1 : 1;
    static constexpr int ELEMS = BX * BY * BZ;
    static constexpr int STRIDE = (ELEMS + 31) / 32 * 32;
    static_assert(STRIDE * 4 % 128 == 0, "TMA destination must stay 128-byte aligned");
};

// Every warp, independently: take the next row item in cost order, stage the
// row's halo box by one TMA copy into its own buffer (bounded wait), and walk
// the table for the row's queued voxels, G lanes each (G chosen from the
// number of queued voxels so that the warp's lanes are used), with the exact
// stop of Algorithm A1 step 4b-ii and the dose-gap bound.  No block barrier:
// a warp moves on as soon as its row is done, as in k_tail.
template <int N, int MINB>
__global__ void __launch_bounds__(256, MINB)
    k_walk_rows(const __grid_constant__ Problem P, const __grid_constant__ CUtensorMap rmap, int use_tma)
{
    using T = ShellTile<N>;
    using B = RowBox<N>;
    // the warps' boxes in dynamic shared memory (8 x B::STRIDE floats, from a
    // 128-byte boundary: TMA destinations)
    extern __shared__ __align__(128) unsigned char dyn_raw[];
    float* boxes = reinterpret_cast<float*>(dyn_raw + ((128u - (smem_addr(dyn_raw) & 127u)) & 127u));
    __shared__ __align__(8) uint64_t bar[8];
    __shared__ TableEntry sh_table[kWalkTableCache];
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const unsigned nrows = P.ctr->row_count;
    const unsigned long long* order = P.sort_tail ? P.row_sorted : P.row_items;
    const int ncache = min(P.ntable, kWalkTableCache);
    for (int i = tid; i < ncache; i += blockDim.x) sh_table[i] = P.table[i];
    if (tid == 0) {
        for (int i = 0; i < 8; ++i) mbar_init(&bar[i], 1);
        mbar_fence_init();
    }
    __syncthreads();
    const float dnorm = resolve_dnorm(P);
    const float rc2 = P.r_cover * P.r_cover;
    const int ntx = (P.nx + T::TX - 1) / T::TX, nty = (P.ny + T::TY - 1) / T::TY;
    float* bx = boxes + (size_t)w * B::STRIDE;
    unsigned my_eval = 0, my_pass = 0, my_over = 0;
    TailStats st;
    uint32_t phase = 0;
    for (;;) {
        unsigned it = 0;
        if (lane == 0) it = atomicAdd(&P.ctr->row_head, 1u);
        it = __shfl_sync(kFull, it, 0);
        if (it >= nrows) break;
        const unsigned long long item = order[it];
        const unsigned mask = (unsigned)item, rid = (unsigned)(item >> 32);
        const unsigned lt = rid >> 3, wr = rid & 7u;
        const int x0 = (int)(lt % (unsigned)ntx) * T::TX;
        const int y = (int)((lt / (unsigned)ntx) % (unsigned)nty) * T::TY + (int)(wr % T::TY);
        const int z = N == 3 ? (int)(lt / (unsigned)ntx / (unsigned)nty) * T::TZ + (int)(wr / T::TY) : 0;
        const int b0x = x0 - 4, b0y = y - B::RH, b0z = N == 3 ? z - B::RH : 0;
        // ---- the row's halo box ----
        bool ok = true;
        if (use_tma) {
            if (lane == 0) {
                fence_async_shared();                 // the box's previous reads come first
                mbar_arrive_expect_tx(&bar[w], B::ELEMS * (uint32_t)sizeof(float));
                if (N == 3) tma_load_3d(bx, &rmap, b0x, b0y, b0z, &bar[w]);
                else tma_load_2d(bx, &rmap, b0x, b0y, &bar[w]);
            }
            ok = mbar_wait_bounded(&bar[w], phase & 1u);
            ++phase;
        } else {
            for (int e = lane; e < B::ELEMS; e += 32) {
                const int ex_ = e % B::BX, ey_ = (e / B::BX) % B::BY, ez_ = e / (B::BX * B::BY);
                const int gx = b0x + ex_, gy = b0y + ey_, gz = b0z + ez_;
                const bool in = (unsigned)gx < (unsigned)P.nx && (unsigned)gy < (unsigned)P.ny &&
                                (N == 2 || (unsigned)gz < (unsigned)P.nz);
                bx[e] = in ? __ldg(P.ev + ((long long)gz * P.ny + gy) * P.nx + gx) : 0.f;
            }
            __syncwarp();
        }
        if (!__all_sync(kFull, ok)) {
            if (lane == 0) {
                atomicOr(&P.ctr->flags, kFlagTimeout);
                mbar_wait_bounded(&bar[w], (phase - 1) & 1u);     // its copy lands before the warp leaves
            }
            break;
        }
        // ---- the row's queued voxels, G lanes each ----
        const int nq = __popc(mask);
        int G = 32;
        while (G > 2 && nq * G > 32) G >>= 1;
        const int slots = 32 / G;
        const int gl = lane & (G - 1);
        const int gbase = lane & ~(G - 1);
        const unsigned gmask = G == 32 ? kFull : (((1u << G) - 1u) << gbase);
        for (int k = lane / G; k < nq; k += slots) {           // group-uniform
            unsigned mk = mask;                                // the k-th queued voxel of the row
            for (int j = 0; j < k; ++j) mk &= mk - 1u;         // (k < popc(mask): mk stays non-zero)
            const int xi = __ffs(mk) - 1;
            const int x = x0 + xi;
            const unsigned v = (unsigned)(((long long)z * P.ny + y) * P.nx + x);
            const float dr = __ldg(P.ref + v);
            const float dD = P.dd_frac * (P.local ? dr : dnorm);
            const float inv = 1.0f / dD;
            float best = P.out[v];                             // gamma^2 over the faces through v
            int t = 0;
            while (t < P.ntable) {
                const int idx = t + gl;
                float key = kInf;
                uint32_t off = 0;
                if (idx < P.ntable) {
                    const TableEntry e = idx < kWalkTableCache ? sh_table[idx] : P.table[idx];
                    key = e.key;
                    off = e.off;
                }
                const float k0 = __shfl_sync(gmask, key, gbase);
                if (k0 * k0 >= best) break;                     // A1 step 4b-ii, exact
                float cb = best;
                if (key * key < best) {
                    if (P.stats) ++st.keyed;
                    cb = visit_cell_box<N, B>(P, bx, b0x, b0y, b0z, x, y, z, unpack10(off, 0),
                                              unpack10(off, 10), unpack10(off, 20), key, dr, inv,
                                              dnorm, best, st);
                }
                best = group_min_rt(cb, G, gmask);
                t += G;
            }
            if (t >= P.ntable && best > rc2) {
                // past a truncated table: the exact scan of the remaining box
                if (gl == 0) ++my_over;
                const float g = sqrtf(best);
                const int ax = (int)ceilf(g / P.hn[0]) + 1;
                const int ay = (int)ceilf(g / P.hn[1]) + 1;
                const int az = N == 3 ? (int)ceilf(g / P.hn[2]) + 1 : 0;
                const int xa = max(-ax - 1, -x), xb = min(ax, P.nx - 1 - x);
                const int ya = max(-ay - 1, -y), yb = min(ay, P.ny - 1 - y);
                const int za = N == 3 ? max(-az - 1, -z) : 0, zb = N == 3 ? min(az, P.nz - 1 - z) : 0;
                const long long wx = xb - xa + 1, wy = yb - ya + 1, wz = zb - za + 1;
                const long long tot = wx * wy * wz;
                const float lim = rc2 * 0.99999f;
                float lb = best;
                for (long long b = gl; b < tot; b += G) {
                    const int cx = xa + (int)(b % wx);
                    const long long rr = b / wx;
                    const int cy = ya + (int)(rr % wy);
                    const int cz = za + (int)(rr / wy);
                    const float axd = (float)max(max(cx, -cx - 1), 0) * P.hn[0];
                    const float ayd = (float)max(max(cy, -cy - 1), 0) * P.hn[1];
                    const float azd = N == 3 ? (float)max(max(cz, -cz - 1), 0) * P.hn[2] : 0.f;
                    float k2 = axd * axd + ayd * ayd + azd * azd;
                    if (k2 == 0.f)
                        k2 = P.key0_far2[(cx & 1) | ((cy & 1) << 1) | ((cz & 1) << 2)];
                    if (k2 < lim || k2 >= lb) continue;
                    lb = visit_cell_box<N, B>(P, bx, b0x, b0y, b0z, x, y, z, cx, cy, cz, sqrtf(k2), dr,
                                              inv, dnorm, lb, st);
                }
                best = group_min_rt(lb, G, gmask);
            }
            if (gl == 0) {
                const float gam = sqrtf(best);
                P.out[v] = gam;
                ++my_eval;
                my_pass += gam <= 1.f;
            }
        }
        __syncwarp();                                          // the box is free again
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        my_eval += __shfl_xor_sync(kFull, my_eval, o);
        my_pass += __shfl_xor_sync(kFull, my_pass, o);
        my_over += __shfl_xor_sync(kFull, my_over, o);
        if (P.stats) {
            st.visited += __shfl_xor_sync(kFull, st.visited, o);
            st.pruned += __shfl_xor_sync(kFull, st.pruned, o);
            st.keyed += __shfl_xor_sync(kFull, st.keyed, o);
        }
    }
    if (lane == 0) {
        if (my_eval) atomicAdd(&P.ctr->n_eval, (unsigned long long)my_eval);
        if (my_pass) atomicAdd(&P.ctr->n_pass, (unsigned long long)my_pass);
        if (my_over) atomicAdd(&P.ctr->overflow_count, my_over);
        if (P.stats) {
            atomicAdd(&P.ctr->cells_visited, st.visited);
            atomicAdd(&P.ctr->cells_pruned, st.pruned);
            atomicAdd(&P.ctr->cells_keyed, st.keyed);
        }
    }
}

// --------------------------------------------------------------------------
// Launchers
// --------------------------------------------------------------------------

int device_sm_count()
{
    int dev = 0, n = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 1;
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 1;
    return n > 0 ? n : 1;
}

static int grid_for(long long n, int threads, int cap)
{
    long long b = (n + threads - 1) / threads;
    if (b < 1) b = 1;
    if (b > cap) b = cap;
    return (int)b;
}

cudaError_t launch_prepare(const Problem& P, cudaStream_t s, int part)
{
    const int sms = device_sm_count();
    k_prepare<false><<<grid_for((P.nvox + 3) / 4, 256, sms * 8), 256, 0, s>>>(P, nullptr, part);
    return cudaGetLastError();
}

// Distance from the origin to the closed simplex with vertices W[0..nv-1] in
// R^3 (KKT enumeration over its faces), for the host-side shell constants.
static double simplex_dist_host(const double (*W)[3], int nv)
{
    double best = INFINITY;
    for (int mask = 1; mask < (1 << nv); ++mask) {
        int idx[4], k = 0;
        for (int i = 0; i < nv; ++i)
            if (mask & (1 << i)) idx[k++] = i;
        const double* w0 = W[idx[0]];
        double E[3][3], G[3][3], r[3], mu[3] = {0, 0, 0};
        const int m = k - 1;
        for (int i = 0; i < m; ++i)
            for (int a = 0; a < 3; ++a) E[i][a] = W[idx[i + 1]][a] - w0[a];
        for (int i = 0; i < m; ++i) {
            r[i] = 0;
            for (int a = 0; a < 3; ++a) r[i] -= E[i][a] * w0[a];
            for (int j = 0; j < m; ++j) {
                G[i][j] = 0;
                for (int a = 0; a < 3; ++a) G[i][j] += E[i][a] * E[j][a];
            }
        }
        // Gaussian elimination (G is symmetric positive definite here)
        bool okk = true;
        for (int c = 0; c < m && okk; ++c) {
            if (!(fabs(G[c][c]) > 1e-300)) { okk = false; break; }
            for (int rr = c + 1; rr < m; ++rr) {
                const double f = G[rr][c] / G[c][c];
                for (int j = c; j < m; ++j) G[rr][j] -= f * G[c][j];
                r[rr] -= f * r[c];
            }
        }
        if (!okk) continue;
        for (int c = m - 1; c >= 0; --c) {
            double acc = r[c];
            for (int j = c + 1; j < m; ++j) acc -= G[c][j] * mu[j];
            mu[c] = acc / G[c][c];
        }
        double sum = 0;
        bool valid = true;
        for (int i = 0; i < m; ++i) {
            sum += mu[i];
            if (mu[i] < -1e-12) valid = false;
        }
        if (sum > 1 + 1e-12) valid = false;
        if (!valid) continue;
        double d2 = 0;
        for (int a = 0; a < 3; ++a) {
            double p = w0[a];
            for (int i = 0; i < m; ++i) p += mu[i] * E[i][a];
            d2 += p * p;
        }
        best = fmin(best, sqrt(d2));
    }
    return best;
}

void key0_far(const double hn_in[3], int nd, double far[8])
{
    const double hn[3] = {hn_in[0], hn_in[1], nd == 3 ? hn_in[2] : 0.0};
    const int full = (1 << nd) - 1;
    for (int s = 0; s < 8; ++s) far[s] = INFINITY;
    for (int s = 1; s <= full; ++s) {
        const int c[3] = {-(s & 1), -((s >> 1) & 1), -((s >> 2) & 1)};
        double f = INFINITY;
        // every owned face is a chain 0 = u0 < u1 < ... < um of axis masks
        for (int u1 = 1; u1 <= full; ++u1)
            for (int u2 = 0; u2 <= full; ++u2)
                for (int u3 = 0; u3 <= full; ++u3) {
                    int chain[4] = {0, u1, u2, u3};
                    int m = 1;
                    if (u2) {
                        if ((u2 & u1) != u1 || u2 == u1) continue;
                        m = 2;
                        if (u3) {
                            if ((u3 & u2) != u2 || u3 == u2) continue;
                            m = 3;
                        }
                    } else if (u3) {
                        continue;
                    }
                    bool has = false;
                    for (int i = 0; i <= m; ++i) has = has || chain[i] == s;
                    if (has) continue;
                    double W[4][3];
                    for (int i = 0; i <= m; ++i)
                        for (int a = 0; a < 3; ++a)
                            W[i][a] = (a < nd) ? (c[a] + ((chain[i] >> a) & 1)) * hn[a] : 0.0;
                    f = fmin(f, simplex_dist_host(W, m + 1));
                }
        double W[1][3];                       // the cell's own corner vertex
        for (int a = 0; a < 3; ++a) W[0][a] = (a < nd) ? c[a] * hn[a] : 0.0;
        f = fmin(f, simplex_dist_host(W, 1));
        far[s] = f * (1.0 - 1e-6);            // absorbs the rounding of the projection
    }
}

using EncodeFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*,
                              const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                              const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                              CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// The driver's tensor-map encoder (looked up once), or null.
static EncodeFn tensor_map_encoder()
{
    static EncodeFn encode = nullptr;
    static bool looked_up = false;
    if (!looked_up) {
        looked_up = true;
        void* fn = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault,
                                             &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            encode = (EncodeFn)fn;
    }
    return encode;
}

bool encode_bf16_2d(CUtensorMap* map, const void* base, unsigned long long inner,
                    unsigned long long rows, unsigned long long row_stride_bytes,
                    unsigned box_inner, unsigned box_rows, bool swizzle)
{
    const EncodeFn encode = tensor_map_encoder();
    if (!encode || ((uintptr_t)base & 15u) || (row_stride_bytes & 15u) || (box_inner * 2) % 16) return false;
    const cuuint64_t dims[2] = {(cuuint64_t)inner, (cuuint64_t)rows};
    const cuuint64_t strides[1] = {(cuuint64_t)row_stride_bytes};
    const cuuint32_t box[2] = {(cuuint32_t)box_inner, (cuuint32_t)box_rows};
    const cuuint32_t es[2] = {1, 1};
    std::memset(map, 0, sizeof(*map));
    return encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box,
                  es, CU_TENSOR_MAP_INTERLEAVE_NONE,
                  swizzle ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_NONE,
                  swizzle ? CU_TENSOR_MAP_L2_PROMOTION_L2_256B : CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Tensor map of the evaluation dose with a tile box of (bx, by, bz) floats,
// zeros or NaN (nan_fill) outside the grid; false when TMA cannot be used for
// it.
static bool encode_box_map(const Problem& P, CUtensorMap* map, int bx, int by, int bz, bool nan_fill = false)
{
    const EncodeFn encode = tensor_map_encoder();
    if (!encode) return false;
    const CUtensorMapFloatOOBfill fill =
        nan_fill ? CU_TENSOR_MAP_FLOAT_OOB_FILL_NAN_REQUEST_ZERO_FMA : CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE;
    if (((uintptr_t)P.ev & 15u) != 0 || (P.nx % 4) != 0) return false;   // TMA alignment rules
    if (P.ndim == 3) {
        const cuuint64_t dims[3] = {(cuuint64_t)P.nx, (cuuint64_t)P.ny, (cuuint64_t)P.nz};
        const cuuint64_t strides[2] = {(cuuint64_t)P.nx * 4, (cuuint64_t)P.nx * P.ny * 4};
        const cuuint32_t box[3] = {(cuuint32_t)bx, (cuuint32_t)by, (cuuint32_t)bz};
        const cuuint32_t es[3] = {1, 1, 1};
        return encode(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, (void*)P.ev, dims, strides, box, es,
                      CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                      CU_TENSOR_MAP_L2_PROMOTION_L2_128B, fill) == CUDA_SUCCESS;
    }
    const cuuint64_t dims[2] = {(cuuint64_t)P.nx, (cuuint64_t)P.ny};
    const cuuint64_t strides[1] = {(cuuint64_t)P.nx * 4};
    const cuuint32_t box[2] = {(cuuint32_t)bx, (cuuint32_t)by};
    const cuuint32_t es[2] = {1, 1};
    return encode(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, (void*)P.ev, dims, strides, box, es,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                  CU_TENSOR_MAP_L2_PROMOTION_L2_128B, fill) == CUDA_SUCCESS;
}

// The shell of a run uses k_shell_w (warp tiles) unless a staged walk needs
// k_shell's tile layout for its queue.
static bool warp_tiled(const Problem& P) { return !P.tile_mask && !P.row_items; }

bool encode_tile_map(const Problem& P, CUtensorMap* map)
{
    if (warp_tiled(P))
        return P.ndim == 3 ? encode_box_map(P, map, WarpTile<3>::BX, WarpTile<3>::BY, WarpTile<3>::BZ, true)
                           : encode_box_map(P, map, WarpTile<2>::BX, WarpTile<2>::BY, 1, true);
    return P.ndim == 3 ? encode_box_map(P, map, ShellTile<3>::BX, ShellTile<3>::BY, ShellTile<3>::BZ, true)
                       : encode_box_map(P, map, ShellTile<2>::BX, ShellTile<2>::BY, 1, true);
}

template <class T>
static long long tile_count(const Problem& P)
{
    const long long nxy = (long long)((P.nx + T::TX - 1) / T::TX) * ((P.ny + T::TY - 1) / T::TY);
    return P.ndim == 3 ? nxy * ((P.nz + T::TZ - 1) / T::TZ) : nxy;
}

int block_tiles(const Problem& P)
{
    const long long tiles = P.ndim == 3 ? tile_count<ShellTile<3>>(P) : tile_count<ShellTile<2>>(P);
    return tiles > 0x3fffffffLL ? -1 : (int)tiles;
}

int shell_tiles(const Problem& P)
{
    if (!warp_tiled(P)) return block_tiles(P);
    const long long tiles = P.ndim == 3 ? tile_count<WarpTile<3>>(P) : tile_count<WarpTile<2>>(P);
    return tiles > 0x3fffffffLL ? -1 : (int)tiles;
}

// k_shell with its register budget chosen for `per_sm` resident blocks.
template <int N, bool BATCH>
static void launch_shell_k(int per_sm, unsigned grid, cudaStream_t s, const Problem& P,
                           const CUtensorMap& map, int use_tma, int t_first, int tiles,
                           unsigned* next, const SlabGate& gate, const BatchDesc* bd)
{
    switch (per_sm) {
    case 1: k_shell<N, 1, BATCH><<<grid, 256, 0, s>>>(P, map, use_tma, t_first, tiles, next, gate, bd); break;
    case 2: k_shell<N, 2, BATCH><<<grid, 256, 0, s>>>(P, map, use_tma, t_first, tiles, next, gate, bd); break;
    case 3: k_shell<N, 3, BATCH><<<grid, 256, 0, s>>>(P, map, use_tma, t_first, tiles, next, gate, bd); break;
    default: k_shell<N, 4, BATCH><<<grid, 256, 0, s>>>(P, map, use_tma, t_first, tiles, next, gate, bd); break;
    }
}

bool shell_gate_ok(const Problem& P)
{
    CUtensorMap map;
    return encode_tile_map(P, &map);
}

template <class T>
static void layers_of(const Problem& P, int* tiles_per_layer, int* layers, int* layer_depth)
{
    *tiles_per_layer = ((P.nx + T::TX - 1) / T::TX) * ((P.ny + T::TY - 1) / T::TY);
    *layers = P.ndim == 3 ? (P.nz + T::TZ - 1) / T::TZ : 1;
    *layer_depth = P.ndim == 3 ? T::TZ : 1;
}

void shell_layers(const Problem& P, int* tiles_per_layer, int* layers, int* layer_depth)
{
    if (warp_tiled(P)) {
        if (P.ndim == 3) layers_of<WarpTile<3>>(P, tiles_per_layer, layers, layer_depth);
        else layers_of<WarpTile<2>>(P, tiles_per_layer, layers, layer_depth);
    } else {
        if (P.ndim == 3) layers_of<ShellTile<3>>(P, tiles_per_layer, layers, layer_depth);
        else layers_of<ShellTile<2>>(P, tiles_per_layer, layers, layer_depth);
    }
}

template <int N, bool BATCH>
static void launch_shell_w_k(int per_sm, unsigned grid, cudaStream_t s, const Problem& P,
                             const CUtensorMap& map, int use_tma, int t_first, int tiles,
                             unsigned* next, const SlabGate& gate, const BatchDesc* bd)
{
    switch (per_sm) {
    case 1: launch_next(k_shell_w<N, 1, BATCH>, grid, 256, 0, s, P, map, use_tma, t_first, tiles, next, gate, bd); break;
    case 2: launch_next(k_shell_w<N, 2, BATCH>, grid, 256, 0, s, P, map, use_tma, t_first, tiles, next, gate, bd); break;
    case 3: launch_next(k_shell_w<N, 3, BATCH>, grid, 256, 0, s, P, map, use_tma, t_first, tiles, next, gate, bd); break;
    default: launch_next(k_shell_w<N, 4, BATCH>, grid, 256, 0, s, P, map, use_tma, t_first, tiles, next, gate, bd); break;
    }
}

cudaError_t launch_shell_range(const Problem& P, int tile_first, int tile_end, int slot,
                               const SlabGate& gate, cudaStream_t s)
{
    if (slot < 0 || slot >= kShellSlots) return cudaErrorInvalidValue;
    CUtensorMap map;
    std::memset(&map, 0, sizeof(map));
    const int use_tma = encode_tile_map(P, &map) ? 1 : 0;
    if (gate.flag && (!use_tma || gate.depth <= 0)) return cudaErrorInvalidValue;
    const int sms = device_sm_count();
    const int per_sm = std::min(4, std::max(1, P.shell_minblocks));
    const int tiles = shell_tiles(P);
    if (tiles < 0 || tile_first < 0 || tile_end > tiles || tile_first > tile_end)
        return cudaErrorInvalidValue;
    if (tile_first == tile_end) return cudaSuccess;
    unsigned* next = &P.ctr->shell_next[slot];
    if (warp_tiled(P)) {
        // eight tiles per block in flight
        const unsigned grid = (unsigned)std::min<long long>((tile_end - tile_first + 7) / 8,
                                                            (long long)sms * per_sm);
        if (P.ndim == 3)
            launch_shell_w_k<3, false>(per_sm, grid, s, P, map, use_tma, tile_first, tile_end, next, gate,
                                       nullptr);
        else
            launch_shell_w_k<2, false>(per_sm, grid, s, P, map, use_tma, tile_first, tile_end, next, gate,
                                       nullptr);
        return cudaGetLastError();
    }
    const unsigned grid =
        (unsigned)std::min<long long>(tile_end - tile_first, (long long)sms * per_sm);
    if (P.ndim == 3)
        launch_shell_k<3, false>(per_sm, grid, s, P, map, use_tma, tile_first, tile_end, next, gate,
                                 nullptr);
    else
        launch_shell_k<2, false>(per_sm, grid, s, P, map, use_tma, tile_first, tile_end, next, gate,
                                 nullptr);
    return cudaGetLastError();
}

cudaError_t launch_shell(const Problem& P, cudaStream_t s)
{
    const int tiles = shell_tiles(P);
    if (tiles < 0) return cudaErrorInvalidValue;
    return launch_shell_range(P, 0, tiles, 0, SlabGate{nullptr, 0u, 0}, s);
}

// Copy the final gamma of every queued voxel from the device map into a
// host map (through its device-mapped pointer) that already holds the rest.
// Block 0 also copies the run's final counters into `host_ctr` (mapped), so
// that reading them needs no copy of its own.
__global__ void __launch_bounds__(256) k_patch_host(const __grid_constant__ Problem P, float* host_out,
                                                    Counters* host_ctr)
{
    if (blockIdx.x == 0 && host_ctr) {
        const unsigned* src = (const unsigned*)P.ctr;
        unsigned* dst = (unsigned*)host_ctr;
        for (unsigned i = threadIdx.x; i < sizeof(Counters) / 4; i += blockDim.x) dst[i] = src[i];
    }
    const unsigned n = min(P.ctr->tail_count, P.tail_cap);
    const unsigned stride = gridDim.x * blockDim.x;
    for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        const unsigned v = P.tail_raw[i];
        host_out[v] = P.out[v];
    }
}

cudaError_t launch_patch_host(const Problem& P, float* host_out_mapped, Counters* host_ctr_mapped,
                              cudaStream_t s)
{
    k_patch_host<<<device_sm_count() * 4, 256, 0, s>>>(P, host_out_mapped, host_ctr_mapped);
    return cudaGetLastError();
}

cudaError_t launch_plane_seed(const Problem& P, cudaStream_t s)
{
    if (!P.plane_raw) return cudaSuccess;
    const int t = seed_threads(P.ndim, false), grid = grid_for(P.nvox, t, device_sm_count() * 8);
    if (P.ndim == 3) launch_next(k_plane_seed<3, false>, grid, t, 0, s, P, nullptr, nullptr);
    else launch_next(k_plane_seed<2, false>, grid, t, 0, s, P, nullptr, nullptr);
    return cudaGetLastError();
}

cudaError_t launch_order_tail(const Problem& P, cudaStream_t s)
{
    if (!P.sort_tail) return cudaSuccess;
    launch_next(k_scatter, grid_for(P.nvox, 256, device_sm_count() * 8), 256, 0, s, P);
    return cudaGetLastError();
}

template <int N, int MINB, bool BATCH>
static void launch_tail_g(const Problem& P, const BatchDesc* bd, int G, int grid, cudaStream_t s)
{
    switch (G) {
    case 2: k_tail<N, 2, MINB, BATCH><<<grid, 256, 0, s>>>(P, bd); break;
    case 4: k_tail<N, 4, MINB, BATCH><<<grid, 256, 0, s>>>(P, bd); break;
    case 8: k_tail<N, 8, MINB, BATCH><<<grid, 256, 0, s>>>(P, bd); break;
    case 16: k_tail<N, 16, MINB, BATCH><<<grid, 256, 0, s>>>(P, bd); break;
    default: k_tail<N, 32, MINB, BATCH><<<grid, 256, 0, s>>>(P, bd); break;
    }
}

// k_tail with G lanes per queued voxel and its register budget sized for
// `per_sm` resident blocks (1 to 3; 3 spills a little and is still the
// fastest on the benchmark workload).
template <int N, bool BATCH>
static void launch_tail_n(const Problem& P, const BatchDesc* bd, int G, int per_sm, int grid,
                          cudaStream_t s)
{
    if (per_sm >= 3) launch_tail_g<N, 3, BATCH>(P, bd, G, grid, s);
    else if (per_sm == 2) launch_tail_g<N, 2, BATCH>(P, bd, G, grid, s);
    else launch_tail_g<N, 1, BATCH>(P, bd, G, grid, s);
}

cudaError_t launch_tail(const Problem& P, int lanes_per_voxel, int tail_minblocks, cudaStream_t s)
{
    const int sms = device_sm_count();
    const int grid = sms * 8;      // persistent: enough warps to fill every SM
    if (P.ndim == 3) launch_tail_n<3, false>(P, nullptr, lanes_per_voxel, tail_minblocks, grid, s);
    else launch_tail_n<2, false>(P, nullptr, lanes_per_voxel, tail_minblocks, grid, s);
    return cudaGetLastError();
}

template <int N, bool BATCH>
static void launch_tail_cq_n(const Problem& P, const BatchDesc* bd, int per_sm, cudaStream_t s)
{
    const int sms = device_sm_count();
    // persistent: one wave of resident blocks (fewer where even a voxel per
    // lane group would leave blocks without work)
    const int grid = BATCH ? sms * per_sm : grid_for(P.nvox, cq_threads(per_sm) / 32, sms * per_sm);
    if (per_sm >= 4) launch_next(k_tail_cq<N, 4, BATCH>, grid, cq_threads(4), 0, s, P, bd);
    else if (per_sm == 3) launch_next(k_tail_cq<N, 3, BATCH>, grid, cq_threads(3), 0, s, P, bd);
    else if (per_sm == 2) launch_next(k_tail_cq<N, 2, BATCH>, grid, cq_threads(2), 0, s, P, bd);
    else launch_next(k_tail_cq<N, 1, BATCH>, grid, cq_threads(1), 0, s, P, bd);
    // (a warp per listed voxel; most often there is none)
    launch_next(k_tail_fix<N, BATCH>, BATCH ? sms * 2 : grid_for(P.nvox, 8, sms * 2), 256, 0, s, P, bd);
}

cudaError_t launch_tail_cq(const Problem& P, int tail_minblocks, cudaStream_t s)
{
    if (!P.fix_list || !P.plane_raw) return cudaErrorInvalidValue;
    const int per_sm = std::min(4, std::max(1, tail_minblocks));
    if (P.ndim == 3) launch_tail_cq_n<3, false>(P, nullptr, per_sm, s);
    else launch_tail_cq_n<2, false>(P, nullptr, per_sm, s);
    return cudaGetLastError();
}

cudaError_t launch_order_tiles(const Problem& P, cudaStream_t s)
{
    if (!P.sort_tail) return cudaSuccess;
    k_scatter_tiles<<<device_sm_count() * 2, 256, 0, s>>>(P);
    return cudaGetLastError();
}

template <int N>
static void launch_walk_n(const Problem& P, const CUtensorMap& map, int use_tma, int per_sm,
                          int grid, cudaStream_t s)
{
    if (per_sm >= 3) k_walk<N, 3><<<grid, 256, 0, s>>>(P, map, use_tma);
    else if (per_sm == 2) k_walk<N, 2><<<grid, 256, 0, s>>>(P, map, use_tma);
    else k_walk<N, 1><<<grid, 256, 0, s>>>(P, map, use_tma);
}

cudaError_t launch_walk(const Problem& P, int walk_minblocks, cudaStream_t s)
{
    if (!P.tile_mask) return cudaErrorInvalidValue;
    CUtensorMap map;
    std::memset(&map, 0, sizeof(map));
    int use_tma;
    if (P.ndim == 3) use_tma = encode_box_map(P, &map, WalkBox<3>::BX, WalkBox<3>::BY, WalkBox<3>::BZ);
    else use_tma = encode_box_map(P, &map, WalkBox<2>::BX, WalkBox<2>::BY, 1);
    const int per_sm = std::min(3, std::max(1, walk_minblocks));
    const int grid = device_sm_count() * per_sm;     // persistent; blocks past the tile list exit
    if (P.ndim == 3) launch_walk_n<3>(P, map, use_tma, per_sm, grid, s);
    else launch_walk_n<2>(P, map, use_tma, per_sm, grid, s);
    return cudaGetLastError();
}

cudaError_t launch_order_rows(const Problem& P, cudaStream_t s)
{
    if (!P.sort_tail) return cudaSuccess;
    k_scatter_rows<<<device_sm_count() * 2, 256, 0, s>>>(P);
    return cudaGetLastError();
}

template <int N, int MINB>
static cudaError_t launch_walk_rows_k(const Problem& P, const CUtensorMap& map, int use_tma, int grid,
                                      cudaStream_t s)
{
    const int smem = 8 * RowBox<N>::STRIDE * (int)sizeof(float) + 128;
    cudaError_t e = cudaFuncSetAttribute(k_walk_rows<N, MINB>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    k_walk_rows<N, MINB><<<grid, 256, smem, s>>>(P, map, use_tma);
    return cudaGetLastError();
}

template <int N>
static cudaError_t launch_walk_rows_n(const Problem& P, const CUtensorMap& map, int use_tma, int per_sm,
                                      int grid, cudaStream_t s)
{
    if (per_sm >= 3) return launch_walk_rows_k<N, 3>(P, map, use_tma, grid, s);
    if (per_sm == 2) return launch_walk_rows_k<N, 2>(P, map, use_tma, grid, s);
    return launch_walk_rows_k<N, 1>(P, map, use_tma, grid, s);
}

cudaError_t launch_walk_rows(const Problem& P, int walk_minblocks, cudaStream_t s)
{
    if (!P.row_items) return cudaErrorInvalidValue;
    CUtensorMap map;
    std::memset(&map, 0, sizeof(map));
    int use_tma;
    if (P.ndim == 3) use_tma = encode_box_map(P, &map, RowBox<3>::BX, RowBox<3>::BY, RowBox<3>::BZ);
    else use_tma = encode_box_map(P, &map, RowBox<2>::BX, RowBox<2>::BY, 1);
    const int per_sm = std::min(3, std::max(1, walk_minblocks));
    const int grid = device_sm_count() * per_sm;     // persistent
    return P.ndim == 3 ? launch_walk_rows_n<3>(P, map, use_tma, per_sm, grid, s)
                       : launch_walk_rows_n<2>(P, map, use_tma, per_sm, grid, s);
}

// --------------------------------------------------------------------------
// Batched launches (one group = pairs of one dimension)
// --------------------------------------------------------------------------

cudaError_t launch_batch_prepare(const BatchGroup& g, cudaStream_t s)
{
    if (g.npairs <= 0) return cudaSuccess;
    const int sms = device_sm_count();
    const int bx = grid_for(g.max_nvox, 256, std::max(1, sms * 8 / std::max(1, g.npairs)) + 1);
    Problem dummy{};
    // (the run's first kernel: a plain launch; the shell checks the evaluation dose)
    k_prepare<true><<<dim3(bx, g.npairs), 256, 0, s>>>(dummy, g.desc, 1);
    return cudaGetLastError();
}

cudaError_t launch_batch_shell(const BatchGroup& g, int shell_minblocks, cudaStream_t s)
{
    if (g.npairs <= 0 || g.total_tiles <= 0) return cudaSuccess;
    const int sms = device_sm_count();
    const int per_sm = std::min(4, std::max(1, shell_minblocks));
    const unsigned grid = (unsigned)std::min<long long>((g.total_tiles + 7) / 8, (long long)sms * per_sm);
    Problem dummy{};
    CUtensorMap map;
    std::memset(&map, 0, sizeof(map));
    if (g.ndim == 3) launch_shell_w_k<3, true>(per_sm, grid, s, dummy, map, 0, 0, g.total_tiles, g.shell_next,
                                          SlabGate{nullptr, 0u, 0}, g.desc);
    else launch_shell_w_k<2, true>(per_sm, grid, s, dummy, map, 0, 0, g.total_tiles, g.shell_next,
                                          SlabGate{nullptr, 0u, 0}, g.desc);
    return cudaGetLastError();
}

cudaError_t launch_batch_plane_seed(const BatchGroup& g, cudaStream_t s)
{
    if (g.npairs <= 0) return cudaSuccess;
    Problem dummy{};
    const int t = seed_threads(g.ndim, true);
    const unsigned grid = g.nblocks * (256u / (unsigned)t);
    if (g.ndim == 3) launch_next(k_plane_seed<3, true>, grid, t, 0, s, dummy, g.desc, g.blocks);
    else launch_next(k_plane_seed<2, true>, grid, t, 0, s, dummy, g.desc, g.blocks);
    return cudaGetLastError();
}

cudaError_t launch_batch_order(const BatchGroup& g, cudaStream_t s)
{
    if (g.npairs <= 0) return cudaSuccess;
    launch_next(k_bucket_scan_batch, 1, 256, 0, s, g.desc);
    launch_next(k_scatter_batch, g.nblocks, 256, 0, s, g.desc, g.blocks);
    return cudaGetLastError();
}

cudaError_t launch_batch_tail(const BatchGroup& g, int walk, int lanes_per_voxel, int tail_minblocks,
                              cudaStream_t s)
{
    if (g.npairs <= 0) return cudaSuccess;
    const int sms = device_sm_count();
    Problem dummy{};
    if (walk == 3) {
        const int per_sm = std::min(4, std::max(1, tail_minblocks));
        if (g.ndim == 3) launch_tail_cq_n<3, true>(dummy, g.desc, per_sm, s);
        else launch_tail_cq_n<2, true>(dummy, g.desc, per_sm, s);
        return cudaGetLastError();
    }
    if (g.ndim == 3) launch_tail_n<3, true>(dummy, g.desc, lanes_per_voxel, tail_minblocks, sms * 8, s);
    else launch_tail_n<2, true>(dummy, g.desc, lanes_per_voxel, tail_minblocks, sms * 8, s);
    return cudaGetLastError();
}

}  // namespace gk
