// Reference and evaluation doses on different grids (each grid with its own
// shape, spacing and origin; same axes).  Eq. 1 as for coincident grids: the
// evaluation surface is the Freudenthal interpolant of the evaluation grid,
// and each reference voxel searches it from its own position, which is in
// general not an evaluation node.
//
//   k_grid_prepare  max of the reference dose (the global dose norm) and a
//                   finite check of both grids
//   k_grid_seed     the evaluated reference voxels, each with a bound from the
//                   affine parts of a few cells around it
//   k_grid_cq       the walk of the cell table in key order from the evaluation
//                   cell that holds the voxel (clamped to the grid), with the
//                   exact stop of A1 step 4b-ii; a cell is skipped when the
//                   distance from the reference point to its box, with its
//                   dose gap, or its affine part already keeps it at the
//                   running gamma, else every face of it is evaluated
//                   (real-valued cell offsets)
//   k_grid_walk     the voxels with a near-singular cell (FP64 redo) or a walk
//                   past a truncated table (box scan), a warp each
//
// The table is keyed by the distance between the box of the voxel's cell and
// the box of the other cell, divided by the DTA: a lower bound on the distance
// from any point of the first box to any face of the second.  It stays a
// lower bound for a voxel outside the evaluation grid, whose clamped cell is
// the grid cell nearest to it: per axis, its distance to any cell is at least
// that cell's gap to the clamped one.
#include <cuda_runtime.h>
#include <math.h>

#include <algorithm>
#include <cmath>
#include <vector>

#include "../../include/gamma.h"
#include "gamma_cell.cuh"
#include "gamma_internal.h"
#include "gamma_launch.cuh"
#include "gamma_plane.cuh"

namespace gk {

// Table key of cell offset c along one axis, in cells: the smallest distance
// from a point in its own cell to cell c.  Variant 8 holds for any point of
// the cell (and, per axis, for a point outside the grid, from its clamped
// cell); variants 0-7 for a point in one half of its cell per axis (bit a of
// the variant: the upper half [0.5, 1) of axis a, else the lower [0, 0.5)).
__host__ __device__ inline double grid_axis_key(int c, int variant, int a)
{
    if (variant == 8 || c == 0) return c == 0 ? 0.0 : (double)(c > 0 ? c - 1 : -c - 1);
    const bool upper = (variant >> a) & 1;
    return c > 0 ? (double)(c - 1) + (upper ? 0.0 : 0.5) : (double)(-c - 1) + (upper ? 0.5 : 0.0);
}

// The table variant for a point at fraction fr of its cell (0-7: its half of
// the cell per axis; 8: outside [0, 1) on some axis, beyond the grid).
__device__ __forceinline__ int grid_variant(const float (&fr)[3], int nd)
{
    int v = 0;
    for (int a = 0; a < nd; ++a) {
        if (!(fr[a] >= 0.f && fr[a] < 1.f)) return 8;
        if (fr[a] >= 0.5f) v |= 1 << a;
    }
    return v;
}

// --------------------------------------------------------------------------
// Prepare: dose norm over the reference grid, finite checks
// --------------------------------------------------------------------------

__global__ void __launch_bounds__(256) k_grid_prepare(const __grid_constant__ GridProblem G)
{
    grid_release();
    grid_wait();
    float m = -kInf;
    bool bad = false;
    const long long stride = (long long)gridDim.x * blockDim.x;
    const long long first = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    for (long long i = first; i < G.nref; i += stride) {
        const float r = __ldg(G.ref + i);
        bad |= !isfinite(r);
        m = fmaxf(m, r);
    }
    for (long long i = first; i < G.neval; i += stride) bad |= !isfinite(__ldg(G.ev + i));
    __shared__ float sh_m[8];                  // one atomic per block
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(kFull, m, o));
    if ((threadIdx.x & 31) == 0) sh_m[threadIdx.x >> 5] = m;
    bad = __syncthreads_or(bad);
    if (threadIdx.x == 0) {
        for (int w = 1; w < (int)(blockDim.x >> 5); ++w) m = fmaxf(m, sh_m[w]);
        atomicMax(&G.ctr->dnorm_enc, fenc(m));
        if (bad) atomicOr(&G.ctr->flags, kFlagNonFinite);
    }
}

// --------------------------------------------------------------------------
// The walk
// --------------------------------------------------------------------------

// Every face of evaluation cell p (its lower corner, grid coordinates) for a
// reference point at u (evaluation voxel units, real), unless the cell's
// key and dose range already keep it at least sqrt(best) away.
template <int N>
__device__ __forceinline__ float grid_cell(const GridProblem& G, const int (&p)[3],
                                           const double (&u)[3], const float (&cf)[3], float key,
                                           float dr, float inv, float dnorm, float best)
{
    const long long sy = G.en[0], sz = (long long)G.en[0] * G.en[1];
    const long long pidx = (long long)p[2] * sz + (long long)p[1] * sy + p[0];
    const bool ex = p[0] + 1 < G.en[0], ey = p[1] + 1 < G.en[1], ez = N == 3 && p[2] + 1 < G.en[2];
    float q[8];
    uint32_t ok = 0;
#pragma unroll
    for (int w = 0; w < 8; ++w) {
        q[w] = kNaN;
        if (w < (1 << N)) {
            const bool present = (!(w & 1) || ex) && (!(w & 2) || ey) && (!(w & 4) || ez);
            if (present) {
                const long long o = pidx + ((w & 1) ? 1 : 0) + ((w & 2) ? sy : 0) + ((w & 4) ? sz : 0);
                q[w] = (__ldg(G.ev + o) - dr) * inv;
                ok |= 1u << w;
            }
        }
    }
    float qmin = kInf, qmax = -kInf;
#pragma unroll
    for (int w = 0; w < 8; ++w)
        if ((ok >> w) & 1u) {
            qmin = fminf(qmin, q[w]);
            qmax = fmaxf(qmax, q[w]);
        }
    const float gap = qmin > 0.f ? qmin : (qmax < 0.f ? -qmax : 0.f);
    if (fmaf(gap, gap, key * key) >= best) return best;
    // the cell's corner relative to the point (voxel units), cf = d - fraction
    CellGeom<float> g;
    cell_geom<N, float>(cf[0], cf[1], N == 3 ? cf[2] : 0.f, G.mt, g);
    bool ill = false;
    const float dmax = G.tau > 0.f ? 0.99f * rsqrtf(G.tau) : kInf;
    float cb = cell_min_d2<N, float>(q, g, G.mt, dmax, kInf, ill);
    if (ill) ill = cell_gram_ill<N>(q, ok, G.mt.kappa, G.tau);
    if (ill) {
        const double drd = dr;
        const double invd = 1.0 / ((double)G.dd_frac * (G.local ? drd : (double)dnorm));
        cb = cell_redo_f64<N, double>(G.ev, pidx, sy, sz, ok, (double)p[0] - u[0],
                                      (double)p[1] - u[1], N == 3 ? (double)p[2] - u[2] : 0.0,
                                      drd, invd, G.mtd, &G.ctr->fp64_cells);
    }
    return fminf(best, cb);
}

// A warp per reference voxel over those that k_grid_cq left in walk_list, each
// from an infinite bound.  The table starts with the voxel's own cell (offset
// 0), so the first round of 32 cells gives a finite bound; later cells are
// skipped when the distance from the point itself to the cell's box, with the
// dose gap, already reaches the running gamma.  The exact stop (A1 step 4b-ii)
// takes the table's key.
template <int N>
__global__ void __launch_bounds__(256, 2) k_grid_walk(const __grid_constant__ GridProblem G)
{
    grid_wait();                       // (the last kernel: nothing is released early)
    const int lane = threadIdx.x & 31;
    const float dnorm = G.dose_norm > 0.f ? G.dose_norm : fdec(G.ctr->dnorm_enc);
    unsigned my_eval = 0, my_pass = 0, my_over = 0;
    const long long nwarps = (long long)gridDim.x * (blockDim.x >> 5);
    const long long nwork = (long long)G.ctr->fix_count;
    for (long long i = (long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); i < nwork;
         i += nwarps) {                                      // warp-uniform
        const long long v = (long long)G.walk_list[i];
        const float dr = __ldg(G.ref + v);
        const long long ix[3] = {v % G.rn[0], (v / G.rn[0]) % G.rn[1], v / ((long long)G.rn[0] * G.rn[1])};
        // the point in evaluation voxel units: its cell c0 (clamped to the
        // grid) and its position fr in that cell (outside [0, 1) beyond the
        // grid), from FP64 on one lane
        double u[3] = {0.0, 0.0, 0.0};
        int c0[3] = {0, 0, 0};
        float fr[3] = {0.f, 0.f, 0.f}, ehf[3] = {0.f, 0.f, 0.f};
#pragma unroll
        for (int a = 0; a < N; ++a) {
            double ua = 0.0, f = 0.0;
            if (lane == 0) {
                ua = (G.ro[a] + (double)ix[a] * G.rh[a] - G.eo[a]) / G.eh[a];
                f = fmin(fmax(floor(ua), 0.0), (double)(G.en[a] - 2));
            }
            u[a] = __shfl_sync(kFull, ua, 0);
            c0[a] = (int)__shfl_sync(kFull, f, 0);
            fr[a] = (float)(u[a] - (double)c0[a]);
            ehf[a] = (float)G.eh[a];
        }
        const float dD = G.dd_frac * (G.local ? dr : dnorm);
        const float inv = 1.0f / dD;
        // the table for the point's half of its cell per axis
        const int var = grid_variant(fr, N);
        const TableEntry* table = G.table + G.toff[var];
        const int ntable = G.tlen[var];
        const float rc2 = G.tcover[var] * G.tcover[var];
        float best = kInf;
        int t = 0;
        while (t < ntable) {
            const int idx = t + lane;
            float key = kInf;
            uint32_t off = 0;
            if (idx < ntable) {
                const TableEntry e = table[idx];
                key = e.key;
                off = e.off;
            }
            const float k0 = __shfl_sync(kFull, key, 0);
            if (k0 * k0 >= best) break;                       // A1 step 4b-ii, exact
            float cb = best;
            if (key * key < best) {
                const int d[3] = {unpack10(off, 0), unpack10(off, 10), N == 3 ? unpack10(off, 20) : 0};
                const int p[3] = {c0[0] + d[0], c0[1] + d[1], c0[2] + d[2]};
                bool in = true;
                // the distance from the point to the cell's box: a lower bound
                // in FP32 from the integer offset and the point's fraction,
                // each axis lowered by its rounding (4 ulp of its operands) and
                // the sum by 1e-5
                float k2 = 0.f;
#pragma unroll
                for (int a = 0; a < N; ++a) {
                    in = in && p[a] >= 0 && p[a] < G.en[a];
                    const float lo = (float)d[a] - fr[a], hi = fr[a] - (float)(d[a] + 1);
                    const float slack = 4.8e-7f * (fabsf(fr[a]) + fabsf((float)d[a]) + 2.f);
                    const float gap = fmaxf(fmaxf(lo, hi) - slack, 0.f) * ehf[a];
                    k2 = fmaf(gap, gap, k2);
                }
                k2 *= 0.99999f;
                if (in && k2 < best) {
                    const float cf[3] = {(float)d[0] - fr[0], (float)d[1] - fr[1], (float)d[2] - fr[2]};
                    cb = grid_cell<N>(G, p, u, cf, sqrtf(fmaxf(k2, key * key)), dr, inv, dnorm, best);
                }
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) cb = fminf(cb, __shfl_xor_sync(kFull, cb, o));
            best = cb;
            t += 32;
        }
        if (t >= ntable && best > rc2) {
            // past a truncated table: every remaining cell of the search box
            if (lane == 0) ++my_over;
            const float gm = sqrtf(best);
            int dlo[3] = {0, 0, 0}, dhi[3] = {0, 0, 0};
#pragma unroll
            for (int a = 0; a < N; ++a) {
                const float l = gm / (float)G.eh[a] + 2.f;
                const int lim = l < (float)G.en[a] ? (int)ceilf(l) : G.en[a];
                dlo[a] = max(-lim, -c0[a]);
                dhi[a] = min(lim, G.en[a] - 1 - c0[a]);
            }
            const long long wx = dhi[0] - dlo[0] + 1, wy = dhi[1] - dlo[1] + 1, wz = dhi[2] - dlo[2] + 1;
            const long long tot = wx * wy * wz;
            const float cut = rc2 * 0.99999f;
            float lb = best;
            for (long long b = lane; b < tot; b += 32) {
                const int d[3] = {dlo[0] + (int)(b % wx), dlo[1] + (int)((b / wx) % wy), dlo[2] + (int)(b / (wx * wy))};
                const int p[3] = {c0[0] + d[0], c0[1] + d[1], c0[2] + d[2]};
                bool in = true;
                float k2 = 0.f;
#pragma unroll
                for (int a = 0; a < N; ++a) {
                    in = in && p[a] >= 0 && p[a] < G.en[a];
                    const float gap = (float)grid_axis_key(d[a], var, a) * (float)G.eh[a];
                    k2 = fmaf(gap, gap, k2);
                }
                if (!in || k2 < cut || k2 >= lb) continue;
                const float cf[3] = {(float)d[0] - fr[0], (float)d[1] - fr[1], (float)d[2] - fr[2]};
                lb = grid_cell<N>(G, p, u, cf, sqrtf(k2), dr, inv, dnorm, lb);
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) lb = fminf(lb, __shfl_xor_sync(kFull, lb, o));
            best = lb;
        }
        if (lane == 0) {
            const float gam = sqrtf(best);
            G.out[v] = gam;
            ++my_eval;
            my_pass += gam <= 1.f;
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        my_eval += __shfl_xor_sync(kFull, my_eval, o);
        my_pass += __shfl_xor_sync(kFull, my_pass, o);
        my_over += __shfl_xor_sync(kFull, my_over, o);
    }
    if (lane == 0) {
        if (my_eval) atomicAdd(&G.ctr->n_eval, (unsigned long long)my_eval);
        if (my_pass) atomicAdd(&G.ctr->n_pass, (unsigned long long)my_pass);
        if (my_over) atomicAdd(&G.ctr->overflow_count, my_over);
    }
}

// --------------------------------------------------------------------------
// Plane seeds and the tiered walk
// --------------------------------------------------------------------------

// A reference voxel's place on the evaluation grid: its cell c0 (clamped to
// the grid) and its position fr in that cell (outside [0, 1) beyond the grid).
template <int N>
struct GridPlace {
    int c0[3];
    float fr[3];
};

template <int N>
__device__ __forceinline__ GridPlace<N> grid_place(const GridProblem& G, unsigned v)
{
    GridPlace<N> p;
    const unsigned r1 = v / (unsigned)G.rn[0];
    const unsigned ix[3] = {v % (unsigned)G.rn[0], r1 % (unsigned)G.rn[1], r1 / (unsigned)G.rn[1]};
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        p.c0[a] = 0;
        p.fr[a] = 0.f;
        if (a < N) {
            const double u = fma((double)ix[a], G.ub[a], G.ua[a]);
            const double f = fmin(fmax(floor(u), 0.0), (double)(G.en[a] - 2));
            p.c0[a] = (int)f;
            p.fr[a] = (float)(u - f);
        }
    }
    return p;
}

// The evaluated reference voxels, in order, with a bound on each one's gamma
// (squared, in out) as k_plane_seed finds it: kGridSteps steps along the affine
// part of one cell, from the cell that holds the point, then every face of the
// last cell (none when it is near singular: an infinite bound).  Bound by the
// latency of the dependent loads: 64 registers (16 bytes spilled) for 32 warps
// per SM; a 160x160x120 reference over a 320x320x240 grid 657.6 to 652.1 us.
constexpr int kGridSteps = 3;

template <int N>
__global__ void __launch_bounds__(256, 4) k_grid_seed(const __grid_constant__ GridProblem G)
{
    grid_release();
    grid_wait();
    const float dnorm = G.dose_norm > 0.f ? G.dose_norm : fdec(G.ctr->dnorm_enc);
    const float thr = cutoff_threshold(G.local, G.cutoff_frac, dnorm);
    const int sy = G.en[0], sz = G.en[0] * G.en[1], lane = threadIdx.x & 31;
    const float dmax = G.tau > 0.f ? 0.99f * rsqrtf(G.tau) : kInf;
    for (long long b = (long long)blockIdx.x * blockDim.x; b < G.nref; b += (long long)gridDim.x * blockDim.x) {
        const long long i = b + threadIdx.x;
        float dr = 0.f;
        bool take = false;
        if (i < G.nref) {
            dr = __ldg(G.ref + i);
            take = dr >= thr && (!G.local || dr > 0.f);
            if (!take) G.out[i] = kNaN;
        }
        const unsigned tk = __ballot_sync(kFull, take);
        unsigned pos = 0;
        if (tk && lane == 0) pos = atomicAdd(&G.ctr->grid_count, (unsigned)__popc(tk));
        pos = __shfl_sync(kFull, pos, 0) + (unsigned)__popc(tk & ((1u << lane) - 1u));
        if (!take) continue;
        const unsigned v = (unsigned)i;
        const GridPlace<N> at = grid_place<N>(G, v);
        const float inv = 1.0f / (G.dd_frac * (G.local ? dr : dnorm)), inv2 = inv * inv;
        int c[3] = {at.c0[0], at.c0[1], at.c0[2]};            // grid coordinates, every vertex inside
        float e[8];
#pragma unroll 1
        for (int it = 0;; ++it) {
            const float* q = G.ev + ((long long)c[2] * sz + (long long)c[1] * sy + c[0]);
#pragma unroll
            for (int u = 0; u < (1 << N); ++u)
                e[u] = __ldg(q + (u & 1) + ((u & 2) ? sy : 0) + ((u & 4) ? sz : 0));
            if (it == kGridSteps) break;
            const CellPlane<N> p = cell_plane<N>(e);
            float L = p.m - dr, D = 0.f, gk[3];
#pragma unroll
            for (int a = 0; a < N; ++a) {
                L = fmaf(-p.G[a], (float)(c[a] - at.c0[a]) - at.fr[a] + 0.5f, L);
                gk[a] = p.G[a] * G.mt.kappa[1 << a];
                D = fmaf(p.G[a], gk[a], D);
            }
            const float r = __fdividef(L * inv2, fmaf(D, inv2, 1.f));
            bool same = true;
#pragma unroll
            for (int a = 0; a < N; ++a) {
                // at most 500 cells away, within the packed offset's range
                const float s = fminf(fmaxf(at.fr[a] - r * gk[a], -500.f), 500.f);
                const int t = max(0, min(G.en[a] - 2, at.c0[a] + __float2int_rd(s)));
                same = same && t == c[a];
                c[a] = t;
            }
            if (same) break;
        }
        float q[8], cf[3] = {0.f, 0.f, 0.f};
#pragma unroll
        for (int u = 0; u < 8; ++u) q[u] = u < (1 << N) ? rel_dose(e[u], dr, inv) : kNaN;
#pragma unroll
        for (int a = 0; a < N; ++a) cf[a] = (float)(c[a] - at.c0[a]) - at.fr[a];
        CellGeom<float> g;
        cell_geom<N, float>(cf[0], cf[1], cf[2], G.mt, g);
        bool ill = false;
        const float cb = cell_min_d2<N, float>(q, g, G.mt, dmax, kInf, ill);
        if (ill) ill = cell_gram_ill<N>(q, (1u << (1 << N)) - 1u, G.mt.kappa, G.tau);
        G.out[v] = ill ? kInf : cb + 0.f;
        G.queue[pos] = v;
        G.skip[pos] = ill ? 0xffffffffu : pack10(c[0] - at.c0[0], c[1] - at.c0[1], N == 3 ? c[2] - at.c0[2] : 0);
    }
}

// The table walk in three tiers, as k_tail_cq's: a warp takes a batch of up to
// 32 queued voxels and walks 32 / gl of them at a time, gl lanes each.  A cell
// below the bound is tested by the distance from the point itself to its box
// and its dose gap (tier 1), by plane_bound (tier 2) and by its faces (tier 3),
// tiers 2 and 3 on full warps of cells from ring buffers.  Each cell is
// evaluated with the arithmetic of grid_cell.  A voxel with a near-singular
// cell, or whose bound lies past a truncated table, goes to walk_list;
// k_grid_walk searches it from scratch (FP64 redo, box scan).
//
// What bounds it: issue (68 %, the ALU pipe at 62 %): 0.56 ms, and 0.09 ms for
// the seeds, for 1.21 M voxels of a 160x160x120 reference against a 320x320x240
// evaluation dose.  The lane walk before it (k_grid_walk for every voxel: from
// an infinite bound, each lane evaluating its own cells, the rest of the warp
// waiting) took 1.91 ms there.
constexpr int kGqRing = 64;

struct GqWarp {
    unsigned ring[2][kGqRing]; // pending cells of tiers 2 and 3: table entry << 5 | slot of the voxel
    unsigned best[32];         // per slot: running squared gamma (float bits),
    unsigned vox[32], skip[32];    // voxel, its seed's cell,
    float dr[32], inv[32], fr[3][32];   // reference dose, 1 / Delta D, place in its cell,
    int c0[3][32], tv[32];     // that cell, and its table variant
    unsigned fixm;             // slots whose voxel is searched again by k_grid_walk
};

template <int N>
__global__ void __launch_bounds__(384, 2) k_grid_cq(const __grid_constant__ GridProblem G)
{
    __shared__ GqWarp gqw[12];
    grid_release();
    grid_wait();
    GqWarp& W = gqw[threadIdx.x >> 5];
    volatile GqWarp& V = gqw[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31, g = G.lanes, gl = lane & (g - 1);
    const unsigned lt_mask = (1u << lane) - 1u;
    const float dnorm = G.dose_norm > 0.f ? G.dose_norm : fdec(G.ctr->dnorm_enc);
    const float dmax = G.tau > 0.f ? 0.99f * rsqrtf(G.tau) : kInf;
    const float eh[3] = {(float)G.eh[0], (float)G.eh[1], (float)G.eh[2]};
    const int sy = G.en[0], sz = G.en[0] * G.en[1];
    const unsigned total = G.ctr->grid_count, nwarps = gridDim.x * (blockDim.x >> 5);
    const unsigned nv = 32u / (unsigned)g;         // voxels per round
    const unsigned nb = min(32u, max(nv, total / (8u * nwarps) / nv * nv));
    unsigned my_eval = 0, my_pass = 0;
    if (lane == 0) W.fixm = 0;
    __syncwarp();
    for (;;) {
        unsigned base = 0;
        if (lane == 0) base = atomicAdd(&G.ctr->head, nb);
        base = __shfl_sync(kFull, base, 0);
        if (base >= total) break;                  // warp-uniform
        const unsigned nlive = min(nb, total - base);
        if ((unsigned)lane < nlive) {
            const unsigned v = G.queue[base + lane];
            const GridPlace<N> at = grid_place<N>(G, v);
            const float dr = __ldg(G.ref + v);
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                V.c0[a][lane] = at.c0[a];
                V.fr[a][lane] = at.fr[a];
            }
            V.tv[lane] = grid_variant(at.fr, N);
            V.dr[lane] = dr;
            V.inv[lane] = 1.0f / (G.dd_frac * (G.local ? dr : dnorm));
            V.best[lane] = __float_as_uint(G.out[v]);
            V.vox[lane] = v;
            V.skip[lane] = G.skip[base + lane];
        }
        __syncwarp();
        unsigned head1 = 0, cnt1 = 0, head2 = 0, cnt2 = 0;   // the rings: [head, head + cnt)
        unsigned r0 = 0;                           // first slot of the next round
        int slot = 0, t = -1;                      // this lane's voxel and table entry (t < 0: no round)
        for (;;) {
            const bool rest = t < 0 && r0 >= nlive;            // every round is done: empty the rings
            if (cnt2 >= 32u || (rest && cnt1 == 0u && cnt2 > 0u)) {
                // ---- tier 3: the faces of the oldest pending cells ----
                const unsigned n = min(cnt2, 32u);
                if ((unsigned)lane < n) {
                    const unsigned w = V.ring[1][(head2 + (unsigned)lane) & (kGqRing - 1)];
                    const int own = (int)(w & 31u);
                    const uint32_t off = G.table[G.toff[V.tv[own]] + (int)(w >> 5)].off;
                    const int d[3] = {unpack10(off, 0), unpack10(off, 10), N == 3 ? unpack10(off, 20) : 0};
                    const int p[3] = {V.c0[0][own] + d[0], V.c0[1][own] + d[1], V.c0[2][own] + d[2]};
                    const bool ex = p[0] + 1 < G.en[0], ey = p[1] + 1 < G.en[1], ez = N == 3 && p[2] + 1 < G.en[2];
                    const float* q = G.ev + ((long long)p[2] * sz + (long long)p[1] * sy + p[0]);
                    const float odr = V.dr[own], oinv = V.inv[own];
                    float cq[8];
                    uint32_t ok = 0;
#pragma unroll
                    for (int u = 0; u < 8; ++u) {
                        cq[u] = kNaN;
                        if (u < (1 << N) && (!(u & 1) || ex) && (!(u & 2) || ey) && (!(u & 4) || ez)) {
                            cq[u] = rel_dose(__ldg(q + (u & 1) + ((u & 2) ? sy : 0) + ((u & 4) ? sz : 0)), odr, oinv);
                            ok |= 1u << u;
                        }
                    }
                    CellGeom<float> cg;
                    cell_geom<N, float>((float)d[0] - V.fr[0][own], (float)d[1] - V.fr[1][own],
                                        N == 3 ? (float)d[2] - V.fr[2][own] : 0.f, G.mt, cg);
                    bool ill = false;
                    const float cb = cell_min_d2<N, float>(cq, cg, G.mt, dmax, kInf, ill);
                    if (ill && cell_gram_ill<N>(cq, ok, G.mt.kappa, G.tau))
                        atomicOr(&W.fixm, 1u << own);                  // searched again
                    else
                        atomicMin(&W.best[own], __float_as_uint(cb + 0.f));   // -0 -> +0
                }
                head2 += n;
                cnt2 -= n;
                __syncwarp();
                continue;
            }
            if (cnt1 >= 32u || (rest && cnt1 > 0u)) {
                // ---- tier 2: plane_bound of the oldest cells past tier 1 ----
                const unsigned n = min(cnt1, 32u);
                bool cand = false;
                unsigned w = 0;
                if ((unsigned)lane < n) {
                    w = V.ring[0][(head1 + (unsigned)lane) & (kGqRing - 1)];
                    const int own = (int)(w & 31u);
                    const uint32_t off = G.table[G.toff[V.tv[own]] + (int)(w >> 5)].off;
                    const int d[3] = {unpack10(off, 0), unpack10(off, 10), N == 3 ? unpack10(off, 20) : 0};
                    const float* q = G.ev + ((long long)(V.c0[2][own] + d[2]) * sz +
                                             (long long)(V.c0[1][own] + d[1]) * sy + (V.c0[0][own] + d[0]));
                    float dose[8], c[3] = {0.f, 0.f, 0.f}, hn2[3], kap[3];
#pragma unroll
                    for (int u = 0; u < (1 << N); ++u)
                        dose[u] = __ldg(q + (u & 1) + ((u & 2) ? sy : 0) + ((u & 4) ? sz : 0));
#pragma unroll
                    for (int a = 0; a < N; ++a) {
                        c[a] = (float)d[a] - V.fr[a][own];
                        hn2[a] = G.mt.hn2[a];
                        kap[a] = G.mt.kappa[1 << a];
                    }
                    cand = off != V.skip[own] &&
                           !(plane_bound<N>(dose, c, V.dr[own], V.inv[own], hn2, kap) >=
                             __uint_as_float(V.best[own]) * kPlaneSlack);
                }
                head1 += n;
                cnt1 -= n;
                const unsigned cm = __ballot_sync(kFull, cand);
                if (cand) V.ring[1][(head2 + cnt2 + (unsigned)__popc(cm & lt_mask)) & (kGqRing - 1)] = w;
                cnt2 += (unsigned)__popc(cm);
                __syncwarp();
                continue;
            }
            if (t < 0) {
                if (r0 >= nlive) break;                        // the batch is done
                slot = (int)r0 + lane / g;                     // the next round
                r0 += nv;
                t = gl;
            }
            // the lane's voxel (from shared memory after every pass of the other tiers)
            const bool live = (unsigned)slot < nlive;
            const int sl = live ? slot : 0;
            int c0[3];
            float fr[3];
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                c0[a] = V.c0[a][sl];
                fr[a] = V.fr[a][sl];
            }
            const float dr = V.dr[sl], inv = V.inv[sl];
            const float best = live ? __uint_as_float(V.best[sl]) : -1.f;   // < 0: nothing is below it
            const TableEntry* const tab = G.table + G.toff[V.tv[sl]];
            const int ntable = G.tlen[V.tv[sl]];
            do {
                // ---- tier 1: one table entry per lane and step ----
                TableEntry e{0u, kInf};
                if (t < ntable) e = tab[t];
                const float key2 = e.key * e.key;
                const bool keyed = key2 < best;
                if (!__any_sync(kFull, keyed)) {               // A1 step 4b-ii, exact
                    t = -1;
                    break;
                }
                const unsigned ent = (unsigned)t;
                t += g;
                bool cand = false, edge = false;               // edge: a cell with vertices outside the grid
                if (keyed) {
                    const int d[3] = {unpack10(e.off, 0), unpack10(e.off, 10), N == 3 ? unpack10(e.off, 20) : 0};
                    int p[3];
                    bool in = true;
                    // the distance from the point to the cell's box: a lower bound
                    // in FP32 from the integer offset and the point's fraction,
                    // each axis lowered by its rounding (4 ulp of its operands) and
                    // the sum by 1e-5
                    float k2 = 0.f;
#pragma unroll
                    for (int a = 0; a < N; ++a) {
                        p[a] = c0[a] + d[a];
                        in = in && (unsigned)p[a] < (unsigned)G.en[a];
                        edge = edge || p[a] + 1 >= G.en[a];
                        const float lo = (float)d[a] - fr[a];
                        const float slack = 4.8e-7f * (fabsf(fr[a]) + fabsf((float)d[a]) + 2.f);
                        const float gap = fmaxf(fmaxf(lo, -1.f - lo) - slack, 0.f) * eh[a];
                        k2 = fmaf(gap, gap, k2);
                    }
                    k2 = fmaxf(k2 * 0.99999f, key2);
                    if (in && k2 < best) {
                        const float* q = G.ev + ((long long)(N == 3 ? p[2] : 0) * sz + (long long)p[1] * sy + p[0]);
                        float dlo = kInf, dhi = -kInf;
                        if (!edge) {
                            float f[8];
#pragma unroll
                            for (int u = 0; u < (1 << N); ++u)
                                f[u] = __ldg(q + (u & 1) + ((u & 2) ? sy : 0) + ((u & 4) ? sz : 0));
                            dlo = fminf(min3(f[0], f[1], f[2]), f[3]);
                            dhi = fmaxf(max3(f[0], f[1], f[2]), f[3]);
                            if constexpr (N == 3) {
                                dlo = min3(min3(dlo, f[4], f[5]), f[6], f[7]);
                                dhi = max3(max3(dhi, f[4], f[5]), f[6], f[7]);
                            }
                        } else {
                            const bool ex = p[0] + 1 < G.en[0], ey = p[1] + 1 < G.en[1],
                                       ez = N == 3 && p[2] + 1 < G.en[2];
#pragma unroll
                            for (int u = 0; u < (1 << N); ++u) {
                                if ((!(u & 1) || ex) && (!(u & 2) || ey) && (!(u & 4) || ez)) {
                                    const float f = __ldg(q + (u & 1) + ((u & 2) ? sy : 0) + ((u & 4) ? sz : 0));
                                    dlo = fminf(dlo, f);
                                    dhi = fmaxf(dhi, f);
                                }
                            }
                        }
                        const float gap = max3(dlo - dr, dr - dhi, 0.f) * inv;
                        cand = fmaf(gap, gap, k2) < best;
                    }
                }
                // a whole cell goes to tier 2, one at the grid's edge to tier 3
                const unsigned cm = __ballot_sync(kFull, cand && !edge);
                if (cand && !edge)
                    V.ring[0][(head1 + cnt1 + (unsigned)__popc(cm & lt_mask)) & (kGqRing - 1)] = ent << 5 | (unsigned)slot;
                cnt1 += (unsigned)__popc(cm);
                const unsigned em = __ballot_sync(kFull, cand && edge);
                if (em) {
                    if (cand && edge)
                        V.ring[1][(head2 + cnt2 + (unsigned)__popc(em & lt_mask)) & (kGqRing - 1)] = ent << 5 | (unsigned)slot;
                    cnt2 += (unsigned)__popc(em);
                }
            } while (max(cnt1, cnt2) < 32u);
            __syncwarp();
        }
        // ---- final values, one voxel per lane ----
        const unsigned fixm = V.fixm;
        if ((unsigned)lane < nlive) {
            const float b = __uint_as_float(V.best[lane]), rc = G.tcover[V.tv[lane]];
            const unsigned v = V.vox[lane];
            if (((fixm >> lane) & 1u) || !(b <= rc * rc)) {
                G.walk_list[atomicAdd(&G.ctr->fix_count, 1u)] = v;     // k_grid_walk finishes it
            } else {
                const float gam = sqrtf(b);
                G.out[v] = gam;
                ++my_eval;
                my_pass += gam <= 1.f;
            }
        }
        __syncwarp();
        if (lane == 0 && fixm) W.fixm = 0;
        __syncwarp();
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        my_eval += __shfl_xor_sync(kFull, my_eval, o);
        my_pass += __shfl_xor_sync(kFull, my_pass, o);
    }
    if (lane == 0) {
        if (my_eval) atomicAdd(&G.ctr->n_eval, (unsigned long long)my_eval);
        if (my_pass) atomicAdd(&G.ctr->n_pass, (unsigned long long)my_pass);
    }
}

// --------------------------------------------------------------------------
// Host side
// --------------------------------------------------------------------------

int build_grid_table(int nd, const double hn[3], const int en[3], long long cap, int variant,
                     std::vector<TableEntry>& table, double& r_cover)
{
    // radius from a ball-volume estimate of about 2 * cap cells
    const double cellvol = hn[0] * hn[1] * (nd == 3 ? hn[2] : 1.0);
    double R = nd == 3 ? std::cbrt(2.0 * (double)cap * cellvol * 3.0 / (4.0 * M_PI))
                       : std::sqrt(2.0 * (double)cap * cellvol / M_PI);
    bool whole = false, packing = false;
    int lo[3] = {0, 0, 0}, hi[3] = {0, 0, 0};
    double diag = 0;
    for (int a = 0; a < nd; ++a) diag += (double)en[a] * en[a] * hn[a] * hn[a];
    diag = std::sqrt(diag) + 1.0;
    if (R > diag) { R = diag; whole = true; }
    for (int a = 0; a < nd; ++a) {
        long long l = (long long)std::ceil(R / hn[a]) + 2;
        l = std::min<long long>(l, en[a]);
        if (l > 511) { l = 511; packing = true; }
        lo[a] = -(int)l;
        hi[a] = (int)l;
    }
    struct Tmp { double key; int x, y, z; };
    std::vector<Tmp> all;
    try {
        for (int z = lo[2]; z <= hi[2]; ++z)
            for (int y = lo[1]; y <= hi[1]; ++y)
                for (int x = lo[0]; x <= hi[0]; ++x) {
                    const int c[3] = {x, y, z};
                    double k2 = 0;
                    for (int a = 0; a < nd; ++a) {
                        const double gap = grid_axis_key(c[a], variant, a) * hn[a];
                        k2 += gap * gap;
                    }
                    const double key = std::sqrt(k2);
                    if (key < R) all.push_back({key, x, y, z});
                }
    } catch (const std::bad_alloc&) {
        return GAMMA_ERR_OOM;
    }
    std::sort(all.begin(), all.end(), [](const Tmp& a, const Tmp& b) {
        if (a.key != b.key) return a.key < b.key;
        // the voxel's own cell first among the key-0 cells (a finite bound
        // from the walk's first round), then z, y, x
        const bool a0 = (a.x | a.y | a.z) == 0, b0 = (b.x | b.y | b.z) == 0;
        if (a0 != b0) return a0;
        if (a.z != b.z) return a.z < b.z;
        if (a.y != b.y) return a.y < b.y;
        return a.x < b.x;
    });
    double cover = whole ? INFINITY : R;
    if (packing) {
        double m = INFINITY;
        for (int a = 0; a < nd; ++a) m = std::min(m, 509.0 * hn[a]);
        cover = std::min(cover, m);
    }
    size_t keep = all.size();
    if ((long long)keep > cap) {
        keep = (size_t)cap;
        cover = std::min(cover, all[keep].key);
    }
    table.resize(keep);
    for (size_t i = 0; i < keep; ++i) {
        table[i].off = pack10(all[i].x, all[i].y, all[i].z);
        float f = (float)all[i].key;
        if ((double)f > all[i].key) f = std::nextafterf(f, -INFINITY);
        table[i].key = f;
    }
    r_cover = cover;
    return GAMMA_OK;
}

cudaError_t launch_grids(const GridProblem& G, cudaStream_t s)
{
    const int sms = device_sm_count();
    const long long nmax = std::max(G.nref, G.neval);
    const int gp = (int)std::max<long long>(1, std::min<long long>((nmax + 255) / 256, (long long)sms * 8));
    k_grid_prepare<<<gp, 256, 0, s>>>(G);
    // bounds from plane seeds, the tiered walk, then a 32-lane search of the
    // voxels it left
    const int gs = (int)std::max<long long>(1, std::min<long long>((G.nref + 255) / 256, (long long)sms * 8));
    if (G.ndim == 3) {
        launch_next(k_grid_seed<3>, gs, 256, 0, s, G);
        launch_next(k_grid_cq<3>, sms * 2, 384, 0, s, G);
        launch_next(k_grid_walk<3>, sms * 2, 256, 0, s, G);
    } else {
        launch_next(k_grid_seed<2>, gs, 256, 0, s, G);
        launch_next(k_grid_cq<2>, sms * 2, 384, 0, s, G);
        launch_next(k_grid_walk<2>, sms * 2, 256, 0, s, G);
    }
    return cudaGetLastError();
}

}  // namespace gk
