// Per-cell helpers shared by the search kernels and the paper-design
// ablation: criteria resolution, the near-singular Gram pre-filter, the FP64
// redo of a cell, and the evaluation of every face a cell owns.
#pragma once
#include <cuda_runtime.h>
#include <cstdint>

#include "gamma_face.cuh"
#include "gamma_internal.h"

namespace gk {

constexpr unsigned kFull = 0xffffffffu;

__device__ __forceinline__ float resolve_dnorm(const Problem& P)
{
    return P.dose_norm > 0.f ? P.dose_norm : fdec(P.ctr->dnorm_enc);
}

// Pre-filter threshold on D for the near-singular Gram test (see face_core).
__device__ __forceinline__ float ill_dmax(const Problem& P)
{
    return P.tau > 0.f ? 0.99f * rsqrtf(P.tau) : kInf;
}

// The cutoff below which a reference voxel is not evaluated: cutoff_frac *
// D_norm.  Global criteria need a positive dose norm (their Delta D is
// dd_frac * D_norm); without one (a reference with no positive dose and no
// norm given) no voxel is evaluated: the threshold is +inf, every voxel gets
// NaN and the run reports GAMMA_ERR_DOSE_NORM, instead of searching with a
// zero Delta D, whose infinite gamma would walk the whole grid per voxel.
__host__ __device__ __forceinline__ float cutoff_threshold(int local, float cutoff_frac, float dnorm)
{
    return (local || dnorm > 0.f) ? cutoff_frac * dnorm : kInf;
}

__device__ __forceinline__ bool is_evaluated(const Problem& P, float dr, float thr)
{
    return dr >= thr && (!P.local || dr > 0.f);
}

// Dose e relative to the reference dose dr in units of Delta D (inv = 1 /
// Delta D).  The rounded product is kept: a compiler that fused it into the
// face evaluation's differences would give another last bit than the walks
// that pass the relative doses on through memory or a call.
__device__ __forceinline__ float rel_dose(float e, float dr, float inv) { return __fmul_rn(e - dr, inv); }

// --------------------------------------------------------------------------
// FP64 redo of one cell whose Gram matrices are near singular
// --------------------------------------------------------------------------

template <int N, typename C = int>
__device__ __noinline__ float cell_redo_f64(const float* __restrict__ ev, long long p, long long sy,
                                            long long sz, uint32_t ok, C cx, C cy, C cz,
                                            double drd, double invd, MetricT<double> mtd,
                                            unsigned int* fp64_counter)
{
    double q[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
        q[u] = (double)kNaN;
        if (u < (1 << N) && ((ok >> u) & 1u)) {
            const long long o = p + ((u & 1) ? 1 : 0) + ((u & 2) ? sy : 0) + ((u & 4) ? sz : 0);
            q[u] = ((double)ev[o] - drd) * invd;
        }
    }
    CellGeom<double> g;
    cell_geom<N, double>(cx, cy, cz, mtd, g);
    bool ill = false;
    const double b = cell_min_d2<N, double>(q, g, mtd, (double)kInf, (double)kInf, ill);
    atomicAdd(fp64_counter, 1u);
    return (float)b;
}

// A cell whose FP32 pass raised the near-singular pre-filter (rare): the
// exact test on the same relative doses, reloaded here from the evaluation
// grid as the caller formed them ((D_e - D_r) * inv), then the FP64 redo when
// the test holds.  Out of line, so that the callers keep no registers for it.
template <int N>
__device__ __noinline__ float cell_recheck(const Problem& P, uint32_t ok, int cx, int cy, int cz,
                                           long long p, float dr, float inv, float dnorm, float cb)
{
    const long long sy = P.nx, sz = (long long)P.nx * P.ny;
    float q[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
        q[u] = kNaN;
        if (u < (1 << N) && ((ok >> u) & 1u)) {
            const long long o = p + ((u & 1) ? 1 : 0) + ((u & 2) ? sy : 0) + ((u & 4) ? sz : 0);
            q[u] = (__ldg(P.ev + o) - dr) * inv;
        }
    }
    if (!cell_gram_ill<N>(q, ok, P.mt.kappa, P.tau)) return cb;
    const double drd = dr;
    const double invd = 1.0 / ((double)P.dd_frac * (P.local ? drd : (double)dnorm));
    return cell_redo_f64<N>(P.ev, p, sy, sz, ok, cx, cy, cz, drd, invd, P.mtd, &P.ctr->fp64_cells);
}

// The voxel itself among the vertices of a cell whose box contains it (lower
// corner at 0 or -1 on every axis): taken out for the walks, so that only the
// cell's faces off the voxel remain.  Those through it have their value from the
// reduced form before any table walk, and the general one could differ from it in
// the last bit.  Other cells are left as they are.
//
// The reduced form's conditions lose their digits where a dose step is some 1e5
// Delta D, and a valid face through the voxel may be left out.  A cell that is
// near singular with the voxel's vertex therefore gets its FP64 evaluation like
// any other: steep says that it may be (D of a face is at most 1 + N (range of the
// vertices)^2 kappa_max; below dmax the Gram matrices need no look), and the test
// of the Gram matrices is asked with the vertex put back.
template <int N>
struct OwnVertex {
    int self;           // its index, or -1
    float q;            // its relative dose
    bool steep;

    __device__ __forceinline__ void take(float (&v)[8], int cx, int cy, int cz, const float (&kappa)[8], float dmax)
    {
        self = -1;
        q = 0.f;
        steep = false;
        if ((unsigned)(cx + 1) < 2u && (unsigned)(cy + 1) < 2u && (N == 2 || (unsigned)(cz + 1) < 2u)) {
            self = (cx & 1) | ((cy & 1) << 1) | (N == 3 ? (cz & 1) << 2 : 0);
            float lo = v[0], hi = v[0];
#pragma unroll
            for (int u = 1; u < (1 << N); ++u) {              // (NaN: no such vertex)
                lo = fminf(lo, v[u]);
                hi = fmaxf(hi, v[u]);
            }
            const float range = hi - lo, k2 = fmaxf(kappa[1], kappa[2]), kmax = N == 3 ? fmaxf(k2, kappa[4]) : k2;
            steep = fmaf((float)N * kmax * range, range, 1.f) > dmax;
#pragma unroll
            for (int u = 0; u < (1 << N); ++u)
                if (u == self) {
                    q = v[u];
                    v[u] = kNaN;
                }
        }
    }
    __device__ __forceinline__ void put(float (&v)[8]) const
    {
#pragma unroll
        for (int u = 0; u < (1 << N); ++u)
            if (u == self) v[u] = q;
    }
};

// Every face of the cell with lower corner (x+cx, y+cy, z+cz) as squared
// gamma (WALK: of a cell whose box contains the voxel only those off the
// voxel), with the FP64 redo of the cell when a face's Gram matrix is near
// singular.  q holds (D_e - dr) * inv of the cell's vertices.  Out of line:
// each kernel keeps one copy, and the callers keep their own registers few.
template <int N, bool WALK>
__device__ __noinline__ float cell_all_faces(const Problem& P, float q0, float q1, float q2,
                                             float q3, float q4, float q5, float q6, float q7,
                                             uint32_t ok, int cx, int cy, int cz, long long p,
                                             float dr, float dnorm)
{
    float q[8] = {q0, q1, q2, q3, q4, q5, q6, q7};
    OwnVertex<N> own;
    if (WALK) own.take(q, cx, cy, cz, P.mt.kappa, ill_dmax(P));
    CellGeom<float> g;
    cell_geom<N, float>(cx, cy, cz, P.mt, g);
    bool ill = false;
    float cb = cell_min_d2<N, float>(q, g, P.mt, ill_dmax(P), kInf, ill);
    if (WALK && (ill || own.steep)) {
        own.put(q);
        ill = true;
    }
    if (ill) ill = cell_gram_ill<N>(q, ok, P.mt.kappa, P.tau);
    if (ill) {
        const double drd = dr;
        const double invd = 1.0 / ((double)P.dd_frac * (P.local ? drd : (double)dnorm));
        const long long sy = P.nx, sz = (long long)P.nx * P.ny;
        cb = cell_redo_f64<N>(P.ev, p, sy, sz, ok, cx, cy, cz, drd, invd, P.mtd, &P.ctr->fp64_cells);
    }
    return cb;
}

}  // namespace gk
