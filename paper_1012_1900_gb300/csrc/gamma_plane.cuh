// A lower bound on the distance to the surface over one cell from its affine
// part: a fraction of the work of its faces, and tight where the dose is smooth
// over the cell.  Used before the faces by the table walks.
#pragma once
#include <cuda_runtime.h>

#include "gamma_near.cuh"

namespace gk {

// The affine part of the 2^N vertex doses e of a cell: the value m at the
// cell's centre, the slope G per voxel along each axis, and eps, a bound on
// how far a vertex (hence, by linearity in each simplex, any point of the
// interpolant) lies from it: the sum of the magnitudes of the remaining
// Walsh-Hadamard coefficients.
template <int N>
struct CellPlane {
    float m, G[3], eps;
};

template <int N>
__device__ __forceinline__ CellPlane<N> cell_plane(const float (&e)[8])
{
    CellPlane<N> c;
    if constexpr (N == 3) {
        const float a0 = e[1] - e[0], a1 = e[3] - e[2], a2 = e[5] - e[4], a3 = e[7] - e[6];
        const float m0 = e[1] + e[0], m1 = e[3] + e[2], m2 = e[5] + e[4], m3 = e[7] + e[6];
        const float xlo = a0 + a1, xhi = a2 + a3, ylo = a1 - a0, yhi = a3 - a2;
        const float plo = m0 + m1, phi = m2 + m3, rlo = m1 - m0, rhi = m3 - m2;
        c.m = 0.125f * (plo + phi);
        c.G[0] = 0.25f * (xlo + xhi);
        c.G[1] = 0.25f * (rlo + rhi);
        c.G[2] = 0.25f * (phi - plo);
        c.eps = 0.125f * ((fabsf(xhi - xlo) + fabsf(ylo + yhi)) + (fabsf(yhi - ylo) + fabsf(rhi - rlo)));
    } else {
        const float a0 = e[1] - e[0], a1 = e[3] - e[2], m0 = e[1] + e[0], m1 = e[3] + e[2];
        c.m = 0.25f * (m0 + m1);
        c.G[0] = 0.5f * (a0 + a1);
        c.G[1] = 0.5f * (m1 - m0);
        c.G[2] = 0.f;
        c.eps = 0.25f * fabsf(a1 - a0);
    }
    return c;
}

// A lower bound on the squared gamma distance from the voxel to the surface
// over the cell with lower corner c (voxels from the voxel).  With p the
// cell's affine part (in units of Delta D), the surface satisfies |d - p(s)|
// <= eps, so its squared distance at s is at least
//     f(s) = |s|^2 + max(|p(s)| - eps, 0)^2 .
// Where the plane's value L at the voxel exceeds eps, f is bounded below by
// the convex |s|^2 + max(+-p(s) - eps, 0)^2, whose minimum is (|L| - eps)^2 / D
// at the foot point s* (D = 1 + |grad p|^2), and which grows by at least
// |s - s*|^2 away from it: so f >= (|L| - eps)^2 / D + dist(s*, box)^2.  Below
// eps the same formula with s* = 0 gives the box distance alone.  eps takes
// up the rounding of L (ten operations on terms whose magnitudes it sums).
template <int N>
__device__ __forceinline__ float plane_bound(const float (&e)[8], const float (&c)[3], float dr, float inv,
                                             const float (&hn2)[3], const float (&kap)[3])
{
    const CellPlane<N> p = cell_plane<N>(e);
    float L = p.m - dr, mag = fabsf(p.m) + fabsf(dr), D = 0.f, gk[3];
#pragma unroll
    for (int a = 0; a < N; ++a) {
        const float t = p.G[a] * (c[a] + 0.5f);
        L -= t;
        mag += fabsf(t);
        gk[a] = p.G[a] * kap[a];
        D = fmaf(p.G[a], gk[a], D);
    }
    const float inv2 = inv * inv;
    D = fmaf(D, inv2, 1.f);
    const float Lm = fmaxf(fabsf(L) - fmaf(2e-6f, mag + p.eps, p.eps), 0.f);     // dose units
    const float r = __fdividef(Lm * inv2, D);
    float b = Lm * r;
    const float sr = L > 0.f ? -r : r;
#pragma unroll
    for (int a = 0; a < N; ++a) {
        const float s = sr * gk[a];                          // the foot point, in voxels
        const float w = max3(c[a] - s, s - (c[a] + 1.f), 0.f);
        b = fmaf(hn2[a] * w, w, b);
    }
    return b;
}
// A cell is left out when plane_bound reaches best by more than its rounding:
// the foot point and the box distance carry a relative error of some 1e-6 of
// the distances involved, which are below sqrt(best) plus a voxel.
constexpr float kPlaneSlack = 1.f + 3e-5f;

}  // namespace gk
