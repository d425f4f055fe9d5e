// Faces of the triangulation that contain the reference voxel's own node:
// the reduced closed form of the Section 2.1 projection used for the key-0
// cells (the 2^n cells whose box contains the voxel).
//
// Such a face is a chain through the voxel v,
//     v - W_b < ... < v - W_1 < v < v + V_1 < ... < v + V_a,
// with W_1 < ... < W_b and V_1 < ... < V_a strictly nested non-empty axis
// sets and W_b, V_a disjoint (a + b = m increments, 75 faces in 3D including
// the vertex itself, 13 in 2D).  In the general closed form (gamma_face.cuh)
// the chain starts at s0 = -W_b * h / dta, so beta_i = 1 for the b increments
// below v and 0 above it, rho^2 = 0, and L telescopes to the voxel's own
// relative dose q_v.  Multiplying D and the validity conditions by dD^2 (both
// sides of every condition scale alike) leaves, with g = D_e(v) - D_r and, for
// an edge from a node to the next one outward over the axis set A,
//     t = Delta^2 kappa_A,   alpha = g (D_e(inner) - D_e(outer)) kappa_A,
//     D~ = dD^2 + sum of t over the face's edges,   dist^2 = g^2 / D~ .
// The conditions on the projection read alike on both sides of v: along each
// side's chain, from v outward, alpha_1 >= alpha_2 >= ... >= 0, and the two
// sides together alpha_1(W) + alpha_1(V) <= D~ (a missing side counts 0).
// The minimum over the faces through v is therefore g^2 / max D~ over the
// faces whose projection is valid (the vertex alone gives D~ = dD^2).  Every
// term is a product or a sum of non-negative terms: there is no cancellation,
// so FP32 needs no double-precision redo here.
//
// How it is computed.  A face's conditions become one slack, the minimum of 0
// and of their differences, with three-operand minima (one instruction each
// for two of them), and D~ + kNearOff * slack takes part in a running
// maximum: D~ itself where the slack is 0, a hugely negative value where any
// condition fails (one missed by less than 1e-30 of D~ would pass: the two
// faces then agree to far below a rounding).  So a face costs three or four
// ALU instructions where a comparison per condition cost four or five, the
// rest runs on the FMA pipe, and that rest works on two voxels at once
// (Near2: packed FP32 pairs).  The slacks and sums of one side's chains are
// shared by all faces through them.  Doses of nodes outside the grid are NaN:
// the D~ of a face that uses one is NaN, which the maximum passes over.
//
// Measured on a 160x160x120 map (1.21 M evaluated voxels, k_shell_w alone):
// 61.5 us and 45.9 M warp instructions with a comparison per condition and one
// voxel per lane (ALU pipe 64 %), 52.9 us and 34.1 M now (ALU 43 %, issue 56 %
// with four warps per scheduler: bound by the latency of its own chains at the
// 128 registers that two blocks per SM leave).
#pragma once
#include <cstdint>

namespace gk {

// Minimum / maximum of three (one instruction on sm_100 and later); like
// fminf, a NaN operand is passed over.
__device__ __forceinline__ float min3(float a, float b, float c)
{
    float r;
    asm("min.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}
__device__ __forceinline__ float max3(float a, float b, float c)
{
    float r;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}

// One voxel, or a pair of voxels in one packed register pair.  Every
// operation is rounded by itself, so both give the same bits.
struct Near1 {
    float v;
    static __device__ __forceinline__ Near1 all(float a) { return {a}; }
};
__device__ __forceinline__ Near1 n_add(Near1 a, Near1 b) { return {__fadd_rn(a.v, b.v)}; }
__device__ __forceinline__ Near1 n_sub(Near1 a, Near1 b) { return {__fsub_rn(a.v, b.v)}; }
__device__ __forceinline__ Near1 n_mul(Near1 a, Near1 b) { return {__fmul_rn(a.v, b.v)}; }
__device__ __forceinline__ Near1 n_fma(Near1 a, Near1 b, Near1 c) { return {__fmaf_rn(a.v, b.v, c.v)}; }
__device__ __forceinline__ Near1 n_min(Near1 a, Near1 b) { return {fminf(a.v, b.v)}; }
__device__ __forceinline__ Near1 n_min3(Near1 a, Near1 b, Near1 c) { return {min3(a.v, b.v, c.v)}; }
__device__ __forceinline__ Near1 n_max3(Near1 a, Near1 b, Near1 c) { return {max3(a.v, b.v, c.v)}; }

struct Near2 {
    unsigned long long v;
    static __device__ __forceinline__ Near2 pack(float a, float b)
    {
        Near2 r;
        asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(a), "f"(b));
        return r;
    }
    static __device__ __forceinline__ Near2 all(float a) { return pack(a, a); }
    __device__ __forceinline__ void get(float& a, float& b) const
    {
        asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
    }
};
__device__ __forceinline__ Near2 n_add(Near2 a, Near2 b)
{
    Near2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ Near2 n_mul(Near2 a, Near2 b)
{
    Near2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ Near2 n_fma(Near2 a, Near2 b, Near2 c)
{
    Near2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
    return r;
}
__device__ __forceinline__ Near2 n_sub(Near2 a, Near2 b) { return n_fma(b, Near2::all(-1.f), a); }
__device__ __forceinline__ Near2 n_min(Near2 a, Near2 b)
{
    float a0, a1, b0, b1;
    a.get(a0, a1);
    b.get(b0, b1);
    return Near2::pack(fminf(a0, b0), fminf(a1, b1));
}
__device__ __forceinline__ Near2 n_min3(Near2 a, Near2 b, Near2 c)
{
    float a0, a1, b0, b1, c0, c1;
    a.get(a0, a1);
    b.get(b0, b1);
    c.get(c0, c1);
    return Near2::pack(min3(a0, b0, c0), min3(a1, b1, c1));
}
__device__ __forceinline__ Near2 n_max3(Near2 a, Near2 b, Near2 c)
{
    float a0, a1, b0, b1, c0, c1;
    a.get(a0, a1);
    b.get(b0, b1);
    c.get(c0, c1);
    return Near2::pack(max3(a0, b0, c0), max3(a1, b1, c1));
}

constexpr float kNearOff = 1e30f;

// The running maximum of D~ over the valid faces, two faces per instruction.
template <class V>
struct NearMax {
    V best, hold;
    bool held = false;
    // (unrolled everywhere: `held` is a compile-time constant at each call)
    __device__ __forceinline__ void face(V D, V slack)
    {
        const V d = n_fma(slack, V::all(kNearOff), D);
        if (held) best = n_max3(best, hold, d);
        else hold = d;
        held = !held;
    }
};

// What the first side leaves for the faces through the voxel: per set W of
// fewer than N axes the edge from the voxel (t, alpha), and (3D) per chain of
// one axis W within a pair U its sum of t and its slack.
template <int N, class V>
struct NearSide {
    V t[1 << N], alpha[1 << N];
    V t2[1 << N][2], sl2[1 << N][2];     // [U][is W the higher axis of U]
};

// One side of the voxel: n[W] its nodes (W = 1 .. 2^N - 1), e0 the voxel's own
// dose.  The faces on this side alone go to `m`; the first side fills `a`, the
// second adds the faces through the voxel as it forms its own chains, one
// inner set X after the other, so that it keeps none of them.
template <int N, bool SECOND, class V>
__device__ __forceinline__ void near_side(const V (&n)[1 << N], V e0, V g, V D0, const V (&kappa)[1 << N],
                                          NearSide<N, V>& a, NearMax<V>& m)
{
    constexpr int NU = 1 << N, ALL = NU - 1;
    // D~ - alpha(W) - alpha(V) is formed one side after the other, the second
    // product not rounded by itself: where g is near a dose step of 1e5 Delta D the
    // difference is all in the last digits (of 3,528 voxels of 1e4 on planes, 144
    // give a gamma off by more than 1e-4; 234 with the sum of the two products
    // taken away).  0.7 % of a map's time.
    const V zero = V::all(0.f), ng = n_sub(zero, g);
    V tx[NU], ax[NU];                        // edges from a pair of axes to all three
    if (N == 3) {
#pragma unroll
        for (int U = 1; U < ALL; ++U)
            if (U & (U - 1)) {
                const V dl = n_sub(n[U], n[ALL]), k = n_mul(dl, kappa[ALL ^ U]);
                tx[U] = n_mul(dl, k);
                ax[U] = n_mul(g, k);
            }
    }
#pragma unroll
    for (int X = 1; X < NU; ++X) {
        const V dl = n_sub(e0, n[X]), k = n_mul(dl, kappa[X]);
        const V t = n_mul(dl, k), al = n_mul(g, k), sl = n_min(al, zero);
        const V D = n_add(D0, t);
        m.face(D, n_min(sl, n_sub(D, al)));
        if (!SECOND) {
            a.t[X] = t;
            a.alpha[X] = al;
        } else {
#pragma unroll
            for (int W = 1; W < ALL; ++W) {
                if (W & X) continue;
                const V Dt = n_add(D, a.t[W]);
                m.face(Dt, n_min3(a.alpha[W], sl, n_fma(ng, k, n_sub(Dt, a.alpha[W]))));
                if (N == 3 && !(W & (W - 1)) && !(X & (X - 1))) {
                    // one axis each: the third one extends the first side's chain
                    const int U = ALL ^ X, h = W != (U & -U);
                    const V Dw = n_add(D, a.t2[U][h]);
                    m.face(Dw, n_min3(a.sl2[U][h], al, n_fma(ng, k, n_sub(Dw, a.alpha[W]))));
                }
            }
        }
#pragma unroll
        for (int U = X + 1; U < NU; ++U) {
            if ((X & U) != X) continue;
            const V d2 = n_sub(n[X], n[U]), k2 = n_mul(d2, kappa[U ^ X]);
            const V t2 = n_add(t, n_mul(d2, k2)), a2 = n_mul(g, k2);
            const V sl2 = n_min3(a2, n_sub(al, a2), zero);
            const V D2 = n_add(D0, t2);
            m.face(D2, n_min(sl2, n_sub(D2, al)));
            if (N == 3 && U != ALL) {        // X one axis, U a pair
                const V D3 = n_add(D2, tx[U]);
                m.face(D3, n_min(n_min3(sl2, ax[U], n_sub(a2, ax[U])), n_sub(D3, al)));
                if (!SECOND) {
                    a.t2[U][X != (U & -U)] = t2;
                    a.sl2[U][X != (U & -U)] = sl2;
                } else {
                    const int W = ALL ^ U;
                    const V Dx = n_add(D2, a.t[W]);
                    m.face(Dx, n_min3(sl2, a.alpha[W], n_fma(ng, k, n_sub(Dx, a.alpha[W]))));
                }
            }
        }
    }
}

// The largest D~ over the valid faces through the voxel: lo[U] / hi[U] the
// doses of the nodes v - U / v + U (U = 1 .. 2^N - 1; NaN outside the grid),
// e0 the voxel's own, g = e0 - D_r, D0 = dD^2.
template <int N, class V>
__device__ __forceinline__ V near_dmax(const V (&lo)[1 << N], const V (&hi)[1 << N], V e0, V g, V D0,
                                       const float (&kap)[8])
{
    constexpr int NU = 1 << N;
    V kappa[NU];
#pragma unroll
    for (int A = 1; A < NU; ++A) kappa[A] = V::all(kap[A]);
    NearMax<V> m;
    m.best = D0;
    m.hold = D0;
    NearSide<N, V> a;
    near_side<N, false, V>(lo, e0, g, D0, kappa, a, m);
    near_side<N, true, V>(hi, e0, g, D0, kappa, a, m);
    return m.held ? n_max3(m.best, m.hold, m.hold) : m.best;
}

// Node v +- U of a staged tile (row stride SY, plane stride SZ).
template <int SY, int SZ>
__device__ __forceinline__ constexpr int near_off(int U)
{
    return (U & 1 ? 1 : 0) + (U & 2 ? SY : 0) + (U & 4 ? SZ : 0);
}

// Squared gamma over the faces through voxel v (node tix of a staged tile
// with x stride 1 and row / plane strides SY / SZ; nodes outside the grid NaN).
template <int N, int SY, int SZ>
__device__ __forceinline__ float near_gamma2(const float* tile, int tix, float dr, float dD,
                                             const float (&kappa)[8])
{
    constexpr int NU = 1 << N;
    Near1 lo[NU], hi[NU];
    lo[0] = hi[0] = {tile[tix]};
#pragma unroll
    for (int U = 1; U < NU; ++U) {
        lo[U] = {tile[tix - near_off<SY, SZ>(U)]};
        hi[U] = {tile[tix + near_off<SY, SZ>(U)]};
    }
    const float g = lo[0].v - dr;
    const Near1 D = near_dmax<N, Near1>(lo, hi, lo[0], {g}, {__fmul_rn(dD, dD)}, kappa);
    return __fmul_rn(g, g) / D.v;
}

// The same for the voxels at tix and tix + SY (two rows) at once.
template <int N, int SY, int SZ>
__device__ __forceinline__ void near_gamma2_pair(const float* tile, int tix, float dr0, float dr1, float dD0,
                                                 float dD1, const float (&kappa)[8], float& r0, float& r1)
{
    constexpr int NU = 1 << N;
    Near2 lo[NU], hi[NU];
    const float* p = tile + tix;
    const float e0 = p[0], e1 = p[SY];
    lo[0] = hi[0] = Near2::pack(e0, e1);
#pragma unroll
    for (int U = 1; U < NU; ++U) {
        const int o = near_off<SY, SZ>(U);
        lo[U] = Near2::pack(p[-o], p[SY - o]);
        hi[U] = Near2::pack(p[o], p[SY + o]);
    }
    const float g0 = e0 - dr0, g1 = e1 - dr1;
    const Near2 D = near_dmax<N, Near2>(lo, hi, lo[0], Near2::pack(g0, g1),
                                        Near2::pack(__fmul_rn(dD0, dD0), __fmul_rn(dD1, dD1)), kappa);
    float m0, m1;
    D.get(m0, m1);
    // (0, not 0 / 0, where the doses agree and dD^2 underflows)
    r0 = g0 != 0.f ? __fmul_rn(g0, g0) / m0 : 0.f;
    r1 = g1 != 0.f ? __fmul_rn(g1, g1) / m1 : 0.f;
}

}  // namespace gk
