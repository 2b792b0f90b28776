// stencil.cuh -- the per-point arithmetic of the 2D step, shared by every 2D
// kernel so that all of them produce the same bits.  The evaluation order is
// fixed by explicit fmaf calls rather than left to contraction.
#pragma once

#include "internal.h"

namespace wave {

// Four points as two pairs, for the packed FP32 instructions (FADD2, FMUL2,
// FFMA2): each half rounds as the scalar instruction does, and one issue slot
// does the work of two.  The pairs of a 16-byte load lie in even registers.
struct Quad {
    float2 a, b;
};
__device__ __forceinline__ Quad quad(float4 v) { return {make_float2(v.x, v.y), make_float2(v.z, v.w)}; }
__device__ __forceinline__ Quad quad(const float* v) { return {make_float2(v[0], v[1]), make_float2(v[2], v[3])}; }
__device__ __forceinline__ Quad quad(float v) { return {make_float2(v, v), make_float2(v, v)}; }
__device__ __forceinline__ Quad operator+(Quad x, Quad y) { return {__fadd2_rn(x.a, y.a), __fadd2_rn(x.b, y.b)}; }
__device__ __forceinline__ Quad operator*(Quad x, Quad y) { return {__fmul2_rn(x.a, y.a), __fmul2_rn(x.b, y.b)}; }
__device__ __forceinline__ Quad fma(Quad x, Quad y, Quad z)
{
    return {__ffma2_rn(x.a, y.a, z.a), __ffma2_rn(x.b, y.b, z.b)};
}
__device__ __forceinline__ void unquad(Quad q, float* o)
{
    o[0] = q.a.x;
    o[1] = q.a.y;
    o[2] = q.b.x;
    o[3] = q.b.y;
}

// The x part of the 8th-order Laplacian (unit spacing) of 4 consecutive points:
// c0 w + c_k (w_{-k} + w_{+k}) for k = 1..4 in that order; w[0..11] are the row
// values x-4 .. x+7 (the points are w[4..7]).  Odd neighbours straddle register
// pairs and stay scalar.
__device__ __forceinline__ Quad lap_x(const float* w, float c0)
{
    Quad l = quad(c0) * quad(w + 4);
    l.a.x = fmaf(kC1, w[3] + w[5], l.a.x);
    l.a.y = fmaf(kC1, w[4] + w[6], l.a.y);
    l.b.x = fmaf(kC1, w[5] + w[7], l.b.x);
    l.b.y = fmaf(kC1, w[6] + w[8], l.b.y);
    l = fma(quad(kC2), quad(w + 2) + quad(w + 6), l);
    l.a.x = fmaf(kC3, w[1] + w[7], l.a.x);
    l.a.y = fmaf(kC3, w[2] + w[8], l.a.y);
    l.b.x = fmaf(kC3, w[3] + w[9], l.b.x);
    l.b.y = fmaf(kC3, w[4] + w[10], l.b.y);
    return fma(quad(kC4), quad(w) + quad(w + 8), l);
}

// 8th-order Laplacian (unit spacing) of 4 consecutive x points.  w as in lap_x;
// zn(k, U, D) gives the values k rows above and k rows below the 4 points,
// k = 1..4, and is called in the loop so that the loads interleave with the
// arithmetic.  Order: 2 c0 w, then along x, then + c_k (U + D) for k = 1..4.
template <class ZN>
__device__ __forceinline__ void lap4(const float* w, ZN zn, float* lap)
{
    const float ck[5] = {kC0, kC1, kC2, kC3, kC4};
    Quad l = lap_x(w, 2.0f * kC0);
#pragma unroll
    for (int k = 1; k <= 4; ++k) {
        float4 U, D;
        zn(k, U, D);
        l = fma(quad(ck[k]), quad(U) + quad(D), l);
    }
    unquad(l, lap);
}

// 3D Laplacian of 4 consecutive x points: w as in lap_x; zn(k, Up, Dn, Zu, Zd)
// returns the 4 points' values k rows away in y (Up, Dn) and k planes away in
// z (Zu, Zd).  Order: 3 c0 w, along x, then + c_k ((Up + Dn) + (Zu + Zd)) for
// k = 1..4.
template <class ZN>
__device__ __forceinline__ void lap4_3d(const float* w, ZN zn, float* lap)
{
    const float ck[5] = {kC0, kC1, kC2, kC3, kC4};
    Quad l = lap_x(w, 3.0f * kC0);
#pragma unroll
    for (int k = 1; k <= 4; ++k) {
        float4 Up, Dn, Zu, Zd;
        zn(k, Up, Dn, Zu, Zd);
        l = fma(quad(ck[k]), (quad(Up) + quad(Dn)) + (quad(Zu) + quad(Zd)), l);
    }
    unquad(l, lap);
}

// 1 / x for the sponge factor (x = 1 + eps >= 1): the hardware approximation
// refined by one Newton-Raphson step for the reciprocal, r <- r + r (1 - x r).
// The result is within about 2^-24 relative of 1 / x before its rounding, so it
// is the rounded reciprocal except next to a rounding boundary, and unbiased
// there.  Three instructions instead of the correctly rounded sequence: the
// 3D steps and the batch sweeps evaluate it for every point at every step.
__device__ __forceinline__ float rcp_sponge(float x)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return fmaf(r, fmaf(-x, r, 1.0f), r);
}

// Leapfrog update of one point: (kap lap + eps um + 2 c - um - src) * inv,
// inv = 1 / (1 + eps); src is the Born secondary source (zero elsewhere).
__device__ __forceinline__ float leap1(float c, float um, float lap, float kap, float eps, float inv, float src)
{
    const float t = fmaf(kap, lap, fmaf(eps, um, fmaf(2.0f, c, -um)));
    return (t - src) * inv;
}

// The same for 4 points.
__device__ __forceinline__ void update4(const float* c, const float* um, const float* lap, const float* kap,
                                        const float* eps, const float* inv, const float* src, float* out)
{
    float t[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) t[e] = fmaf(2.0f, c[e], -um[e]);
    unquad(fma(quad(kap), quad(lap), fma(quad(eps), quad(um), quad(t))), t);
#pragma unroll
    for (int e = 0; e < 4; ++e) t[e] -= src[e];
    unquad(quad(t) * quad(inv), out);
}

// The same update where the sponge is absent (eps = 0, inv = 1) and there is no
// secondary source: equal to update4 up to the sign of zero results.
__device__ __forceinline__ void update4_interior(const float* c, const float* um, const float* lap, const float* kap,
                                                 float* out)
{
#pragma unroll
    for (int e = 0; e < 4; ++e) out[e] = fmaf(kap[e], lap[e], fmaf(2.0f, c[e], -um[e]));
}

}  // namespace wave
