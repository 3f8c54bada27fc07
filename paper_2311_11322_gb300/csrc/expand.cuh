// expand.cuh -- per-sphere quantities formed by more than one kernel, bitwise
// identical wherever they are formed: sphere centres from the per-aggregate
// record, gravity from the integer accumulators.
#pragma once

#include "dem_internal.h"
#include "devmath.cuh"

namespace dem {

// Sphere centre relative to the pile frame, r_i - O = (r_A - O) + R(q_A) b_i.
// Mixed: float-float, bitwise identical wherever it is inlined.
__device__ __forceinline__ void expand_mixed(const AggRecMixed &rec, float4 bh, float4 bl,
                                             ff &px, ff &py, ff &pz)
{
    ff rx = ff_dot3(rec.Rh + 0, rec.Rl + 0, bh.x, bh.y, bh.z, bl.x, bl.y, bl.z);
    ff ry = ff_dot3(rec.Rh + 3, rec.Rl + 3, bh.x, bh.y, bh.z, bl.x, bl.y, bl.z);
    ff rz = ff_dot3(rec.Rh + 6, rec.Rl + 6, bh.x, bh.y, bh.z, bl.x, bl.y, bl.z);
    ff cx = {rec.ch[0], rec.cl[0]}, cy = {rec.ch[1], rec.cl[1]}, cz = {rec.ch[2], rec.cl[2]};
    px = ff_add(cx, rx);
    py = ff_add(cy, ry);
    pz = ff_add(cz, rz);
}

__device__ __forceinline__ double3 expand_64(const AggRec64 &rec, const double *b)
{
    const double *R = rec.R;
    double x = __fma_rn(R[2], b[2], __fma_rn(R[1], b[1], __dmul_rn(R[0], b[0])));
    double y = __fma_rn(R[5], b[2], __fma_rn(R[4], b[1], __dmul_rn(R[3], b[0])));
    double zz = __fma_rn(R[8], b[2], __fma_rn(R[7], b[1], __dmul_rn(R[6], b[0])));
    return d3(__dadd_rn(rec.c[0], x), __dadd_rn(rec.c[1], y), __dadd_rn(rec.c[2], zz));
}

// Planet's force on a sphere of mass m at r (space frame) from the planet at P:
// GM m (P - r) / |P - r|^3.
__device__ __forceinline__ double3 planet_force(double GM, double m, double3 P, double3 r)
{
    const double3 d = P - r;
    return (GM * m * inv_r3(dot(d, d))) * d;
}

// Mixed symmetric gravity: sphere i's force F = G m sum 2^-k from its integer
// accumulators, which are cleared for the next step.
struct GaccSums {
    longlong2 xy, zw;
};
__device__ __forceinline__ GaccSums gacc_load(const Arrays &a, int64_t i)
{
    const longlong2 *g = (const longlong2 *)(a.gacc + 4 * i);
    return GaccSums{g[0], g[1]};
}
__device__ __forceinline__ dbl4 gacc_force(const Arrays &a, const PileStatic &S, int64_t i, const GaccSums &s)
{
    longlong2 *g = (longlong2 *)(a.gacc + 4 * i);
    g[0] = make_longlong2(0, 0);
    g[1] = make_longlong2(0, 0);
    const double gm = S.G * a.m64[i] * S.ginv;
    return make_dbl4(gm * (double)s.xy.x, gm * (double)s.xy.y, gm * (double)s.zw.x, 0.0);
}

}  // namespace dem
