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

// The record of aggregate g by four 32-byte loads (field by field it is 30
// four-byte ones: 53 us for the gather of the 1M lattice, 51 so).
__device__ __forceinline__ AggRecMixed load_rec(const AggRecMixed *recs, int64_t g)
{
    static_assert(sizeof(AggRecMixed) == 128, "four 32-byte loads");
    const float4 *r = (const float4 *)(recs + g);
    AggRecMixed rec;
    float4 v[8];
#pragma unroll
    for (int k = 0; k < 4; ++k) ld_f4x2(r + 2 * k, v[2 * k], v[2 * k + 1]);
    const float f[32] = {v[0].x, v[0].y, v[0].z, v[0].w, v[1].x, v[1].y, v[1].z, v[1].w,
                         v[2].x, v[2].y, v[2].z, v[2].w, v[3].x, v[3].y, v[3].z, v[3].w,
                         v[4].x, v[4].y, v[4].z, v[4].w, v[5].x, v[5].y, v[5].z, v[5].w,
                         v[6].x, v[6].y, v[6].z, v[6].w, v[7].x, v[7].y, v[7].z, v[7].w};
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        rec.Rh[k] = f[k];
        rec.Rl[k] = f[9 + k];
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        rec.ch[k] = f[18 + k];
        rec.cl[k] = f[21 + k];
        rec.vb[k] = f[24 + k];
        rec.w[k] = f[27 + k];
    }
    return rec;
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
