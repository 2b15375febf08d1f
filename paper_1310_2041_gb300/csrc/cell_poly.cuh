// cell_poly.cuh -- the field inside one cell as a trilinear polynomial of the
// offset (shared by the step kernels, so that all form the same bits).
#pragma once

#include "hpf_internal.cuh"

namespace hpf {

// Ghosted-array index of the lower corner of cell (flx, fly, flz) (periodic
// image; see axis_gather for why no fix-up is needed).
__device__ __forceinline__ int cell_base(const MeshGeom& g, float flx, float fly, float flz) {
    const float fmx = (float)g.mx, fmy = (float)g.my, fmz = (float)g.mz;
    float wx = __fmaf_rn(-fmx, floorf((flx + 0.5f) * g.inv_m[0]), flx);
    float wy = __fmaf_rn(-fmy, floorf((fly + 0.5f) * g.inv_m[1]), fly);
    float wz = __fmaf_rn(-fmz, floorf((flz + 0.5f) * g.inv_m[2]), flz);
    wx = fminf(fmaxf(wx, 0.0f), fmx - 1.0f);
    wy = fminf(fmaxf(wy, 0.0f), fmy - 1.0f);
    wz = fminf(fmaxf(wz, 0.0f), fmz - 1.0f);
    return (int)wz * g.gxy + (int)wy * g.gx + (int)wx;
}

// The eight corners (x, y, z offsets in {0, 1}) of cell (flx, fly, flz).
struct Corners {
    float4 g000, g100, g010, g110, g001, g101, g011, g111;
};

// q: the cell's lower corner in the ghosted field array of one species.
__device__ __forceinline__ Corners load_corners_at(const float4* __restrict__ q, const MeshGeom& g) {
    Corners k;
    k.g000 = __ldg(q);
    k.g100 = __ldg(q + 1);
    k.g010 = __ldg(q + g.gx);
    k.g110 = __ldg(q + g.gx + 1);
    k.g001 = __ldg(q + g.gxy);
    k.g101 = __ldg(q + g.gxy + 1);
    k.g011 = __ldg(q + g.gxy + g.gx);
    k.g111 = __ldg(q + g.gxy + g.gx + 1);
    return k;
}

__device__ __forceinline__ Corners load_corners(const float4* __restrict__ Gt, const MeshGeom& g,
                                                float flx, float fly, float flz) {
    return load_corners_at(Gt + cell_base(g, flx, fly, flz), g);
}

// One component's polynomial c0 + c1 fx + c2 fy + c3 fz + c4 fx fy + c5 fx fz
// + c6 fy fz + c7 fx fy fz from its corner values: lo = c0..c3, hi = c4..c7.
#define HPF_CORNERS(k, comp) \
    k.g000.comp, k.g100.comp, k.g010.comp, k.g110.comp, k.g001.comp, k.g101.comp, k.g011.comp, \
        k.g111.comp
__device__ __forceinline__ void cell_coefs(float g000, float g100, float g010, float g110,
                                           float g001, float g101, float g011, float g111,
                                           float4& lo, float4& hi) {
    const float a2 = g010 - g000, a3 = g001 - g000, a6 = (g011 - g010) - a3;
    lo = make_float4(g000, g100 - g000, a2, a3);
    hi = make_float4((g110 - g100) - a2, (g101 - g100) - a3, a6,
                     ((g111 - g110) - (g101 - g100)) - a6);
}

// -(trilinear polynomial) of the cached cell at offset (fx, fy, fz).
__device__ __forceinline__ float cell_poly(const float4 lo, const float4 hi, float fx, float fy,
                                           float fz) {
    // lo = (c0, c1, c2, c3), hi = (c4, c5, c6, c7)
    float a = fmaf(fz, hi.w, hi.x);
    a = fmaf(fy, a, lo.y);
    a = fmaf(fz, hi.y, a);
    const float b = fmaf(fz, hi.z, lo.z);
    float v = fmaf(fx, a, lo.x);
    v = fmaf(fy, b, v);
    return fmaf(fz, lo.w, v);
}

// Friction and field force of one component, -fric v - poly in one rounding.
// Written out, here and in the packed form (pair_force): left to the compiler
// the product is fused in one kernel and not in another, and a run's bits then
// depend on which kernel its steps go through (seen at gamma m = 0.7, whose
// products round; at 1 they are exact).
__device__ __forceinline__ float drag_field(float fric, float v, float poly) {
    return fmaf(-fric, v, -poly);
}

}  // namespace hpf
