// Double-float (fp32 pair) arithmetic and the terrain clearance in it, shared by the rollout
// kernels.
#pragma once

#include "fmdp_internal.cuh"

namespace fmdp {

// exact sums of fp32 numbers
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
    s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}
__device__ __forceinline__ void fast_two_sum(float a, float b, float& s, float& e) {
    s = __fadd_rn(a, b);
    e = __fsub_rn(b, __fsub_rn(s, a));
}
// (hi, lo) += (dh, dl)
__device__ __forceinline__ void df_add(float& hi, float& lo, float dh, float dl) {
    float s, e;
    two_sum(hi, dh, s, e);
    e = __fadd_rn(e, __fadd_rn(lo, dl));
    fast_two_sum(s, e, hi, lo);
}

struct TerrainCell {  // heightmap cell under a successor, and the position in it
    int ix, iy;
    float ax, ay;
    float h00, h10, h01, h11;
};
__device__ __forceinline__ TerrainCell terrain_cell(float sx, float sy, float box0, float box1, float hm_sx, float hm_sy,
                                                    int hm_nx, int hm_ny) {
    TerrainCell t;
    const float ux = __fsub_rn(sx, box0), uy = __fsub_rn(sy, box1);
    t.ix = (int)floorf(__fmul_rn(ux, hm_sx)), t.iy = (int)floorf(__fmul_rn(uy, hm_sy));
    t.ix = min(max(t.ix, 0), hm_nx - 2);
    t.iy = min(max(t.iy, 0), hm_ny - 2);
    t.ax = fmaf(ux, hm_sx, -(float)t.ix);
    t.ay = fmaf(uy, hm_sy, -(float)t.iy);
    return t;
}
__device__ __forceinline__ void terrain_nodes(TerrainCell& t, const float* __restrict__ hm, int hm_nx) {
    const float* r0 = hm + (size_t)t.iy * hm_nx + t.ix;
    t.h00 = __ldg(r0);
    t.h10 = __ldg(r0 + 1);
    t.h01 = __ldg(r0 + hm_nx);
    t.h11 = __ldg(r0 + hm_nx + 1);
}
__device__ __forceinline__ float terrain_height(const TerrainCell& t) {
    const float bx = __fsub_rn(1.f, t.ax), by = __fsub_rn(1.f, t.ay);
    const float lo = fmaf(bx, t.h00, __fmul_rn(t.ax, t.h10)), hi = fmaf(bx, t.h01, __fmul_rn(t.ax, t.h11));
    return fmaf(by, lo, __fmul_rn(t.ay, hi));
}

// Heightmap origin, node spacing and nodes per metre as double-float.
struct DeckGrid {
    float bxh, bxl, byh, byl, cxh, cxl, cyh, cyl, sxh, sxl, syh, syl;
};
__device__ __forceinline__ DeckGrid deck_grid(const Model& m) {
    DeckGrid g;
    auto df = [](double v, float& h, float& l) {
        h = (float)v;
        l = (float)(v - (double)h);
    };
    const double wx = m.box[3] - m.box[0], wy = m.box[4] - m.box[1];
    const double nx = (double)(m.hm_nx - 1), ny = (double)(m.hm_ny - 1);
    df(m.box[0], g.bxh, g.bxl), df(m.box[1], g.byh, g.byl);
    df(wx / nx, g.cxh, g.cxl), df(wy / ny, g.cyh, g.cyl);
    df(nx / wx, g.sxh, g.sxl), df(ny / wy, g.syh, g.syl);
    return g;
}
// double-float products and sums (relative error of a few 2^-46)
__device__ __forceinline__ float2 df_mul(float2 a, float2 b) {
    const float p = __fmul_rn(a.x, b.x);
    const float e = fmaf(a.x, b.x, -p) + fmaf(a.x, b.y, __fmul_rn(a.y, b.x));
    float2 r;
    fast_two_sum(p, e, r.x, r.y);
    return r;
}
__device__ __forceinline__ float2 df_sum(float2 a, float2 b) {
    float s, e;
    two_sum(a.x, b.x, s, e);
    e = __fadd_rn(e, __fadd_rn(a.y, b.y));
    float2 r;
    fast_two_sum(s, e, r.x, r.y);
    return r;
}
__device__ __forceinline__ float2 df_diff(float a, float b) {
    float2 r;
    two_sum(a, -b, r.x, r.y);
    return r;
}

// Clearance penalty of a successor (double-float position) whose fp32 clearance lies in the FP64
// band (one lane; step k). The band is wide because fp32 coordinates are, and a path along the
// clearance limit enters it in a quarter of its steps; the FP64 evaluation takes some 5000
// cycles here. In double-float the clearance c is good to nanometres plus what the position
// has drifted from the exact state (one rounding per step), so both the decision c < clearance
// and the fp32 value of deck - c are those of FP64 unless one lies within that error of a
// threshold, or the position beside the cell t: then, and only then, FP64 decides. Returns the
// penalty, or -1 for FP64 to decide. Compared with FP64 on the host in test_deck_band_cpu.py.
static __device__ __noinline__ float deck_band(const Model& m, const DeckGrid g, const TerrainCell t, float hx, float lx, float hy,
                                        float ly, float hz, float lz, int k) {
    // position in the cell: offset from its node (b + i c), times the nodes per metre
    auto frac = [](float h, float l, int i, float bh, float bl, float ch, float cl, float sh, float sl) {
        const float2 at = df_mul(make_float2((float)i, 0.f), make_float2(ch, cl));
        const float2 u = df_sum(df_sum(make_float2(h, l), make_float2(-bh, -bl)), make_float2(-at.x, -at.y));
        return df_mul(u, make_float2(sh, sl));
    };
    const float2 ax = frac(hx, lx, t.ix, g.bxh, g.bxl, g.cxh, g.cxl, g.sxh, g.sxl);
    const float2 ay = frac(hy, ly, t.iy, g.byh, g.byl, g.cyh, g.cyl, g.syh, g.syl);
    // the cell comes from an fp32 position: within that rounding of a node line it may be the
    // neighbour of the one FP64 takes, whose surface is another one (not on the grid's border,
    // where FP64 goes on with the last cell too)
    auto beside = [](float2 f, int i, int n) {
        return (f.x < 0.f && i > 0) || ((f.x > 1.f || (f.x == 1.f && f.y > 0.f)) && i < n - 2);
    };
    if (beside(ax, t.ix, m.hm_nx) || beside(ay, t.iy, m.hm_ny)) return -1.f;
    const float2 lo = df_sum(make_float2(t.h00, 0.f), df_mul(ax, df_diff(t.h10, t.h00)));
    const float2 hi = df_sum(make_float2(t.h01, 0.f), df_mul(ax, df_diff(t.h11, t.h01)));
    const float2 T = df_sum(lo, df_mul(ay, df_sum(hi, make_float2(-lo.x, -lo.y))));
    const float2 c = df_sum(make_float2(hz, lz), make_float2(-T.x, -T.y));
    const float2 over = df_sum(c, make_float2(-(float)m.clearance, -(float)(m.clearance - (double)(float)m.clearance)));
    const float deckh = (float)m.deck;
    const float2 V = df_sum(make_float2(deckh, (float)(m.deck - (double)deckh)), make_float2(-c.x, -c.y));
    // error of c: the position's drift times the slope, and the arithmetic above
    const float H = fmaxf(fmaxf(fabsf(t.h00), fabsf(t.h10)), fmaxf(fabsf(t.h01), fabsf(t.h11)));
    const float slope = 1.f + 4.f * H * fmaxf(g.sxh, g.syh);
    const float err = 1e-14f * (float)(k + 2) * (fabsf(hx) + fabsf(hy) + fabsf(hz)) * slope + 1e-11f * (H + fabsf(hz) + deckh) +
                      1e-12f * slope * (fabsf(hx) + fabsf(hy) + fabsf(g.bxh) + fabsf(g.byh));
    // half the spacing of fp32 numbers at V: the rounding of deck - c is certain if |V.y| is clear of it
    const float half = 0.5f * (__uint_as_float(__float_as_uint(fabsf(V.x)) + 1u) - fabsf(V.x));
    if (fabsf(over.x) > 2.f * err) {
        if (over.x > 0.f) return 0.f;
        if (fabsf(V.y) < half - 2.f * err && V.x > 1.f) return V.x;
    }
    return -1.f;
}

}  // namespace fmdp
