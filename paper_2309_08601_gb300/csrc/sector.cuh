// Neighbours of a small group of centres in one radial bin, one angular sector at a time.
//
// The group's centres lie in a rectangle a few cells wide (reference point (gx, gy), half extents
// (hx, hy)). The cells of the catalog's grid are split into S sectors by the direction of the cell's
// centre from the reference point: every cell belongs to exactly one sector, because both sectors
// of a boundary evaluate the same column bound for it. sector_runs gives a lane its cell row's part
// of a sector, cut by the annulus grown by the group's extents, as at most two runs of the sorted
// catalog.
#pragma once

#include "common.cuh"

namespace mp3 {

// geometry shared by every sector of one (group, bin)
struct SectorGeom {
    float gx, gy, hx, hy;  // reference point and half extents of the group, quanta from the grid origin
    float Ro, Ri;          // outer and inner radius of the annulus, quanta
    float S, iS;           // cell side and its inverse
    int ncx, ncy;
};

// nearest integer of |x| < 2^22 by the FP32 addition that rounds it into the mantissa: the conversion
// and rounding instructions run on the FP64 pipe (16 cycles a warp), and the column bounds only have
// to be the same function on both sides of a ray
__host__ __device__ __forceinline__ int near_int(float x)
{
    const float y = x + 12582912.0f;
#ifdef __CUDA_ARCH__
    return __float_as_int(y) - 0x4b400000;
#else
    return (int)(y - 12582912.0f);
#endif
}

// first and last row of a sector (as FP32 integers); sn0 <= sn1: the sines of its rays
__host__ __device__ __forceinline__ void sector_rows(const SectorGeom& g, bool upper, float sn0, float sn1, float& iy0,
                                                     float& iy1)
{
    const float m = 0.75f * g.S + g.hx + g.hy + 8.0f;  // cell half diagonal and group extents
    const float ya = fmaxf((g.Ri - m) * sn0, 0.0f) - 8.0f, yb = (g.Ro + m) * sn1 + 8.0f;
    const float r0 = upper ? (g.gy + ya) : (g.gy - yb), r1 = upper ? (g.gy + yb) : (g.gy - ya);
    iy0 = fmaxf(floorf(r0 * g.iS - 0.5f), 0.0f);
    iy1 = fminf(ceilf(r1 * g.iS - 0.5f), (float)(g.ncy - 1));
}

// the runs (start, length) of cell row iy that meet the annulus of some centre of the group, within
// columns [c0, c1]; dy = the row's centre from the reference point
__host__ __device__ __forceinline__ void annulus_runs(const SectorGeom& g, float iy, float dy, int c0, int c1,
                                                      const int* __restrict__ row_start, int& st0, int& n0, int& st1,
                                                      int& n1)
{
    const float ady = fabsf(dy), wide = (float)(g.ncx + 1), x = g.gx * g.iS;
    const float half = 0.5f * g.S, pad = 8.0f + 2e-6f * g.Ro;
    const float dymin = fmaxf(ady - half - g.hy, 0.0f), dymax = ady + half + g.hy;
    const float o2 = g.Ro * g.Ro * 1.000002f - dymin * dymin;
    if (!(o2 >= 0.0f)) return;
    const float dxo = (sqrtf(o2) + half + g.hx + pad) * g.iS;
    c0 = max(c0, near_int(fmaxf(x - dxo, 0.0f)));
    c1 = min(c1, near_int(fminf(x + dxo, wide) - 1.0f));
    if (c0 > c1) return;
    int h0 = 1, h1 = 0;  // columns wholly inside the inner radius for every centre
    const float i2 = g.Ri * g.Ri * 0.999998f - dymax * dymax;
    if (i2 > 0.0f) {
        const float dxi = (sqrtf(i2) - half - g.hx - pad) * g.iS;
        if (dxi > 0.0f) {
            h0 = near_int(fmaxf(x - dxi, 0.0f));
            h1 = near_int(fminf(x + dxi, wide) - 1.0f);
        }
    }
    const int* cs = row_start + near_int(iy) * (long long)g.ncx;
    if (h0 <= h1 && h0 <= c1 && h1 >= c0) {
        if (h0 > c0) {
            st0 = cs[c0];
            n0 = cs[h0] - st0;
        }
        if (h1 < c1) {
            st1 = cs[h1 + 1];
            n1 = cs[c1 + 1] - st1;
        }
    } else {
        st0 = cs[c0];
        n0 = cs[c1 + 1] - st0;
    }
}

// the same for the part of the row in the sector between the rays of cotangent ct0 > ct1
// (first: the sector's ray 0 is the x axis, last: its ray 1 is the negative x axis)
__host__ __device__ __forceinline__ void sector_runs(const SectorGeom& g, bool upper, bool first, bool last, float ct0,
                                                     float ct1, float iy, const int* __restrict__ row_start, int& st0,
                                                     int& n0, int& st1, int& n1)
{
    n0 = n1 = st0 = st1 = 0;
    const float dy = (iy + 0.5f) * g.S - g.gy;
    if ((dy > 0.0f) != upper) return;
    // a column belongs to the sector if its centre lies between the rays; q is the first column
    // right of a ray, the same expression, rounded the same way, for the sectors on both of its sides
    const float wide = (float)(g.ncx + 1), x = g.gx * g.iS, t = fabsf(dy) * (upper ? g.iS : -g.iS);
    int c0 = 0, c1 = g.ncx - 1;
    const int q0 = near_int(fminf(fmaxf(fmaf(t, ct0, x), -1.0f), wide));
    const int q1 = near_int(fminf(fmaxf(fmaf(t, ct1, x), -1.0f), wide));
    if (upper) {
        if (!first) c1 = min(c1, q0 - 1);
        if (!last) c0 = max(c0, q1);
    } else {
        if (!first) c0 = max(c0, q0);
        if (!last) c1 = min(c1, q1 - 1);
    }
    annulus_runs(g, iy, dy, c0, c1, row_start, st0, n0, st1, n1);
}

}  // namespace mp3
