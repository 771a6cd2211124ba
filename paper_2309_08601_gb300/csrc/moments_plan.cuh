// Which form of stage (a) takes which radial bins, and the side of the cell grid that the forms share
// (host arithmetic only).
#pragma once

#include <math.h>

#include <algorithm>

#include "moments_far.cuh"

namespace mp3 {

// The sector form (moments_far.cu) takes the bins [b_far, b_hi): groups of eight centres in strips of
// `rows` cell rows and at most `cols` columns, on cells of side `side`.
struct FarPlan {
    int b_far = 0, rows = 1, cols = 1;
    int b[kFarPlans + 1] = {0};  // bins [b[v + 1], b[v]) take variant v (b[0] = b_hi)
    double side = 1.0;
};

struct MomentsPlanInput {
    int n_max, nz;
    bool fp64, sectors;    // sectors: the sector form may be taken (FP32 only)
    int occupancy;         // configured galaxies per cell (0: automatic)
    const long long* e2q;  // all bins' squared edges
    int b_lo, b_hi;        // bins computed
    int64_t n, nc;         // galaxies, centres
    double extent;         // the longer side of the galaxies' extent, quanta
    double area, carea;    // of the extents of the galaxies and of the centres, quanta^2
};

// the warp-per-centre form takes [b_lo, b_near), the block-per-centre form [b_near, far.b_far)
struct MomentsPlan {
    FarPlan far;
    int b_near = 0;
    double side = 1.0;  // the grid's side is its ceiling
};

// largest angle from a sector's axis for which the terms beyond PW (PAB) of every order up to
// 2 n_max (n_max + 3) stay below 3e-8: m delta_max <= x(P), the argument at which the Bessel
// functions J_p, p >= P, sum to half of that
inline double far_dmax(int n_max, int v)
{
    auto x = [](int P) { return P >= 32 ? 15.5 : P >= 28 ? 12.5 : P >= 24 ? 9.6 : P >= 20 ? 6.9 : P >= 18 ? 5.6 : P >= 16 ? 4.45 : 3.3; };
    return std::min({0.5, x(kFarPW[v]) / std::max(2 * n_max, 1), x(kFarPAB[v]) / (n_max + 3)});
}

// Expected neighbours of a (centre, bin) below which the warp-per-centre form (moments_near.cu) is
// faster than the block-per-centre form. FP32: about 300 + 16 N warp instructions a bin against 300 n_max +
// n_max N / 2 at n_max 30; the line is flat (36 to 150 n_max: within 1 %). FP64: both form about as many of the
// 16-cycle instructions a member, the block-per-centre form has its reduction on top. Lines at 100, 400,
// 800, 1600, 3200 neighbours: 12 000 galaxies, n_max 10 14.6, 14.3, 14.23, 14.20, 14.19 ms, six catalogs in
// three z-bins 55.2, 54.0, 52.95, 52.96, 53.0; 20 000 galaxies up to 40', n_max 20 164.5, 164.4, -, 165.4, 167.5,
// n_max 30 263, 260, -, 258.6, 258.0.
inline double near_line(int n_max, bool fp64) { return fp64 ? 1000.0 : std::max(60.0, 36.0 * n_max); }

// estimated warp instructions of a (centre, bin) with N neighbours by the cheaper of those two forms; which of
// them runs is near_line's decision, from the measurements (between the two lines they differ by 1 % of a call)
inline double small_cost(int n_max, double N)
{
    const int sw = std::max(2 * n_max, n_max + 3) / 16 + 1, sab = (n_max + 3) / 16 + 1;
    return std::min(300.0 + (2.0 + 2.5 * sw + sab) * N, 300.0 * n_max + 0.5 * n_max * N);
}

// least: the smallest cell side the rest of the call allows
inline FarPlan plan_far(const MomentsPlanInput& in, double least)
{
    FarPlan f;
    f.b_far = in.b_hi;
    if (!in.sectors || in.nc < 1 || in.n >= (1 << 27)) return f;  // 32-bit byte offsets into the sorted catalog
    const double rho = (double)in.n / in.nz / in.area;  // galaxies per quantum^2 and z-bin
    const double occ = in.occupancy > 0 ? (double)in.occupancy : 1.0;
    f.side = std::max(least, sqrt(occ / rho));
    const double per_cell = (double)in.nc / in.carea * f.side * f.side;  // centres
    f.rows = (int)std::min(4.0, std::max(1.0, floor(sqrt(8.0 / per_cell) + 0.5)));
    f.cols = (int)std::min(5.0, ceil(8.0 / (per_cell * f.rows)) + 1.0);
    // sparse centres would leave most lanes of a group empty
    if (per_cell * f.rows * f.cols < 4.0) return f;
    // the direction from a centre to a galaxy differs from the sector's axis by at most half a
    // sector plus the angle the cell's and the group's extents subtend
    const double reach = f.side * (0.7072 + 0.5 * sqrt((double)f.rows * f.rows + (double)f.cols * f.cols)) + 8.0;
    int b = in.b_hi;
    f.b[0] = in.b_hi;
    for (int v = 0; v < kFarPlans; ++v) {
        const int sectors = kFarSectors[v], terms = kFarPW[v] + 2 * kFarPAB[v];
        const double free_angle = far_dmax(in.n_max, v) - M_PI / sectors;
        const double r_min = free_angle > 0.0 ? reach / sin(free_angle) : 1e300;
        while (b > in.b_lo && (double)in.e2q[b - 1] >= r_min * r_min) {
            // per centre: the sectors' enumeration and reduction, the FFT and orders, the pairs
            const double N = M_PI * rho * (double)(in.e2q[b] - in.e2q[b - 1]);
            const double cost = 150.0 * sectors + 0.35 * terms * sectors + N * (1.25 * terms + 30.0) / 24.0;
            if (cost >= small_cost(in.n_max, N)) break;
            --b;
        }
        f.b[v + 1] = b;
    }
    f.b_far = b;
    return f;
}

// ~4 galaxies per cell and z-bin, about one with sector bins, and at most kMaxRows cell rows per annulus of the
// bins below them (the block-per-centre form keeps a list of rows; for the sector form coarser cells are no
// loss at such distances: 200' to 400' at 8.6 galaxies per arcmin^2, n_max 30 8.3 ms, without the limit 8.8).
// The sector form's angles hold for the side it was planned with, so where the limit asks for a larger one it
// is planned again, each time with a larger side. With n_max 50 and a first edge at 200' the angles of the
// first plan would reach 0.063 on those cells, 0.056 is what its terms allow.
inline MomentsPlan plan_moments(const MomentsPlanInput& in)
{
    MomentsPlan p;
    const double occ = in.occupancy > 0 ? (double)in.occupancy : 4.0;
    // at most 2^26 cells and 2^22 - 4 columns or rows: the column arithmetic of sector.cuh (near_int) is FP32
    double least = std::max({1.0, sqrt(in.area * in.nz / (double)(1 << 26)), in.extent / (double)((1 << 22) - 5)});
    for (;;) {
        p.far = plan_far(in, least);
        const bool sectors = p.far.b_far < in.b_hi;
        const double rows = (2.0 * sqrt((double)in.e2q[p.far.b_far]) + 16.0) / (kMaxRows - 4);
        p.side = sectors ? p.far.side : std::max({least, rows, sqrt(in.area * occ / std::max(1.0, (double)in.n / in.nz))});
        if (rows <= p.side) break;
        least = rows;
    }
    p.b_near = in.b_lo;
    while (p.b_near < p.far.b_far &&
           M_PI * (double)in.n / in.nz / in.area * (double)(in.e2q[p.b_near + 1] - in.e2q[p.b_near]) <
               near_line(in.n_max, in.fp64))
        ++p.b_near;
    return p;
}

}  // namespace mp3
