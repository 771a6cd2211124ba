// The direct estimator of the third-order aperture mass (paper Sec. 5.3, Eq. MapDirectEstimator),
// an estimate independent of the 3PCF route: at an aperture centre c and radii (t1, t2, t3),
//   num = sum over distinct i, j, k of w_i w_j w_k Q_t1(r_i) Q_t2(r_j) Q_t3(r_k) gt_i gt_j gt_k,
//   den = the same sum without the tangential shears,
// with r_i = |x_i - c|, gt_i the tangential shear about c (gt = -Re(gamma e^{-2 i zeta}), zeta the
// polar angle of x_i - c, Eq. gammatx_def) and Q the filter of Eq. CrittendenQ,
// Q_t(r) = r^2 / (4 pi t^4) exp(-r^2 / (2 t^2)); galaxies farther than rcut from c are left out
// (the paper keeps galaxies within 4 max(t)). The sums over distinct triplets follow from seven
// sums per aperture by inclusion-exclusion over the coincidences i = j, i = k, j = k: with
// A = sum a_i, AB = sum a_i b_i, ABC = sum a_i b_i c_i (a, b, c the factors of the three slots),
//   sum_{i, j, k distinct} a_i b_j c_k = A B C - AB C - AC B - BC A + 2 ABC,
// so each aperture costs one pass over the catalog. Block per (aperture, radii triple), threads
// over the galaxies, FP64 sums reduced over the block.
#include <math.h>

#include <algorithm>

#include "common.cuh"

namespace mp3 {

constexpr int kDirThreads = 256;

__global__ void __launch_bounds__(kDirThreads) map3_direct_kernel(int64_t n, const int32_t* __restrict__ xq,
                                                                  const int32_t* __restrict__ yq,
                                                                  const float* __restrict__ g1,
                                                                  const float* __restrict__ g2,
                                                                  const float* __restrict__ w, double quantum,
                                                                  int n_ap, const double* __restrict__ centres,
                                                                  const double* __restrict__ theta,
                                                                  double rcut_factor, double* __restrict__ out)
{
    __shared__ double red[14][kDirThreads / 32];
    const int64_t job = blockIdx.x;  // centre * n_ap + radii triple
    const int64_t t = job / n_ap;
    const int a = (int)(job % n_ap);
    const double cx = centres[2 * t], cy = centres[2 * t + 1];
    double th[3], inv2[3], nrm[3];
    for (int l = 0; l < 3; ++l) {
        th[l] = theta[3 * a + l];
        inv2[l] = 1.0 / (2.0 * th[l] * th[l]);
        nrm[l] = 1.0 / (4.0 * M_PI * th[l] * th[l] * th[l] * th[l]);
    }
    const double rcut = rcut_factor * fmax(th[0], fmax(th[1], th[2]));
    double s[14];
#pragma unroll
    for (int v = 0; v < 14; ++v) s[v] = 0.0;
    for (int64_t i = threadIdx.x; i < n; i += blockDim.x) {
        const double dx = (double)xq[i] * quantum - cx, dy = (double)yq[i] * quantum - cy;
        const double r2 = dx * dx + dy * dy;
        if (r2 == 0.0 || sqrt(r2) > rcut) continue;
        // tangential shear about c: -Re((g1 + i g2) (dx - i dy)^2 / r^2)
        const double gt = -((double)g1[i] * (dx * dx - dy * dy) + 2.0 * (double)g2[i] * dx * dy) / r2;
        double b[3], c[3];
#pragma unroll
        for (int l = 0; l < 3; ++l) {
            b[l] = (double)w[i] * r2 * nrm[l] * exp(-r2 * inv2[l]);  // w Q_tl(r)
            c[l] = b[l] * gt;
        }
        s[0] += c[0];
        s[1] += c[1];
        s[2] += c[2];
        s[3] += c[0] * c[1];
        s[4] += c[0] * c[2];
        s[5] += c[1] * c[2];
        s[6] += c[0] * c[1] * c[2];
        s[7] += b[0];
        s[8] += b[1];
        s[9] += b[2];
        s[10] += b[0] * b[1];
        s[11] += b[0] * b[2];
        s[12] += b[1] * b[2];
        s[13] += b[0] * b[1] * b[2];
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int v = 0; v < 14; ++v) {
        double x = s[v];
        for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
        if (lane == 0) red[v][warp] = x;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double q[14];
        for (int v = 0; v < 14; ++v) {
            q[v] = 0.0;
            for (int k = 0; k < kDirThreads / 32; ++k) q[v] += red[v][k];
        }
        out[2 * job] = q[0] * q[1] * q[2] - q[3] * q[2] - q[4] * q[1] - q[5] * q[0] + 2.0 * q[6];
        out[2 * job + 1] = q[7] * q[8] * q[9] - q[10] * q[9] - q[11] * q[8] - q[12] * q[7] + 2.0 * q[13];
    }
}

// The same sums from a cell-sorted copy of the catalog: a block per (aperture, radii triple) reads only
// the cells its cut-off circle meets, warps over the cell rows (each a contiguous run), lanes over the
// galaxies. Bound by FP64 arithmetic on the galaxies inside (two FP64 lanes per SM and cycle), so a
// radius that occurs twice in a triple is evaluated once, and equal radii need three powers of one
// factor. 200 000 galaxies, 900 apertures x 3 triples: 67.5 ms by scanning the catalog, 2.7 ms by cells.
// A row with more than `limit` galaxies in the circle (a strip, an outlier that makes the cells huge, a cluster) is
// left out by this kernel, as the block would wait for the one warp that has it; the aperture is noted and
// map3_direct_long_kernel does it again with such rows taken by the whole block. Uneven fields of 200 000 galaxies,
// by scanning and by cells: an outlier 50 and 33 ms, a strip 79 and 13, a cluster 23 and 12. (With both
// loops in one kernel the even field took 1 to 2 % longer.)
template <int R>  // distinct radii of the triple: 1 (all equal), 2 (the first two equal) or 3
__device__ __forceinline__ void direct_sums(double (&s)[14], const double (&b)[3], double gt)
{
    double c[3];
#pragma unroll
    for (int l = 0; l < R; ++l) c[l] = b[l] * gt;
    const int i1 = R == 3 ? 1 : 0, i2 = R - 1;
    s[0] += c[0];
    s[7] += b[0];
    const double c01 = c[0] * c[i1], b01 = b[0] * b[i1];
    s[3] += c01;
    s[10] += b01;
    s[6] += c01 * c[i2];
    s[13] += b01 * b[i2];
    if (R > 1) {
        s[2] += c[i2];
        s[4] += c[0] * c[i2];
        s[9] += b[i2];
        s[11] += b[0] * b[i2];
    }
    if (R > 2) {
        s[1] += c[1];
        s[5] += c[1] * c[2];
        s[8] += b[1];
        s[12] += b[1] * b[2];
    }
}

// BLOCK: long rows by the block, else not at all; returns whether the calling warp has left one out
template <int R, bool BLOCK>
__device__ __forceinline__ bool direct_cells(double (&s)[14], int limit, const int2* __restrict__ pos,
                                             const float4* __restrict__ gw, const int* __restrict__ start,
                                             const GridDesc& g, double quantum, double cx, double cy, double rcut,
                                             double r2max, const double (&inv2)[3], const double (&nrm)[3])
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // in cells, two quanta wider than the circle; fmin and fmax drop NaNs (the whole grid)
    const double is = 1.0 / (double)g.side, xc = (cx / quantum - (double)g.x0) * is, yc = (cy / quantum - (double)g.y0) * is;
    const double rc = (rcut / quantum + 2.0) * is * (1.0 + 1e-9);
    const int iy0 = (int)fmin(fmax(floor(yc - rc), 0.0), (double)g.ncy), iy1 = (int)fmax(fmin(floor(yc + rc), (double)g.ncy - 1.0), -1.0);
    bool later = false;
#pragma unroll 1
    for (int pass = 0; pass < (BLOCK ? 2 : 1); ++pass) {
        const int first = pass ? (int)threadIdx.x : lane, step = pass ? kDirThreads : 32;
        for (int iy = iy0 + (pass ? 0 : warp); iy <= iy1; iy += pass ? 1 : kDirThreads / 32) {
            const double dy = fmax(fmax((double)iy - yc, yc - (double)iy - 1.0), 0.0);
            const double hx = sqrt(fmax(rc * rc - dy * dy, 0.0)) + 1e-6 * rc;
            const int ix0 = (int)fmin(fmax(floor(xc - hx), 0.0), (double)g.ncx), ix1 = (int)fmax(fmin(floor(xc + hx), (double)g.ncx - 1.0), -1.0);
            if (ix0 > ix1) continue;
            const int k0 = start[iy * g.ncx + ix0], k1 = start[iy * g.ncx + ix1 + 1];
            if ((k1 - k0 > limit) != (pass == 1)) {
                later = true;
                continue;
            }
            for (int k = k0 + first; k < k1; k += step) {
                const int2 p = pos[k];
                const double dx = (double)p.x * quantum - cx, dyk = (double)p.y * quantum - cy;
                const double r2 = dx * dx + dyk * dyk;
                if (r2 == 0.0 || r2 > r2max) continue;
                const float4 v = gw[k];
                const double gt = -((double)v.x * (dx * dx - dyk * dyk) + 2.0 * (double)v.y * dx * dyk) / r2;
                const double wr = (double)v.z * r2;
                double b[3];
#pragma unroll
                for (int l = 0; l < R; ++l) {
                    const int i = R == 2 && l == 1 ? 2 : l;
                    b[l] = wr * nrm[i] * exp(-r2 * inv2[i]);
                }
                direct_sums<R>(s, b, gt);
            }
        }
    }
    return !BLOCK && later;
}

// one (aperture, radii triple) by the block; returns whether a row was left out
template <bool BLOCK>
__device__ __forceinline__ bool direct_aperture(int64_t job, int limit, const int2* __restrict__ pos,
                                                const float4* __restrict__ gw, const int* __restrict__ start,
                                                const GridDesc* __restrict__ grid, double quantum, int n_ap,
                                                const double* __restrict__ centres, const double* __restrict__ theta,
                                                double rcut_factor, double* __restrict__ out)
{
    __shared__ double red[14][kDirThreads / 32];
    const int64_t t = job / n_ap;
    const int a = (int)(job % n_ap);
    double th[3], inv2[3], nrm[3];
    for (int l = 0; l < 3; ++l) th[l] = theta[3 * a + l];
    // equal radii first: the sums over distinct triplets are symmetric in the slots
    if (th[0] != th[1]) {
        if (th[0] == th[2]) {
            const double x = th[1];
            th[1] = th[2];
            th[2] = x;
        } else if (th[1] == th[2]) {
            const double x = th[0];
            th[0] = th[2];
            th[2] = x;
        }
    }
    for (int l = 0; l < 3; ++l) {
        inv2[l] = 1.0 / (2.0 * th[l] * th[l]);
        nrm[l] = 1.0 / (4.0 * M_PI * th[l] * th[l] * th[l] * th[l]);
    }
    const double rcut = rcut_factor * fmax(th[0], fmax(th[1], th[2]));
    // the largest r^2 whose square root is not above rcut: the same galaxies as sqrt(r2) > rcut leaves
    double r2max = rcut * rcut;
    for (int i = 0; i < 4 && sqrt(r2max) > rcut; ++i) r2max = __longlong_as_double(__double_as_longlong(r2max) - 1);
    for (int i = 0; i < 4 && r2max > 0.0; ++i) {
        const double up = __longlong_as_double(__double_as_longlong(r2max) + 1);
        if (!(sqrt(up) <= rcut)) break;
        r2max = up;
    }
    if (!(rcut >= 0.0)) r2max = rcut;  // NaN: no galaxy is left out; negative: all are
    double s[14];
#pragma unroll
    for (int v = 0; v < 14; ++v) s[v] = 0.0;
    const GridDesc g = *grid;
    const double cx = centres[2 * t], cy = centres[2 * t + 1];
    bool later;
    const bool e01 = th[0] == th[1], e12 = th[1] == th[2];
    if (e01 && e12) {
        later = direct_cells<1, BLOCK>(s, limit, pos, gw, start, g, quantum, cx, cy, rcut, r2max, inv2, nrm);
        s[1] = s[2] = s[0];
        s[4] = s[5] = s[3];
        s[8] = s[9] = s[7];
        s[11] = s[12] = s[10];
    } else if (e01) {
        later = direct_cells<2, BLOCK>(s, limit, pos, gw, start, g, quantum, cx, cy, rcut, r2max, inv2, nrm);
        s[1] = s[0];
        s[5] = s[4];
        s[8] = s[7];
        s[12] = s[11];
    } else {
        later = direct_cells<3, BLOCK>(s, limit, pos, gw, start, g, quantum, cx, cy, rcut, r2max, inv2, nrm);
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int v = 0; v < 14; ++v) {
        double x = s[v];
        for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
        if (lane == 0) red[v][warp] = x;
    }
    later = __syncthreads_or(later) != 0;
    if (threadIdx.x == 0) {
        double q[14];
        for (int v = 0; v < 14; ++v) {
            q[v] = 0.0;
            for (int k = 0; k < kDirThreads / 32; ++k) q[v] += red[v][k];
        }
        out[2 * job] = q[0] * q[1] * q[2] - q[3] * q[2] - q[4] * q[1] - q[5] * q[0] + 2.0 * q[6];
        out[2 * job + 1] = q[7] * q[8] * q[9] - q[10] * q[9] - q[11] * q[8] - q[12] * q[7] + 2.0 * q[13];
    }
    return later;
}

__global__ void __launch_bounds__(kDirThreads) map3_direct_cells_kernel(const int2* __restrict__ pos,
                                                                        const float4* __restrict__ gw,
                                                                        const int* __restrict__ start,
                                                                        const GridDesc* __restrict__ grid, double quantum,
                                                                        int limit, int n_ap,
                                                                        const double* __restrict__ centres,
                                                                        const double* __restrict__ theta,
                                                                        double rcut_factor, double* __restrict__ out,
                                                                        uint8_t* __restrict__ again)
{
    const int64_t job = blockIdx.x;
    const bool later = direct_aperture<false>(job, limit, pos, gw, start, grid, quantum, n_ap, centres, theta, rcut_factor, out);
    if (threadIdx.x == 0) again[job] = later;
}

__global__ void __launch_bounds__(kDirThreads) map3_direct_long_kernel(int64_t jobs, const int2* __restrict__ pos,
                                                                       const float4* __restrict__ gw,
                                                                       const int* __restrict__ start,
                                                                       const GridDesc* __restrict__ grid, double quantum,
                                                                       int limit, int n_ap,
                                                                       const double* __restrict__ centres,
                                                                       const double* __restrict__ theta,
                                                                       double rcut_factor, double* __restrict__ out,
                                                                       const uint8_t* __restrict__ again)
{
    for (int64_t job = blockIdx.x; job < jobs; job += gridDim.x) {
        if (!again[job]) continue;
        direct_aperture<true>(job, limit, pos, gw, start, grid, quantum, n_ap, centres, theta, rcut_factor, out);
        __syncthreads();  // the reduction's buffer
    }
}

cudaError_t launch_map3_direct_cells(int64_t n, const int2* pos, const float4* gw, const int* start, const GridDesc* grid,
                                     double quantum, int64_t n_cen, const double* centres, int n_ap, const double* theta,
                                     double rcut_factor, double* out, uint8_t* again, int n_sm, cudaStream_t st)
{
    // long: a row by a warp takes as long as the scan of an eighth of the catalog by the block; 128 steps of a
    // warp are not worth the second kernel
    const int limit = (int)std::min<int64_t>(4096, std::max<int64_t>(256, n / 8));
    const int64_t jobs = n_cen * n_ap;
    map3_direct_cells_kernel<<<(unsigned)jobs, kDirThreads, 0, st>>>(pos, gw, start, grid, quantum, limit, n_ap, centres, theta,
                                                                     rcut_factor, out, again);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    map3_direct_long_kernel<<<(unsigned)std::min<int64_t>(jobs, 2 * n_sm), kDirThreads, 0, st>>>(
        jobs, pos, gw, start, grid, quantum, limit, n_ap, centres, theta, rcut_factor, out, again);
    return cudaGetLastError();
}

cudaError_t launch_map3_direct(int64_t n, const int32_t* xq, const int32_t* yq, const float* g1, const float* g2,
                               const float* w, double quantum, int64_t n_cen, const double* centres, int n_ap,
                               const double* theta, double rcut_factor, double* out, cudaStream_t st)
{
    const int64_t jobs = n_cen * (int64_t)n_ap;
    if (jobs < 1) return cudaSuccess;
    if (jobs > 0x7fffffffLL) return cudaErrorInvalidValue;
    map3_direct_kernel<<<(unsigned)jobs, kDirThreads, 0, st>>>(n, xq, yq, g1, g2, w, quantum, n_ap, centres, theta,
                                                               rcut_factor, out);
    return cudaGetLastError();
}

}  // namespace mp3
