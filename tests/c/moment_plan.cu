// Host check of moments_plan.cuh: for random calls, every bin of the sector form keeps its members within the
// angle its Chebyshev terms allow on the cells the grid really gets, the bins below it cross at most
// kMaxRows cell rows, and the ranges of bins fit together.
// usage: moment_plan seed calls; prints how many sector bins were checked.
#include <stdio.h>
#include <stdlib.h>

#include <random>
#include <vector>

#include "../../paper_2309_08601_gb300/csrc/moments_plan.cuh"

using namespace mp3;

int main(int argc, char** argv)
{
    if (argc < 3) return 2;
    std::mt19937 rng(atoi(argv[1]));
    auto uni = [&](double a, double b) { return a + (b - a) * (rng() / 4294967296.0); };
    auto logu = [&](double a, double b) { return exp(uni(log(a), log(b))); };
    long long checked = 0;
    for (int call = 0; call < atoi(argv[2]); ++call) {
        MomentsPlanInput in;
        in.n_max = rng() % (kMaxNmax + 1);
        in.nz = rng() % 3 ? 1 : 1 + rng() % kMaxNz;
        in.fp64 = rng() % 8 == 0;
        in.sectors = !in.fp64 && rng() % 8;
        in.occupancy = rng() % 2 ? 0 : 1 + rng() % 64;
        const double ex = floor(logu(1.0, 16777215.0)), ey = rng() % 3 ? ex : floor(logu(1.0, 16777215.0));
        in.extent = std::max(ex, ey) + 1.0;
        in.area = (ex + 1.0) * (ey + 1.0);
        in.n = (int64_t)logu(1.0, 2e7);
        in.nc = (int64_t)ceil(in.n * logu(1e-3, 1.0));
        in.carea = in.nc < in.n ? std::max(1.0, in.area * logu(1e-3, 1.0)) : in.area;
        const int nb = 1 + rng() % kMaxBins;
        const double hi = logu(10.0, 3e9), lo = hi * logu(1e-4, 0.99);
        std::vector<long long> e2(nb + 1);
        for (int b = 0; b <= nb; ++b) {
            const double t = lo * pow(hi / lo, (double)b / nb);
            e2[b] = (long long)ceil(t * t);
        }
        in.e2q = e2.data();
        in.b_lo = rng() % 4 ? 0 : rng() % nb;
        in.b_hi = rng() % 4 ? nb : in.b_lo + rng() % (nb - in.b_lo + 1);
        const MomentsPlan p = plan_moments(in);
        const FarPlan& f = p.far;
        if (!(in.b_lo <= p.b_near && p.b_near <= f.b_far && f.b_far <= in.b_hi)) return printf("ranges of bins\n"), 1;
        const double side = ceil(p.side);
        if (side < 1.0 || (ex / side) * (ey / side) * in.nz > 2.0 * (1 << 26) + ex + ey) return printf("too many cells\n"), 1;
        if (floor(in.extent / side) + 2.0 >= (1 << 22)) return printf("columns beyond near_int's range\n"), 1;
        if ((2.0 * sqrt((double)e2[f.b_far]) + 16.0) / side > kMaxRows - 4) return printf("more cell rows than listed\n"), 1;
        if (f.b_far == in.b_hi) continue;
        if (!in.sectors || f.b[0] != in.b_hi || f.b[kFarPlans] != f.b_far) return printf("ranges of variants\n"), 1;
        // a cell's half diagonal and the group's, as seen from the inner edge
        const double reach = side * (sqrt(0.5) + 0.5 * sqrt((double)f.rows * f.rows + (double)f.cols * f.cols));
        for (int v = 0; v < kFarPlans; ++v)
            for (int b = f.b[v + 1]; b < f.b[v]; ++b, ++checked)
                if (reach > sqrt((double)e2[b]) * sin(far_dmax(in.n_max, v) - M_PI / kFarSectors[v]))
                    return printf("n_max %d: variant %d takes a bin that is too near\n", in.n_max, v), 1;
    }
    printf("%lld\n", checked);
    return 0;
}
