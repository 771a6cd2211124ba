// Compile-time check of moments.cuh: every candidate a warp stages has an index that its list can hold.
#include "../../paper_2309_08601_gb300/csrc/moments.cuh"

using namespace mp3;

template <typename T, int NMAX>
constexpr bool holds()
{
    using PL = MomPlan<T, NMAX>;
    using Index = typename MomSmem<T, PL::P, PL::SCR>::Index;
    return (Index)(PL::SCR - 1) == PL::SCR - 1;
}
static_assert(holds<float, 10>() && holds<float, 30>() && holds<float, 50>(), "FP32");
static_assert(holds<double, 10>() && holds<double, 50>(), "FP64");
