// The moments of wide radial bins by angular sectors (moments_far.cu) and of narrow ones by a warp per
// centre (moments_near.cu).
#pragma once

#include <vector>

#include "common.cuh"

namespace mp3 {

// A radial bin for the FP32 distance test: with r^2 = fma(dx, dx, dy dy) (off by at most 2^-23 r^2)
// and d = |r^2 - mid|, d < d_in is inside, d >= d_out outside; in between the integers decide.
struct BinGeom {
    float Ri, Ro, mid, d_in, d_out, pad;
    long long e0, e1;
};
std::vector<BinGeom> bin_geometry(const std::vector<long long>& e2q);

// tables of a context (they depend on n_max only): offsets into one float array of all variants
constexpr int kFarPlans = 4;  // variants, widest bins first
// Their sectors, terms of W, terms of A and B. Widest: few terms, the centre group must subtend a small
// angle; last: the bins nearest to the group.
constexpr int kFarSectors[kFarPlans] = {64, 64, 32, 32}, kFarPW[kFarPlans] = {18, 20, 28, 32},
              kFarPAB[kFarPlans] = {14, 16, 20, 24};
struct FarTables {
    int off_ray = 0, off_sin = 0, off_axis = 0, off_rot = 0, off_coef = 0;
};
void far_tables(int n_max, FarTables (&t)[kFarPlans], std::vector<float>* v);

struct FarArgs {
    MomentArgs<float> m;   // bins, pointers and outputs as in the direct form
    const int32_t* order;  // rows of the centres in strip order: (strip, column, row)
    int none;              // index of an entry of posf and pay far from every galaxy, with zero payload
    int strip_rows;        // cell rows of a strip
    int max_cols;          // columns a group may span
    int parts;             // work items a group's (bin, z) pairs are split into
    const float* table;
    int off_ray, off_sin, off_axis, off_rot, off_coef;
    unsigned long long* queue;  // items claimed beyond the first gridDim.x (zero at launch)
    float* gvw;                 // adjoint: the gradient slots of AdjArgs (m.G, m.W: dL/dG, dL/dW)
};

cudaError_t launch_moments_far(const FarArgs& a, int plan, int n_sm, cudaStream_t st);

cudaError_t launch_moments_far_adjoint(const FarArgs& a, int plan, int n_sm, cudaStream_t st);

template <typename T>
struct NearArgs {
    MomentArgs<T> m;
    unsigned long long* queue;  // items claimed beyond the first gridDim.x * warps (zero at launch)
    int parts;                  // set by the launcher: work items the bins of a centre are split into
};
cudaError_t launch_moments_near(const NearArgs<float>& a, int n_sm, cudaStream_t st);
cudaError_t launch_moments_near(const NearArgs<double>& a, int n_sm, cudaStream_t st);

}  // namespace mp3
