// Stage (a) for the narrow radial bins, those with few neighbours: the same sums as moments.cuh.
//
// The block-per-centre form spends some 9000 warp instructions per (centre, bin) on barriers, range
// set-up, half-empty batches and the reduction over lanes, whatever the bin holds. Here a warp works
// on a centre by itself and its lanes are the orders: lane l of either half keeps W_m, A_m and B_m of
// m = l, l + 16, ... The warp tests 32 candidates at a time, one per lane; once 32 members are found
// (or the bin ends) the lanes store the powers of their directions, and the members are added two at a
// time, one by each half, every lane stepping from z^l by z^16: about 16 warp instructions a member at
// n_max = 30, no barrier, one exchange between the halves at a bin's end. (All 32 lanes on one member took
// 27, as 34 and 61 orders fill two words of 32 badly and each power was a product first: 20 000 galaxies,
// 20 bins, n_max 30 4.69 -> 4.43 ms, 3 000 galaxies, 10 bins, n_max 10 0.233 -> 0.221.) The direct form's
// 14 a member plus its overhead are less from a few hundred members on. Bound by issue and the latency of
// the chains in small bins. The order of the sums is fixed.
#include <algorithm>

#include "moments_far.cuh"
#include "sector.cuh"

namespace mp3 {

namespace near {

constexpr int kQueue = 128;
static_assert(kMaxNmax <= 55, "launch() needs more orders a lane");

// warps of a block (the stored powers take 3.3 KB a warp in FP32) and blocks per SM the registers are
// sized for
template <typename T>
struct Block {
    static constexpr int kWarps = sizeof(T) == 8 ? 4 : 8, kThreads = kWarps * 32, kMin = sizeof(T) == 8 ? 4 : 3;
};

template <typename T>
struct alignas(16) Member {
    T a, b, w, pad;
};

__device__ __forceinline__ cx<float> direction(float dx, float dy, float)
{
    const float r2 = fmaf(dx, dx, dy * dy);
    float inv = rsqrtf(r2);
    inv = inv * (1.5f - 0.5f * r2 * inv * inv);
    return {dx * inv, dy * inv};
}
__device__ __forceinline__ cx<double> direction(float dx, float dy, double)
{
    const double x = dx, y = dy, inv = rsqrt(x * x + y * y);
    return {x * inv, y * inv};
}

__device__ __forceinline__ void cacc(cx<float>& s, float v, cx<float> c)
{
    const float2 r = __ffma2_rn(make_float2(v, v), make_float2(c.x, c.y), make_float2(s.x, s.y));
    s = cx<float>{r.x, r.y};
}
__device__ __forceinline__ void cacc(cx<double>& s, double v, cx<double> c)
{
    s.x = fma(v, c.x, s.x);
    s.y = fma(v, c.y, s.y);
}

// stored powers of a member: z^0..z^16; in FP64 with up to 32 orders all of them, as an FP64 instruction
// takes 16 cycles whatever the number of lanes that need it
template <typename T, int SW>
struct Powers {
    static constexpr bool kAll = sizeof(T) == 8 && SW <= 2;
    static constexpr int kPow = kAll ? 16 * SW + 1 : 17;
};

// the halves' sums of x[2 k] and x[2 k + 1], the even one to the lower half, the odd one to the upper
template <typename T, int S>
__device__ __forceinline__ cx<T> exchange(const cx<T> (&x)[S], int k, bool upper)
{
    const cx<T> even = x[2 * k], odd = 2 * k + 1 < S ? x[2 * k + 1 < S ? 2 * k + 1 : 0] : cx<T>{T(0), T(0)};
    const cx<T> keep = upper ? odd : even, send = upper ? even : odd;
    return {keep.x + __shfl_xor_sync(0xffffffffu, send.x, 16), keep.y + __shfl_xor_sync(0xffffffffu, send.y, 16)};
}

// SW, SAB: orders of W and of A, B a lane
template <typename T, int SW, int SAB>
__global__ void __launch_bounds__(Block<T>::kThreads, Block<T>::kMin) near_moments_kernel(const NearArgs<T> A)
{
    constexpr int kWarps = Block<T>::kWarps, kThreads = Block<T>::kThreads;
    constexpr unsigned FULL = 0xffffffffu;
    const MomentArgs<T>& m = A.m;
    __shared__ BinGeom bins[kMaxBins];
    constexpr bool kAll = Powers<T, SW>::kAll;
    constexpr int kPow = Powers<T, SW>::kPow;
    extern __shared__ __align__(16) unsigned char smem_raw[];  // powers [kWarps][32 kPow]
    __shared__ int queue[kWarps][kQueue], founds[kWarps][64];
    __shared__ Member<T> mem[kWarps][32];
    const int mtop = max(2 * A.m.n_max, A.m.n_max + 3);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, half = lane >> 4;
    const unsigned lt_mask = (1u << lane) - 1u;
    const int nz = m.nz, n_max = m.n_max;
    const size_t plane = (size_t)m.n_centres * nz * m.nbp;
    for (int b = threadIdx.x; b < m.nb; b += kThreads) {
        bins[b] = A.m.bins[b];
    }
    __syncthreads();
    int* qu = queue[warp];
    int* found = founds[warp];
    cx<T>* P = reinterpret_cast<cx<T>*>(smem_raw) + warp * 32 * kPow;
    Member<T>* V = mem[warp];
    SectorGeom g;
    g.hx = g.hy = 0.0f;
    g.S = (float)m.g.side;
    g.iS = 1.0f / g.S;
    g.ncx = m.g.ncx;
    g.ncy = m.g.ncy;
    unsigned long long my_pairs = 0;

    const long long nitems = (long long)m.n_centres * A.parts;
    for (long long item = blockIdx.x * kWarps + warp; item < nitems;) {
        const int c = (int)(item / A.parts), part = (int)(item - (long long)c * A.parts);
        const float2 pc = A.m.posf[m.centre_idx[c]];
        g.gx = pc.x;
        g.gy = pc.y;
        for (int z = 0; z < nz; ++z) {
            const int* row_start = m.cell_start + (size_t)z * m.g.ncells;
            for (int b = part; b < m.nb; b += A.parts) {
                const BinGeom bg = bins[b];
                g.Ri = bg.Ri;
                g.Ro = bg.Ro;
                cx<T> aw[SW], aa[SAB], ab[SAB];
#pragma unroll
                for (int s = 0; s < SW; ++s) aw[s] = cx<T>{T(0), T(0)};
#pragma unroll
                for (int s = 0; s < SAB; ++s) aa[s] = ab[s] = cx<T>{T(0), T(0)};
                // the first cnt members found: their powers by the lanes, then one member after the other
                auto add_members = [&](int cnt) {
                    if (lane < cnt + (cnt & 1)) {  // an odd last one is paired with itself at weight zero
                        const int i = found[min(lane, cnt - 1)];
                        const float2 p = A.m.posf[i];
                        const Pay<T> v = m.pay[i];
                        V[lane] = lane < cnt ? Member<T>{v.a, v.b, v.w, T(0)} : Member<T>{T(0), T(0), T(0), T(0)};
                        const cx<T> z1 = direction(p.x - pc.x, p.y - pc.y, T(0));
                        cx<T>* q = P + lane * kPow;
                        cx<T> lo[8];
                        lo[0] = cx<T>{T(1), T(0)};
                        lo[1] = z1;
#pragma unroll
                        for (int k = 2; k < 8; ++k) lo[k] = cmul(lo[k / 2], lo[k - k / 2]);
                        cx<T> hi = cmul(lo[4], lo[4]);
                        const cx<T> z8 = hi;
#pragma unroll
                        for (int k = 0; k < 8; ++k) q[k] = lo[k];
#pragma unroll
                        for (int k = 8; k < kPow; ++k) {
                            if (kAll && k > mtop) break;
                            if (k % 8 == 0 && k > 8) hi = cmul(hi, z8);
                            q[k] = k % 8 == 0 ? hi : cmul(hi, lo[k % 8]);
                        }
                    }
                    __syncwarp();
                    my_pairs += cnt;
                    const cx<T>* q = P + half * kPow;
#pragma unroll 2
                    for (int j = half; j < cnt + half; j += 2, q += 2 * kPow) {
                        const Member<T> v = V[j];
                        cx<T> zc = q[lane & 15];
#pragma unroll
                        for (int s = 0; s < SW; ++s) {
                            cacc(aw[s], v.w, zc);
                            if (s < SAB) {
                                cacc(aa[s], v.a, zc);
                                cacc(ab[s], v.b, zc);
                            }
                            if (s + 1 < SW) zc = kAll ? q[(lane & 15) + 16 * (s + 1)] : cmul(zc, q[16]);
                        }
                    }
                    __syncwarp();
                };
                int nm = 0;  // members found and not yet added
                const float ro = g.Ro + 8.0f;
                const float iy0 = fmaxf(floorf((g.gy - ro) * g.iS), 0.0f);
                const float iy1 = fminf(floorf((g.gy + ro) * g.iS), (float)(g.ncy - 1));
                for (float iy = iy0 + (float)lane; iy - (float)lane <= iy1; iy += 32.0f) {
                    int st0 = 0, n0 = 0, st1 = 0, n1 = 0;
                    if (iy <= iy1)
                        annulus_runs(g, iy, (iy + 0.5f) * g.S - g.gy, 0, g.ncx - 1, row_start, st0, n0, st1, n1);
                    while (true) {
                        // list the rows' candidates in row order
                        const int len = n0 + n1;
                        int incl = len;
#pragma unroll
                        for (int o = 1; o < 32; o <<= 1) {
                            const int y = __shfl_up_sync(FULL, incl, o);
                            if (lane >= o) incl += y;
                        }
                        const int total = __shfl_sync(FULL, incl, 31);
                        if (total == 0) break;
                        const int off = incl - len;
                        const int put = max(0, min(len, kQueue - off));
                        for (int j = 0; j < put; ++j) qu[off + j] = j < n0 ? st0 + j : st1 + (j - n0);
                        const int t0 = min(put, n0);
                        st0 += t0;
                        n0 -= t0;
                        st1 += put - t0;
                        n1 -= put - t0;
                        const int n = min(total, kQueue);
                        __syncwarp();
                        for (int t = lane; t < n + lane; t += 32) {
                            const int i = qu[min(t, n - 1)];
                            const float2 p = A.m.posf[i];
                            const float dx = p.x - pc.x, dy = p.y - pc.y;  // exact
                            const float d = fabsf(fmaf(dx, dx, dy * dy) - bg.mid);
                            bool in = d < bg.d_in;
                            if (!in && d < bg.d_out) {
                                const long long q2 = (long long)(int)dx * (int)dx + (long long)(int)dy * (int)dy;
                                in = q2 >= bg.e0 && q2 < bg.e1;
                            }
                            const unsigned mask = __ballot_sync(FULL, in && t < n);
                            if (in && t < n) found[nm + __popc(mask & lt_mask)] = i;
                            nm += __popc(mask);
                            __syncwarp();
                            if (nm >= 32) {
                                add_members(32);
                                if (lane < nm - 32) found[lane] = found[32 + lane];
                                nm -= 32;
                                __syncwarp();
                            }
                        }
                        if (total <= kQueue) break;
                    }
                }
                if (nm > 0) add_members(nm);
                const size_t row = ((size_t)c * nz + z) * m.nbp + b;
#pragma unroll
                for (int k = 0; k < (SW + 1) / 2; ++k) {
                    const int mm = lane + 32 * k;
                    const cx<T> wm = exchange(aw, k, half != 0);
                    if (mm <= 2 * n_max) m.W[(size_t)mm * plane + row] = wm;
                    if (2 * k < SAB) {
                        const int ka = 2 * k < SAB ? k : 0;
                        const cx<T> a = exchange(aa, ka, half != 0), bb = exchange(ab, ka, half != 0);
                        if (mm <= n_max - 1) m.G[(size_t)(mm + n_max + 3) * plane + row] = cx<T>{a.x - bb.y, a.y + bb.x};
                        if (mm >= 1 && mm <= n_max + 3)
                            m.G[(size_t)(n_max + 3 - mm) * plane + row] = cx<T>{a.x + bb.y, bb.x - a.y};
                    }
                }
            }
        }
        long long nx = 0;
        if (lane == 0) nx = (long long)atomicAdd(A.queue, 1ull) + (long long)gridDim.x * kWarps;
        item = __shfl_sync(FULL, nx, 0);
    }
    if (lane == 0 && my_pairs) atomicAdd(m.pairs, my_pairs);
}

template <typename T, int SW, int SAB>
static cudaError_t launch(NearArgs<T> a, int n_sm, cudaStream_t st)
{
    constexpr int kWarps = Block<T>::kWarps, kThreads = Block<T>::kThreads;
    const size_t smem = sizeof(cx<T>) * kWarps * 32 * Powers<T, SW>::kPow;
    int per_sm = 0;
    cudaError_t e = set_smem_attr(near_moments_kernel<T, SW, SAB>, smem);
    if (e != cudaSuccess) return e;
    e = occupancy(&per_sm, near_moments_kernel<T, SW, SAB>, kThreads, smem);
    if (e != cudaSuccess) return e;
    const int64_t slots = (int64_t)n_sm * std::max(per_sm, 1) * kWarps;
    if (a.m.n_centres < 1) return cudaSuccess;
    // few centres: the bins of a centre go to several warps (a chain of small bins is all latency)
    a.parts = (int)std::min<int64_t>(a.m.nb, std::max<int64_t>(1, 4 * slots / a.m.n_centres));
    const int64_t grid = (std::min<int64_t>((int64_t)a.m.n_centres * a.parts, slots) + kWarps - 1) / kWarps;
    near_moments_kernel<T, SW, SAB><<<(unsigned)grid, kThreads, smem, st>>>(a);
    return cudaGetLastError();
}

template <typename T>
static cudaError_t dispatch(const NearArgs<T>& a, int n_sm, cudaStream_t st)
{
    // orders 0 .. max(2 n_max, n_max + 3) of W and 0 .. n_max + 3 of A, B, 16 lanes
    const int sw = std::max(2 * a.m.n_max, a.m.n_max + 3) / 16 + 1, sab = (a.m.n_max + 3) / 16 + 1;
    if (sw == 1) return launch<T, 1, 1>(a, n_sm, st);
    if (sw == 2 && sab == 1) return launch<T, 2, 1>(a, n_sm, st);
    if (sw == 2) return launch<T, 2, 2>(a, n_sm, st);
    if (sw == 3) return launch<T, 3, 2>(a, n_sm, st);
    if (sw == 4) return launch<T, 4, 3>(a, n_sm, st);
    if (sw <= 6) return launch<T, 6, 4>(a, n_sm, st);
    return launch<T, 7, 4>(a, n_sm, st);  // kMaxNmax is 50
}

}  // namespace near

cudaError_t launch_moments_near(const NearArgs<float>& a, int n_sm, cudaStream_t st) { return near::dispatch(a, n_sm, st); }
cudaError_t launch_moments_near(const NearArgs<double>& a, int n_sm, cudaStream_t st) { return near::dispatch(a, n_sm, st); }

}  // namespace mp3
