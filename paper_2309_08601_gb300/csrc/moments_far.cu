// Stage (a) for the wide radial bins: the same sums as moments.cuh, G_m = sum_k w_k gamma_k e^{i m phi}
// and W_m = sum_k w_k e^{i m phi} (paper Sec. 3.1), by angular sectors.
//
// The direct form steps every pair through all orders (about 400 FMAs a pair at n_max = 30). Here the
// circle is cut into S sectors with axes phi_s = 2 pi (s + 1/2) / S, and with delta = phi - phi_s
//   e^{i m phi} = e^{i m phi_s} sum_p i^{p mod 2} c_{m,p} T_p(u),  u = sin(delta) / sin(delta_max),
// T_p the Chebyshev polynomials and c_{m,p} the (real) expansion coefficients of cos and sin of
// m asin(sin(delta_max) u). A pair then only adds w T_p, w gamma_1 T_p (p < PAB) and w gamma_2 T_p to
// its sector's sums M_{s,p} (30 packed FMAs in the variant for the widest bins, 54 for the nearest), and per (centre,
// bin) a real FFT over the sectors and a short sum over p give every order:
//   W_m = e^{i pi m / S} sum_p i^{p mod 2} c_{m,p} F_{m,p},  F_{m,p} = sum_s M_{s,p} e^{2 pi i m s / S}.
// delta_max follows from n_max, PW and PAB so that the dropped terms stay below 3e-8 (far_dmax), so
// the result differs from the direct form's by FP32 rounding only.
//
// A block of eight warps works on a group of up to eight neighbouring centres; a warp takes a sector
// at a time, lane = (centre, one of four candidate streams): every candidate loaded serves eight
// centres, and the cells of a sector come from the grid (sector.cuh), so nothing is sorted per
// centre and the order of the sums is fixed (reproducible run to run).
//
// Measured with the narrow bins in moments_near.cu, moments of the whole call: 200 000 galaxies, 20
// bins to 120', n_max 30: 314 -> 84 ms; 10 000 centres of 400 000 galaxies, 30 bins to 240',
// n_max 40: 98.5 -> 19 ms. The candidate loop is 80 % of it, bound by issue (53 to 63 % of the slots with 16
// warps an SM) and latency; FMA pipe 47 to 58 %, ALU pipe 25 to 44 %; the next candidates' loads come from L2.
#include <math.h>

#include <algorithm>
#include <vector>

#include "moments_plan.cuh"
#include "sector.cuh"

namespace mp3 {

namespace far {

constexpr int kWarps = 8, kThreads = kWarps * 32;
constexpr int kC = 8;       // centres of a group
constexpr int kSub = 4;     // candidate streams of a warp (kC * kSub = 32 lanes)
constexpr int kQueue = 128; // candidates listed at a time per warp
constexpr int kAhead = 6;   // filler entries of a lane behind the list

// S sectors, PW terms of W, PAB terms of A and B
template <int S_, int PW_, int PAB_>
struct Plan {
    static constexpr int S = S_, PW = PW_, PAB = PAB_, PT = PW + 2 * PAB;
    static constexpr int KS = PT * kC + ((PT * kC) % 32 == 0 ? 8 : 0);  // floats per sector (bank spread)
};
template <int V>
using Variant = Plan<kFarSectors[V], kFarPW[V], kFarPAB[V]>;

// cos(2 pi k / 64); folds to a literal once the loops are unrolled
__device__ __forceinline__ float cos64(int k)
{
    const float t[17] = {1.000000000f, 0.995184727f, 0.980785280f, 0.956940336f, 0.923879533f, 0.881921264f,
                         0.831469612f, 0.773010453f, 0.707106781f, 0.634393284f, 0.555570233f, 0.471396737f,
                         0.382683432f, 0.290284677f, 0.195090322f, 0.098017140f, 0.000000000f};
    k &= 63;
    if (k > 32) k = 64 - k;
    return k <= 16 ? t[k] : -t[32 - k];
}
__device__ __forceinline__ float sin64(int k) { return cos64(k + 48); }

__device__ __forceinline__ constexpr int bit_reverse(int i, int bits)
{
    int r = 0;
    for (int b = 0; b < bits; ++b) r |= ((i >> b) & 1) << (bits - 1 - b);
    return r;
}

// complex FFT of N = 2^BITS points in registers, sum_j z_j e^{SIGN 2 pi i j k / N}; input in bit-reversed
// order
template <int BITS, int SIGN>
__device__ __forceinline__ void complex_fft(float (&re)[1 << BITS], float (&im)[1 << BITS])
{
    constexpr int N = 1 << BITS;
#pragma unroll
    for (int st = 0; st < BITS; ++st) {
        const int h = 1 << st;
#pragma unroll
        for (int b = 0; b < N / 2; ++b) {
            const int j = b & (h - 1), i0 = ((b >> st) << (st + 1)) + j, i1 = i0 + h;
            const int k = j * (32 >> st);  // twiddle e^{2 pi i j / (2 h)} as a 64th root
            const float c = cos64(k), s = SIGN * sin64(k);
            float tr, ti;
            if (k == 0) {
                tr = re[i1];
                ti = im[i1];
            } else if (k == 16) {
                tr = -SIGN * im[i1];
                ti = SIGN * re[i1];
            } else {
                tr = re[i1] * c - im[i1] * s;
                ti = re[i1] * s + im[i1] * c;
            }
            re[i1] = re[i0] - tr;
            im[i1] = im[i0] - ti;
            re[i0] += tr;
            im[i0] += ti;
        }
    }
}

// F_k = sum_s x_s e^{+2 pi i k s / S} of a real series, in registers: Re F_k at x[k] (k <= S/2),
// Im F_k at x[S - k] (0 < k < S/2). A complex FFT of the even and odd samples as real and imaginary
// parts, then the usual separation.
template <int S>
__device__ __forceinline__ void real_fft(float (&x)[S])
{
    constexpr int N = S / 2;
    constexpr int BITS = S == 64 ? 5 : S == 32 ? 4 : 3;
    float re[N], im[N];
#pragma unroll
    for (int j = 0; j < N; ++j) {
        re[j] = x[2 * bit_reverse(j, BITS)];
        im[j] = x[2 * bit_reverse(j, BITS) + 1];
    }
    complex_fft<BITS, 1>(re, im);
    x[0] = re[0] + im[0];
    x[N] = re[0] - im[0];
#pragma unroll
    for (int k = 1; k <= N / 2; ++k) {
        // E = (Z_k + Z*_{N-k}) / 2, O = (Z_k - Z*_{N-k}) / (2 i), F_k = E + w O, F_{N-k} = (E - w O)*
        const float er = 0.5f * (re[k] + re[N - k]), ei = 0.5f * (im[k] - im[N - k]);
        const float orr = 0.5f * (im[k] + im[N - k]), oi = -0.5f * (re[k] - re[N - k]);
        const float c = cos64(k * (64 / S)), s = sin64(k * (64 / S));
        const float wr = orr * c - oi * s, wi = orr * s + oi * c;
        x[k] = er + wr;
        x[S - k] = ei + wi;
        if (k < N / 2) {
            x[N - k] = er - wr;
            x[S - (N - k)] = wi - ei;
        }
    }
}

// the transpose of real_fft: from r_k = x[k] (k <= S/2) and i_k = x[S - k] (0 < k < S/2) to
// x_s = sum_k r_k cos(2 pi k s / S) + i_k sin(2 pi k s / S)
template <int S>
__device__ __forceinline__ void real_fft_adjoint(float (&x)[S])
{
    constexpr int N = S / 2;
    constexpr int BITS = S == 64 ? 5 : S == 32 ? 4 : 3;
    // the Hermitian spectrum Y_k = (r_k + i i_k) / 2 folded to N points whose transform has x_{2j} as real
    // and x_{2j+1} as imaginary part: C_k = Y_k + Y*_{N-k} + i e^{-2 pi i k / S} (Y_k - Y*_{N-k})
    float cr[N], ci[N], re[N], im[N];
    cr[0] = x[0] + x[N];
    ci[0] = x[0] - x[N];
#pragma unroll
    for (int k = 1; k <= N / 2; ++k) {
        const float ar = 0.5f * x[k], ai = 0.5f * x[S - k];
        const float br = 0.5f * x[N - k], bi = -0.5f * x[S - (N - k)];
        const float sr = ar + br, si = ai + bi, dr = ar - br, di = ai - bi;
        const float c = cos64(k * (64 / S)), s = sin64(k * (64 / S));
        const float tr = dr * s - di * c, ti = dr * c + di * s;  // i e^{-i theta k} d
        cr[k] = sr + tr;
        ci[k] = si + ti;
        if (k < N / 2) {
            cr[N - k] = sr - tr;
            ci[N - k] = ti - si;
        }
    }
#pragma unroll
    for (int j = 0; j < N; ++j) {
        re[j] = cr[bit_reverse(j, BITS)];
        im[j] = ci[bit_reverse(j, BITS)];
    }
    complex_fft<BITS, -1>(re, im);
#pragma unroll
    for (int j = 0; j < N; ++j) {
        x[2 * j] = re[j];
        x[2 * j + 1] = im[j];
    }
}

// one warp's sums of a sector: pairs (p, p + 1) of Chebyshev terms in packed FP32 lanes
template <int PW, int PAB>
struct Sums {
    float2 w[PW / 2], a[PAB / 2], b[PAB / 2];

    __device__ __forceinline__ void reset()
    {
#pragma unroll
        for (int j = 0; j < PW / 2; ++j) w[j] = make_float2(0.f, 0.f);
#pragma unroll
        for (int j = 0; j < PAB / 2; ++j) a[j] = b[j] = make_float2(0.f, 0.f);
    }

    // v_j = s_j (T_{2j}, T_{2j+1}), s_j = +, +, -, -, ...: T_{p+2} = 2 T_2 T_p - T_{p-2} then needs no
    // negated addend (v_{j+1} = +-2 T_2 v_j + v_{j-1}); value() applies the signs
    __device__ __forceinline__ void add(float av, float bv, float wv, float u)
    {
        const float2 a2 = make_float2(av, av), b2 = make_float2(bv, bv), w2 = make_float2(wv, wv);
        const float t2 = fmaf(2.f * u, u, -1.f), k = 2.f * t2;
        float2 v0 = make_float2(1.f, u), v1 = make_float2(t2, fmaf(k, u, -u));
        const float2 kp = make_float2(k, k), km = make_float2(-k, -k);
#pragma unroll
        for (int j = 0; j < PW / 2; ++j) {
            if (j < PAB / 2) {
                a[j] = __ffma2_rn(a2, v0, a[j]);
                b[j] = __ffma2_rn(b2, v0, b[j]);
            }
            w[j] = __ffma2_rn(w2, v0, w[j]);
            if (j + 1 < PW / 2) {
                const float2 v2 = __ffma2_rn((j & 1) ? kp : km, v1, v0);
                v0 = v1;
                v1 = v2;
            }
        }
    }

    // flat index: W terms, A terms, B terms
    __device__ __forceinline__ float value(int i) const
    {
        const float2 v = i < PW ? w[i / 2] : i < PW + PAB ? a[(i - PW) / 2] : b[(i - PW - PAB) / 2];
        const int p = i < PW ? i : i < PW + PAB ? i - PW : i - PW - PAB;
        const float x = (p & 1) ? v.y : v.x;
        return ((p / 2) & 2) ? -x : x;
    }
};

// the adjoint of Sums: dL/d(sum) of a sector as the coefficients of Chebyshev series in u, whose values at
// a member are dL/d(w gamma_1), dL/d(w gamma_2) and dL/dw (signs as in Sums)
template <int PW, int PAB>
struct Series {
    float2 w[PW / 2], a[PAB / 2], b[PAB / 2];

    __device__ __forceinline__ void load(const float* m, bool on)
    {
        auto get = [&](int base, int j) {
            const float s = (j & 2) ? -1.f : 1.f;
            return on ? make_float2(s * m[(base + 2 * j) * kC], s * m[(base + 2 * j + 1) * kC]) : make_float2(0.f, 0.f);
        };
#pragma unroll
        for (int j = 0; j < PW / 2; ++j) w[j] = get(0, j);
#pragma unroll
        for (int j = 0; j < PAB / 2; ++j) {
            a[j] = get(PW, j);
            b[j] = get(PW + PAB, j);
        }
    }

    __device__ __forceinline__ void eval(float u, float& av, float& bv, float& wv) const
    {
        const float t2 = fmaf(2.f * u, u, -1.f), k = 2.f * t2;
        float2 v0 = make_float2(1.f, u), v1 = make_float2(t2, fmaf(k, u, -u));
        const float2 kp = make_float2(k, k), km = make_float2(-k, -k);
        float2 sa = make_float2(0.f, 0.f), sb = sa, sw = sa;
#pragma unroll
        for (int j = 0; j < PW / 2; ++j) {
            if (j < PAB / 2) {
                sa = __ffma2_rn(a[j], v0, sa);
                sb = __ffma2_rn(b[j], v0, sb);
            }
            sw = __ffma2_rn(w[j], v0, sw);
            if (j + 1 < PW / 2) {
                const float2 v2 = __ffma2_rn((j & 1) ? kp : km, v1, v0);
                v0 = v1;
                v1 = v2;
            }
        }
        av = sa.x + sa.y;
        bv = sb.x + sb.y;
        wv = sw.x + sw.y;
    }
};

// p[i] by a 32-bit byte offset (the caller keeps the arrays below 4 GB): the 64-bit multiply-add of
// the usual address runs on the FP64 pipe
template <typename U>
__device__ __forceinline__ U at32(const U* p, int i)
{
    return *reinterpret_cast<const U*>(reinterpret_cast<const char*>(p) + (uint32_t)i * (uint32_t)sizeof(U));
}

__device__ __forceinline__ float rsqrt_approx(float x)
{
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// the candidates of a sector in batches of up to kQueue, listed in row order: batch(n) is called by the
// whole warp with their indexes in queue[0 .. n), followed by kAhead kSub times `none`, a galaxy far from
// everything (so the candidate loop needs no test for its end)
template <typename F>
__device__ __forceinline__ void sector_batches(const SectorGeom& g, bool upper, bool first, bool last, float ct0, float ct1,
                                               float sn0, float sn1, const int* __restrict__ row_start, int none,
                                               int* queue, int lane, F&& batch)
{
    constexpr unsigned FULL = 0xffffffffu;
    float iy0, iy1;
    sector_rows(g, upper, sn0, sn1, iy0, iy1);
    for (float iy = iy0 + (float)lane; iy - (float)lane <= iy1; iy += 32.0f) {
        int st0 = 0, n0 = 0, st1 = 0, n1 = 0;
        if (iy <= iy1) sector_runs(g, upper, first, last, ct0, ct1, iy, row_start, st0, n0, st1, n1);
        while (true) {
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
            for (int j = 0; j < put; ++j) queue[off + j] = j < n0 ? st0 + j : st1 + (j - n0);
            const int t0 = min(put, n0);
            st0 += t0;
            n0 -= t0;
            st1 += put - t0;
            n1 -= put - t0;
            const int n = min(total, kQueue);
            if (lane < kAhead * kSub) queue[n + lane] = none;
            __syncwarp();
            batch(n);
            __syncwarp();
            if (total <= kQueue) break;
        }
    }
}

// ADJ: the transposed chain. m.G and m.W hold dL/dG and dL/dW; the transposes of the order sums and of
// the FFT give dL/dM_{s,p}, and every member of a sector gets the value of the Chebyshev series with these
// coefficients, summed over the group's centres before one atomic addition per component to A.gvw
// (the block-per-centre form evaluates the 2 n_max + 3 and 2 n_max + 1 orders per pair, about 500 FMAs, and adds
// every pair atomically).
template <class PL, bool ADJ>
__global__ void __launch_bounds__(kThreads, 2) far_moments_kernel(const FarArgs A)
{
    constexpr int S = PL::S, PW = PL::PW, PAB = PL::PAB, PT = PL::PT, KS = PL::KS;
    constexpr unsigned FULL = 0xffffffffu;
    extern __shared__ __align__(16) float M[];  // [S][KS]: sums of (sector, term, centre), then their FFT
    __shared__ int queue[kWarps][kQueue + kAhead * kSub];
    __shared__ float2 s_pos[kC];
    __shared__ int s_row[kC], s_cell[kC];
    __shared__ int s_next, s_item;

    const MomentArgs<float>& m = A.m;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int ce = lane & (kC - 1), sub = lane / kC;  // this lane's centre and candidate stream
    const int nz = m.nz, n_max = m.n_max;
    const size_t plane = (size_t)m.n_centres * nz * m.nbp;
    const int ngroups = (m.n_centres + kC - 1) / kC;
    const int nitems = ngroups * A.parts;
    const float4* axis = reinterpret_cast<const float4*>(A.table + A.off_axis);
    const float* ray = A.table + A.off_ray;
    const float2* rot = reinterpret_cast<const float2*>(A.table + A.off_rot);
    const float* coef = A.table + A.off_coef;
    unsigned long long my_pairs = 0;

    for (int item = blockIdx.x; item < nitems;) {
        const int group = item / A.parts, part = item % A.parts;
        if (tid < kC) {
            const int i = group * kC + tid;
            int row = -1, cell = 0;
            float2 p = make_float2(0.f, 0.f);
            if (i < m.n_centres) {
                row = A.order[i];
                p = m.posf[m.centre_idx[row]];
                cell = (int)p.y / (m.g.side * A.strip_rows) * m.g.ncx + (int)p.x / m.g.side;
            }
            s_row[tid] = row;
            s_pos[tid] = p;
            s_cell[tid] = cell;
        }
        __syncthreads();
        unsigned left = 0;  // centres not yet done
        for (int i = 0; i < kC; ++i) left |= (s_row[i] >= 0 ? 1u : 0u) << i;
        while (left) {
            // a compact subset: the first centre left and those of its strip within max_cols columns
            const int f = __ffs(left) - 1, fc = s_cell[f];
            unsigned act = 0;
            float x0 = 3e38f, x1 = -3e38f, y0 = 3e38f, y1 = -3e38f;
            for (int i = 0; i < kC; ++i) {
                const int d = s_cell[i] - fc;
                if (!((left >> i) & 1u) || d < 0 || d >= A.max_cols || fc / m.g.ncx != s_cell[i] / m.g.ncx) continue;
                act |= 1u << i;
                x0 = fminf(x0, s_pos[i].x);
                x1 = fmaxf(x1, s_pos[i].x);
                y0 = fminf(y0, s_pos[i].y);
                y1 = fmaxf(y1, s_pos[i].y);
            }
            left &= ~act;
            SectorGeom g;
            g.gx = 0.5f * (x0 + x1);
            g.gy = 0.5f * (y0 + y1);
            g.hx = 0.5f * (x1 - x0) + 1.0f;
            g.hy = 0.5f * (y1 - y0) + 1.0f;
            g.S = (float)m.g.side;
            g.iS = 1.0f / g.S;
            g.ncx = m.g.ncx;
            g.ncy = m.g.ncy;
            const bool mine = (act >> ce) & 1u;
            // lanes without a centre repeat the first one's sums (not counted, not written)
            const float2 pc = s_pos[mine ? ce : f];

            for (int zb = part; zb < nz * m.nb; zb += A.parts) {
                // widest bins first, so that the last items of the queue are short
                const int b = m.nb - 1 - zb / nz, z = zb % nz;
                // from memory, not from the integer edges: 64-bit conversions run on the FP64 pipe, and
                // the compiler would repeat them in the candidate loop
                const BinGeom* bg = m.bins + b;
                const float mid = bg->mid, d_in = bg->d_in, d_out = bg->d_out;
                g.Ri = bg->Ri;
                g.Ro = bg->Ro;
                const int* row_start = m.cell_start + (size_t)z * m.g.ncells;
                if (tid == 0) s_next = kWarps;
                __syncthreads();

                if constexpr (ADJ) {
                    // ---- transposed order sums: thread (centre, k) adds the orders m = +-k mod S
                    const int c8 = tid & (kC - 1);
                    const size_t at = ((size_t)s_row[c8] * nz + z) * m.nbp + b;
                    const int mtop = max(2 * n_max, n_max + 3);
                    const float on = (act >> c8) & 1u ? 1.f : 0.f;
                    for (int k = tid / kC; k <= S / 2; k += kThreads / kC) {
                        float* Fr = M + k * KS + c8;
                        float* Fi = M + ((S - k) & (S - 1)) * KS + c8;
                        const bool edge = k == 0 || k == S / 2;
                        for (int p = 0; p < PT; ++p) {
                            Fr[p * kC] = 0.f;
                            if (!edge) Fi[p * kC] = 0.f;
                        }
                        for (int j = 0; j * S - k <= mtop; ++j)
                            for (int h = edge ? 1 : 0; h < 2; ++h) {
                                const int mm = h ? j * S + k : j * S - k;
                                if (mm < 0 || mm > mtop || on == 0.f) continue;
                                const float fi = edge ? 0.f : h ? 1.f : -1.f;
                                const float* cm = coef + mm * PW;
                                const float2 ro = rot[mm];
                                auto order = [&](int base, int P, cx<float> g) {
                                    const float vr = g.x * ro.x + g.y * ro.y, vi = g.y * ro.x - g.x * ro.y;
#pragma unroll 4
                                    for (int p = 0; p < P; p += 2) {
                                        const float ca = cm[p], cb = cm[p + 1];
                                        Fr[(base + p) * kC] += ca * vr;
                                        Fr[(base + p + 1) * kC] += cb * vi;
                                        if (!edge) {
                                            Fi[(base + p) * kC] += fi * ca * vi;
                                            Fi[(base + p + 1) * kC] -= fi * cb * vr;
                                        }
                                    }
                                };
                                if (mm <= 2 * n_max) order(0, PW, m.W[(size_t)mm * plane + at]);
                                if (mm <= n_max + 3) {
                                    cx<float> ga{0.f, 0.f}, gb{0.f, 0.f};
                                    if (mm <= n_max - 1) {
                                        const cx<float> y = m.G[(size_t)(mm + n_max + 3) * plane + at];
                                        ga = y;
                                        gb = cx<float>{y.y, -y.x};
                                    }
                                    if (mm >= 1) {
                                        const cx<float> y = m.G[(size_t)(n_max + 3 - mm) * plane + at];
                                        ga = cx<float>{ga.x + y.x, ga.y - y.y};
                                        gb = cx<float>{gb.x + y.y, gb.y + y.x};
                                    }
                                    order(PW, PAB, ga);
                                    order(PW + PAB, PAB, gb);
                                }
                            }
                    }
                    __syncthreads();
                    for (int q = tid; q < PT * kC; q += kThreads) {
                        float x[S];
#pragma unroll
                        for (int s = 0; s < S; ++s) x[s] = M[s * KS + q];
                        real_fft_adjoint<S>(x);
#pragma unroll
                        for (int s = 0; s < S; ++s) M[s * KS + q] = x[s];
                    }
                    __syncthreads();
                }

                // ---- the sectors: sums of their members, or the members' gradients
                for (int s = warp; s < S;) {
                    const bool upper = s < S / 2;
                    const int sp = upper ? s : s - S / 2;
                    const float4 ax = axis[s];  // (cos, sin) / sin(delta_max), angle offset of the rounded axis
                    const float sn0 = A.table[A.off_sin + 2 * sp], sn1 = A.table[A.off_sin + 2 * sp + 1];
                    int* qu = queue[warp];
                    if constexpr (ADJ) {
                        Series<PW, PAB> ser;
                        ser.load(M + s * KS + ce, mine);
                        auto add = [&](int i, bool in, float u) {
                            float a, b, w;
                            ser.eval(u, a, b, w);
                            a = in ? a : 0.f;
                            b = in ? b : 0.f;
                            w = in ? w : 0.f;
                            // over the eight centres (lane bits 0..2), ending with a, b or w in a lane
                            const bool u2 = (lane & 4) != 0, u1 = (lane & 2) != 0;
                            const float r0 = __shfl_xor_sync(FULL, u2 ? a : w, 4), r1 = __shfl_xor_sync(FULL, u2 ? b : 0.f, 4);
                            const float k0 = (u2 ? w : a) + r0, k1 = (u2 ? 0.f : b) + r1;
                            float v = (u1 ? k1 : k0) + __shfl_xor_sync(FULL, u1 ? k0 : k1, 2);
                            v += __shfl_xor_sync(FULL, v, 1);
                            if (!(lane & 1) && v != 0.f) atomicAdd(A.gvw + 4 * (size_t)i + (u2 ? 2 : u1 ? 1 : 0), v);
                        };
                        sector_batches(g, upper, sp == 0, sp == S / 2 - 1, ray[sp], ray[sp + 1], sn0, sn1, row_start, A.none, qu, lane,
                                       [&](int n) {
                            int odd = 0;
                            auto one = [&](int i, float2 p) {
                                const float dx = p.x - pc.x, dy = p.y - pc.y;  // exact
                                const float r2 = fmaf(dx, dx, dy * dy), d = fabsf(r2 - mid);
                                const bool in = d < d_in;
                                odd += d < d_out && !in ? 1 : 0;
                                add(i, in && mine, fmaf(fmaf(dy, ax.x, -dx * ax.y), rsqrt_approx(r2), ax.z));
                            };
                            const int* q = qu + sub;
                            int i0, i1, i2, i3;
                            float2 p0, p1, p2, p3;
                            auto fetch = [&](int at, int& i, float2& p) {
                                i = q[at * kSub];
                                p = at32(m.posf, i);
                            };
                            fetch(0, i0, p0);
                            fetch(1, i1, p1);
                            fetch(2, i2, p2);
                            fetch(3, i3, p3);
                            for (int rest = n; ; q += 4 * kSub) {
                                one(i0, p0);
                                one(i1, p1);
                                if ((rest -= 2 * kSub) <= 0) break;
                                fetch(4, i0, p0);
                                fetch(5, i1, p1);
                                one(i2, p2);
                                one(i3, p3);
                                if ((rest -= 2 * kSub) <= 0) break;
                                fetch(6, i2, p2);
                                fetch(7, i3, p3);
                            }
                            if (__any_sync(FULL, odd))  // rare: the candidates near an edge, by the integers
                                for (int t = sub; t < n + sub; t += kSub) {
                                    const int i = qu[min(t, n - 1)];
                                    const float2 p = at32(m.posf, i);
                                    const float dx = p.x - pc.x, dy = p.y - pc.y;
                                    const float r2 = fmaf(dx, dx, dy * dy), d = fabsf(r2 - mid);
                                    const long long q2 = (long long)(int)dx * (int)dx + (long long)(int)dy * (int)dy;
                                    const bool in = d < d_out && !(d < d_in) && t < n && q2 >= bg->e0 && q2 < bg->e1;
                                    add(i, in && mine, fmaf(fmaf(dy, ax.x, -dx * ax.y), rsqrt_approx(r2), ax.z));
                                }
                        });
                    } else {
                        Sums<PW, PAB> sum;
                        sum.reset();
                        int count = 0, maybe = 0;
                        sector_batches(g, upper, sp == 0, sp == S / 2 - 1, ray[sp], ray[sp + 1], sn0, sn1, row_start, A.none, qu, lane,
                                       [&](int n) {
                            // candidates sub, sub + 4, ...: two to four loads ahead
                            auto one = [&](float2 p, const Pay<float>& v) {
                                const float dx = p.x - pc.x, dy = p.y - pc.y;  // exact
                                const float r2 = fmaf(dx, dx, dy * dy), d = fabsf(r2 - mid);
                                const bool in = d < d_in;
                                count += in ? 1 : 0;
                                maybe += d < d_out ? 1 : 0;
                                const float u = fmaf(fmaf(dy, ax.x, -dx * ax.y), rsqrt_approx(r2), ax.z);
                                sum.add(in ? v.a : 0.f, in ? v.b : 0.f, in ? v.w : 0.f, u);
                            };
                            // two at a time in one stretch of code, so that the direction of one is
                            // formed while the other is added
                            const int* q = qu + sub;
                            float2 p0, p1, p2, p3;
                            Pay<float> v0, v1, v2, v3;
                            auto fetch = [&](int at, float2& p, Pay<float>& v) {
                                const int i = q[at * kSub];
                                p = at32(m.posf, i);
                                v = at32(m.pay, i);
                            };
                            fetch(0, p0, v0);
                            fetch(1, p1, v1);
                            fetch(2, p2, v2);
                            fetch(3, p3, v3);
                            for (int rest = n; ; q += 4 * kSub) {
                                one(p0, v0);
                                one(p1, v1);
                                if ((rest -= 2 * kSub) <= 0) break;
                                fetch(4, p0, v0);
                                fetch(5, p1, v1);
                                one(p2, v2);
                                one(p3, v3);
                                if ((rest -= 2 * kSub) <= 0) break;
                                fetch(6, p2, v2);
                                fetch(7, p3, v3);
                            }
                            if (__any_sync(FULL, maybe != count)) {
                                // rare: the candidates near an edge, by the integers
                                for (int t = sub; t < n; t += kSub) {
                                    const float2 p = at32(m.posf, qu[t]);
                                    const Pay<float> v = at32(m.pay, qu[t]);
                                    const float dx = p.x - pc.x, dy = p.y - pc.y;
                                    const float r2 = fmaf(dx, dx, dy * dy), d = fabsf(r2 - mid);
                                    if (!(d < d_out) || d < d_in) continue;
                                    const long long q2 = (long long)(int)dx * (int)dx + (long long)(int)dy * (int)dy;
                                    if (q2 < bg->e0 || q2 >= bg->e1) continue;
                                    count += 1;
                                    sum.add(v.a, v.b, v.w, fmaf(fmaf(dy, ax.x, -dx * ax.y), rsqrt_approx(r2), ax.z));
                                }
                                maybe = count;
                            }
                        });
                        if (mine) my_pairs += (unsigned long long)count;
                        // reduce over the four streams, each keeping a quarter of the terms
                        constexpr int Q = (PT + 3) / 4;
                        float h[2 * Q];
#pragma unroll
                        for (int i = 0; i < 2 * Q; ++i) {
                            const float lo = sum.value(i), hi = i + 2 * Q < PT ? sum.value(i + 2 * Q) : 0.f;
                            const bool up = (sub & 2) != 0;
                            h[i] = (up ? hi : lo) + __shfl_xor_sync(FULL, up ? lo : hi, 2 * kC);
                        }
                        float* out = M + s * KS + ce;
#pragma unroll
                        for (int i = 0; i < Q; ++i) {
                            const bool up = (sub & 1) != 0;
                            const float v = (up ? h[i + Q] : h[i]) + __shfl_xor_sync(FULL, up ? h[i] : h[i + Q], kC);
                            const int p = (sub >> 1) * 2 * Q + (sub & 1) * Q + i;
                            if (p < PT) out[p * kC] = v;
                        }
                    }
                    int nx = 0;
                    if (lane == 0) nx = atomicAdd(&s_next, 1);
                    s = __shfl_sync(FULL, nx, 0);
                }
                __syncthreads();
                if constexpr (!ADJ) {
                    // ---- FFT over the sectors of every (term, centre)
                    for (int q = tid; q < PT * kC; q += kThreads) {
                        float x[S];
    #pragma unroll
                        for (int s = 0; s < S; ++s) x[s] = M[s * KS + q];
                        real_fft<S>(x);
    #pragma unroll
                        for (int s = 0; s < S; ++s) M[s * KS + q] = x[s];
                    }
                    __syncthreads();

                    // ---- the orders: thread (centre, m)
                    const int c8 = tid & (kC - 1);
                    if ((act >> c8) & 1u) {
                        const size_t at = ((size_t)s_row[c8] * nz + z) * m.nbp + b;
                        const int mtop = max(2 * n_max, n_max + 3);
                        for (int mm = tid / kC; mm <= mtop; mm += kThreads / kC) {
                            int k = mm & (S - 1);
                            const bool cj = k > S / 2;
                            if (cj) k = S - k;
                            const float* Fr = M + k * KS + c8;
                            const float* Fi = M + ((S - k) & (S - 1)) * KS + c8;
                            const float fi = (k == 0 || k == S / 2) ? 0.f : (cj ? -1.f : 1.f);
                            const float* cm = coef + mm * PW;
                            const float2 ro = rot[mm];
                            auto order = [&](int base, int P) {
                                float er = 0.f, ei = 0.f, orr = 0.f, oi = 0.f;
    #pragma unroll 4
                                for (int p = 0; p < P; p += 2) {
                                    const float ca = cm[p], cb = cm[p + 1];
                                    er = fmaf(ca, Fr[(base + p) * kC], er);
                                    ei = fmaf(ca, Fi[(base + p) * kC], ei);
                                    orr = fmaf(cb, Fr[(base + p + 1) * kC], orr);
                                    oi = fmaf(cb, Fi[(base + p + 1) * kC], oi);
                                }
                                // even terms + i odd terms, then the half-sector rotation
                                const float vr = er - fi * oi, vi = fi * ei + orr;
                                return cx<float>{vr * ro.x - vi * ro.y, vr * ro.y + vi * ro.x};
                            };
                            if (mm <= 2 * n_max) m.W[(size_t)mm * plane + at] = order(0, PW);
                            if (mm <= n_max + 3) {
                                const cx<float> a = order(PW, PAB), bb = order(PW + PAB, PAB);
                                if (mm <= n_max - 1)
                                    m.G[(size_t)(mm + n_max + 3) * plane + at] = cx<float>{a.x - bb.y, a.y + bb.x};
                                if (mm >= 1)
                                    m.G[(size_t)(n_max + 3 - mm) * plane + at] = cx<float>{a.x + bb.y, bb.x - a.y};
                            }
                        }
                    }
                    __syncthreads();
                }
            }
        }
        if (tid == 0) s_item = (int)min(atomicAdd(A.queue, 1ull) + gridDim.x, (unsigned long long)nitems);
        __syncthreads();
        item = s_item;
    }
    for (int o = 16; o > 0; o >>= 1) my_pairs += __shfl_xor_sync(FULL, my_pairs, o);
    if (lane == 0 && my_pairs) atomicAdd(m.pairs, my_pairs);
}

template <class PL, bool ADJ>
static cudaError_t launch(const FarArgs& a, int n_sm, cudaStream_t st)
{
    const size_t smem = sizeof(float) * PL::S * PL::KS;
    cudaError_t e = set_smem_attr(far_moments_kernel<PL, ADJ>, smem);
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    e = occupancy(&per_sm, far_moments_kernel<PL, ADJ>, kThreads, smem);
    if (e != cudaSuccess) return e;
    const int64_t items = (int64_t)((a.m.n_centres + kC - 1) / kC) * a.parts;
    const int64_t grid = std::min<int64_t>(items, (int64_t)n_sm * std::max(per_sm, 1));
    if (grid < 1) return cudaSuccess;
    far_moments_kernel<PL, ADJ><<<(unsigned)grid, kThreads, smem, st>>>(a);
    return cudaGetLastError();
}

template <int V>
static void tables(int n_max, FarTables* t, std::vector<float>* out)
{
    using PL = Variant<V>;
    constexpr int S = PL::S, K = 48;  // K Chebyshev nodes, symmetric: half of them are needed
    const double sd = sin(far_dmax(n_max, V));
    const int mtop = std::max(2 * n_max, n_max + 3);
    t->off_ray = (int)out->size();
    t->off_sin = t->off_ray + S / 2 + 4;
    t->off_axis = (t->off_sin + S + 3) / 4 * 4;
    t->off_rot = t->off_axis + 4 * S;
    t->off_coef = t->off_rot + 2 * (mtop + 1);
    out->resize((t->off_coef + (size_t)(mtop + 1) * PL::PW + 3) / 4 * 4, 0.f);
    float* v = out->data();
    for (int j = 1; j < S / 2; ++j) v[t->off_ray + j] = (float)(cos(2 * M_PI * j / S) / sin(2 * M_PI * j / S));
    for (int j = 0; j < S / 2; ++j) {
        const double s0 = sin(2 * M_PI * j / S), s1 = sin(2 * M_PI * (j + 1) / S);
        v[t->off_sin + 2 * j] = (float)std::min(s0, s1);
        v[t->off_sin + 2 * j + 1] = (float)std::max(s0, s1);
    }
    for (int s = 0; s < S; ++s) {
        const double phi = 2 * M_PI * (s + 0.5) / S;
        // the rounded axis (c, s) points at phi + eps: sin(delta) about phi is its cross product plus eps
        const float c = (float)(cos(phi) / sd), sn = (float)(sin(phi) / sd);
        const double eps = atan2((double)sn * cos(phi) - (double)c * sin(phi), (double)c * cos(phi) + (double)sn * sin(phi));
        float* a = v + t->off_axis + 4 * s;
        a[0] = c;
        a[1] = sn;
        a[2] = (float)(eps / sd);
    }
    double ct[PL::PW][K / 2], er[K / 2], ei[K / 2], fr[K / 2], fi[K / 2];
    for (int q = 0; q < K / 2; ++q) {
        const double th = (q + 0.5) * M_PI / K, u = cos(th);
        for (int p = 0; p < PL::PW; ++p) ct[p][q] = p == 0 ? 1.0 : p == 1 ? u : 2 * u * ct[p - 1][q] - ct[p - 2][q];
        er[q] = sqrt(1.0 - sd * sd * u * u);  // e^{i asin(sd u)}
        ei[q] = sd * u;
        fr[q] = 1.0;
        fi[q] = 0.0;
    }
    for (int m = 0; m <= mtop; ++m) {
        v[t->off_rot + 2 * m] = (float)cos(M_PI * m / S);
        v[t->off_rot + 2 * m + 1] = (float)sin(M_PI * m / S);
        for (int p = 0; p < PL::PW; ++p) {
            const double* f = (p & 1) ? fi : fr;
            double c = 0.0;
            for (int q = 0; q < K / 2; ++q) c += f[q] * ct[p][q];
            v[t->off_coef + (size_t)m * PL::PW + p] = (float)(c * (p ? 4.0 : 2.0) / K);
        }
        for (int q = 0; q < K / 2; ++q) {
            const double r = fr[q] * er[q] - fi[q] * ei[q];
            fi[q] = fr[q] * ei[q] + fi[q] * er[q];
            fr[q] = r;
        }
    }
}

}  // namespace far

std::vector<BinGeom> bin_geometry(const std::vector<long long>& e2q)
{
    std::vector<BinGeom> v(e2q.size() - 1);
    for (size_t b = 0; b + 1 < e2q.size(); ++b) {
        BinGeom& g = v[b];
        const double e0 = (double)e2q[b], e1 = (double)e2q[b + 1];  // exact
        g.e0 = e2q[b];
        g.e1 = e2q[b + 1];
        g.Ri = (float)sqrt(e0);
        g.Ro = (float)sqrt(e1);
        g.mid = (float)(0.5 * (e0 + e1));
        // r^2, the subtraction and the bounds themselves round by at most 2^-23 + 2 2^-24 of e1
        const double lo = (double)g.mid - e0, hi = e1 - (double)g.mid, err = 2.5e-7 * e1;
        g.d_in = (float)(std::min(lo, hi) - err);
        g.d_out = (float)(std::max(lo, hi) + err);
        g.pad = 0.f;
    }
    return v;
}

void far_tables(int n_max, FarTables (&t)[kFarPlans], std::vector<float>* v)
{
    far::tables<0>(n_max, &t[0], v);
    far::tables<1>(n_max, &t[1], v);
    far::tables<2>(n_max, &t[2], v);
    far::tables<3>(n_max, &t[3], v);
}

cudaError_t launch_moments_far(const FarArgs& a, int plan, int n_sm, cudaStream_t st)
{
    switch (plan) {
        case 0: return far::launch<far::Variant<0>, false>(a, n_sm, st);
        case 1: return far::launch<far::Variant<1>, false>(a, n_sm, st);
        case 2: return far::launch<far::Variant<2>, false>(a, n_sm, st);
        default: return far::launch<far::Variant<3>, false>(a, n_sm, st);
    }
}

cudaError_t launch_moments_far_adjoint(const FarArgs& a, int plan, int n_sm, cudaStream_t st)
{
    switch (plan) {
        case 0: return far::launch<far::Variant<0>, true>(a, n_sm, st);
        case 1: return far::launch<far::Variant<1>, true>(a, n_sm, st);
        case 2: return far::launch<far::Variant<2>, true>(a, n_sm, st);
        default: return far::launch<far::Variant<3>, true>(a, n_sm, st);
    }
}

}  // namespace mp3
