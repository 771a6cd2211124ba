// Adjoint (reverse mode) of stages (b) and (a): given dL/dUpsilon and dL/dN for a real loss L,
// the gradient with respect to every galaxy's w gamma and w (paper Sec. 3.1: Eqs.
// Upsilon0_Derivation, Upsilon1-3, 3PCF_Normalization, tomoGn for (b); the moment sums of
// Sec. 3.1 for (a)).
//
// Convention: for a complex quantity z, grad z = dL/dRe z + i dL/dIm z. For y = a z,
// grad z += conj(a) grad y; for y = a conj(z), grad z += a conj(grad y); for a real parameter t in
// y = t h, dL/dt += Re(conj(grad y) h).
//
// Stage (b), per group (Z-triplet, component, n) with y(b1, b2) = sum_i c_i X_i(b1) Y_i(b2):
//   grad X_i(b1) = conj(c_i) sum_b2 grad y(b1, b2) conj(Y_i(b2)),
//   grad Y_i(b2) = conj(c_i) sum_b1 grad y(b1, b2) conj(X_i(b1)),
//   grad c_i     = sum_b1 conj(X_i(b1)) sum_b2 grad y(b1, b2) conj(Y_i(b2)),
// with an extra conjugation where the moment enters conjugated. dL/dG and dL/dW are gathered per
// output moment element (each written once): an element receives the X or Y role of
// at most eight (component, n) groups.
//
// Stage (a): G_m(i, b) = sum_k v_k e^{i m phi_ik} and W_m(i, b) = sum_k w_k e^{i m phi_ik}, so
//   grad v_k += sum_{i, m} grad G_m(i, b_ik) e^{-i m phi_ik},
//   dL/dw_k  += Re sum_{i, m} grad W_m(i, b_ik) e^{-i m phi_ik}.
// For each (centre, bin) the adjoint moments are the coefficients of a trigonometric polynomial
// evaluated at every neighbour's angle by Horner's rule (in u = e^{-i phi} for m >= 0 and in
// z = e^{i phi} for m < 0), one neighbour per lane, and added to the neighbour's gradient with
// atomics (the gradient is therefore not bit-reproducible). Neighbours are found per bin from
// the cell grid of the forward pass: for every cell row, the one or two runs of cells that meet
// the annulus. The bins that the forward took by angular sectors go through the transpose of that
// form instead (far_moments_kernel<PL, 1>, moments_far.cu).
#include <math.h>

#include <algorithm>

#include "moments_far.cuh"
#include "sector.cuh"

namespace mp3 {

namespace adj {

__device__ __forceinline__ cx<double> ldd(const double* p, size_t i)
{
    return cx<double>{p[2 * i], p[2 * i + 1]};
}

template <typename T>
__device__ __forceinline__ cx<T> to_t(cx<double> v)
{
    return cx<T>{(T)v.x, (T)v.y};
}

// ------------------------------------------------------------------ stage (b): dL/dG, dL/dW

// the gradient tables of AdjArgs (tabX transposed so that the X role reads consecutive bins)
template <typename T>
__global__ void grad_tables(const AdjArgs<T> a, int64_t n_ups_groups, int64_t total)
{
    const int nb = a.nb, nbb = nb * nb;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t g = i / nbb;
        const int o = (int)(i % nbb), b1 = o / nb, b2 = o % nb;
        const cx<double> v = g < n_ups_groups ? ldd(a.gups, i) : ldd(a.gnorm, i - n_ups_groups * nbb);
        a.tabY[i] = to_t<T>(v);
        a.tabX[g * nbb + (int64_t)b2 * nb + b1] = to_t<T>(v);
    }
}

template <int B>
__device__ __forceinline__ void cp_async(void* dst, const void* src)
{
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(d), "l"(src), "n"(B) : "memory");
}

// (r, i) += t (y.x, y.y) with t's real and imaginary part apart: t y = (r.x - i.y, r.y + i.x) and
// t conj(y) = (r.x + i.y, i.x - r.y), so the partners are staged as they lie in memory
__device__ __forceinline__ void mac_parts(cx<float>& r, cx<float>& i, cx<float> t, cx<float> y)
{
    const float2 v = make_float2(y.x, y.y);
    const float2 a = __ffma2_rn(make_float2(t.x, t.x), v, make_float2(r.x, r.y));
    const float2 b = __ffma2_rn(make_float2(t.y, t.y), v, make_float2(i.x, i.y));
    r = cx<float>{a.x, a.y};
    i = cx<float>{b.x, b.y};
}

__device__ __forceinline__ void mac_parts(cx<double>& r, cx<double>& i, cx<double> t, cx<double> y)
{
    r.x = fma(t.x, y.x, r.x);
    r.y = fma(t.x, y.y, r.y);
    i.x = fma(t.y, y.x, i.x);
    i.y = fma(t.y, y.y, i.y);
}

constexpr int kTileC = 64, kPer = 4, kAdjThreads = 320;

// one role of an order slot: the gradient table at g (X role: transposed), the partner's order slot and
// z-bin, pconj: the partner enters conjugated, mconj: this moment does
struct Role {
    size_t g;
    int qp, z1, zo, kind;
    bool is_x, pconj, mconj;
};

// role r (0..7) of order slot q and z-bin z with centres of z-bin z1 and partners of z-bin zo
__device__ __forceinline__ bool role_of(int r, int q, int z, int z1, int zo, int nz, int nmax, int nbb, Role& o)
{
    const int MG = 2 * nmax + 3, NN = nmax + 1, NW = 2 * nmax + 1, of = nmax + 3;
    o.is_x = (r & 1) == 0;
    o.z1 = z1;
    o.zo = zo;
    // as X this moment is of Z2 and the partner of Z3, as Y the other way round
    const size_t zt = o.is_x ? (size_t)(z1 * nz + z) * nz + zo : (size_t)(z1 * nz + zo) * nz + z;
    if (q >= MG) {
        // N_n: w W_n(b1) conj(W_n(b2))
        const int m = q - MG;
        o.kind = 4;
        o.qp = m;
        o.pconj = o.is_x;
        o.mconj = !o.is_x;
        o.g = ((size_t)nz * nz * nz * 4 * NN + zt * NW + m) * nbb;
        return r < 2;
    }
    const int m = q - of;
    int n, p;
    o.kind = r >> 1;
    switch (r) {
        case 0: n = m + 3; p = -n - 3; break;   // kind 0: -v G_{n-3}(b1) G_{-n-3}(b2)
        case 1: n = -m - 3; p = n - 3; break;
        case 2: n = m + 1; p = -n - 1; break;   // kind 1: -conj(v) G_{n-1}(b1) G_{-n-1}(b2)
        case 3: n = -m - 1; p = n - 1; break;
        case 4: n = -m - 1; p = -n - 3; break;  // kind 2: -v conj(G_{-n-1}(b1)) G_{-n-3}(b2)
        case 5: n = -m - 3; p = -n - 1; break;
        case 6: n = m + 3; p = n - 1; break;    // kind 3: -v G_{n-3}(b1) conj(G_{n-1}(b2))
        default: n = m + 1; p = n - 3; break;
    }
    o.qp = p + of;
    o.pconj = r == 5 || r == 6;
    o.mconj = r == 4 || r == 7;
    o.g = ((zt * 4 + o.kind) * NN + n) * nbb;
    return n >= 0 && n <= nmax;
}

// grid: x = centre tiles, y = output order slot (G slots 0..MG-1, then W slots), z = z-bin. Per role of the
// slot (X or Y of one group, at most eight a partner z-bin) the block stages the group's dL/dy, transposed
// for the X role, and the partner rows of its kTileC centres in shared memory, the next role's while this
// one is worked on (stages 2; 1 where two do not fit); a thread owns one bin of kPer centres, so a table
// element serves kPer products. The X role also gives the gradient of the centre's own coefficient, sum_b1
// conj(X(b1)) sum_b2 dL/dy conj(Y(b2)): the inner sum is the role's. It is reduced over the bins and added
// atomically (every group has exactly one X role). Bound by shared-memory reads and issue. 100 000 centres,
// 20 bins, n_max 30: 7.7 ms; one stage, scalar products and shared atomics 10.4; table and partner elements from
// global memory and the coefficients' gradient in a kernel of its own 22.5.
template <typename T>
__global__ void __launch_bounds__(kAdjThreads, sizeof(T) == 4 ? 2 : 1) contract_adjoint_moments(const AdjArgs<T> a, int stages)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int nb = a.nb, nz = a.nz, nmax = a.n_max, nbp = nb_pad(nb), nbb = nb * nb, nbbp = nbb + (nbb & 1);
    const int MG = 2 * nmax + 3;
    // per stage: [nb][nb] table, the summed bin first, then [kTileC][nbp] partner rows
    cx<T>* buf = reinterpret_cast<cx<T>*>(smem_raw);
    const int stage_len = nbbp + kTileC * nbp;
    __shared__ T gc[3 * kTileC];  // dL/dv (re, im), dL/dw of the centres
    __shared__ cx<T> s_v[kTileC];
    __shared__ T s_w[kTileC];
    __shared__ int s_z[kTileC];
    const int q = blockIdx.y, z = blockIdx.z, c0 = blockIdx.x * kTileC, nc = min(kTileC, a.n_centres - c0);
    const bool isG = q < MG;
    const int slot = isG ? q : q - MG;
    const size_t plane = (size_t)a.n_centres * nz * nbp;
    for (int i = threadIdx.x; i < kTileC; i += blockDim.x) {
        cx<T> v{T(0), T(0)};
        T w = T(0);
        int zc = -1;
        if (i < nc) {
            const int d = a.centre_idx[c0 + i];
            const Pay<T> pv = a.pay[d];
            v = cx<T>{pv.a, pv.b};
            w = pv.w;
            zc = a.zs ? (int)a.zs[d] : 0;
        }
        s_v[i] = v;
        s_w[i] = w;
        s_z[i] = zc;
    }
    for (int i = threadIdx.x; i < 3 * kTileC; i += blockDim.x) gc[i] = T(0);
    __syncthreads();
    const int z_lo = s_z[0], roles = (s_z[nc - 1] - z_lo + 1) * nz * 8;  // the centres are sorted by z-bin
    const cx<T>* M = isG ? a.G : a.W;
    cx<T>* out = (isG ? a.gG : a.gW) + (size_t)slot * plane;
    // the first role from k on (roles: none)
    auto find = [&](int k, Role& o) {
        for (; k < roles; ++k)
            if (role_of(k & 7, q, z, z_lo + (k >> 3) / nz, (k >> 3) % nz, nz, nmax, nbb, o)) break;
        return k;
    };
    auto stage_in = [&](cx<T>* dst, const Role& o) {
        const cx<T>* src = (o.is_x ? a.tabX : a.tabY) + o.g;
        for (int i = threadIdx.x; i < nbb; i += blockDim.x) cp_async<sizeof(cx<T>)>(dst + i, src + i);
        const cx<T>* pr = M + (size_t)o.qp * plane + ((size_t)c0 * nz + o.zo) * nbp;
        cx<T>* part = dst + nbbp;
        constexpr int E = 16 / sizeof(cx<T>);  // elements per 16 bytes
        if (nz == 1) {                         // the rows follow one another
            for (int i = threadIdx.x * E; i < nc * nbp; i += blockDim.x * E) cp_async<16>(part + i, pr + i);
        } else {
            for (int r = threadIdx.x >> 5; r < nc; r += blockDim.x >> 5)
                for (int i = (threadIdx.x & 31) * E; i < nbp; i += 32 * E)
                    cp_async<16>(part + r * nbp + i, pr + (size_t)r * nz * nbp + i);
        }
    };
    // thread -> (bin b, centres i0 + j kTileC / kPer), in passes over the items
    constexpr int kGroups = kTileC / kPer;
    for (int it0 = 0; it0 < kGroups * nb; it0 += blockDim.x) {
        const int it = it0 + threadIdx.x;
        const bool on = it < kGroups * nb;
        const int b = on ? it % nb : 0, i0 = on ? it / nb : 0;
        cx<T> acc[kPer], own[kPer];
        T gr[kPer], gi[kPer];  // the coefficient's gradient (W slots: gr, of the weight)
#pragma unroll
        for (int j = 0; j < kPer; ++j) {
            const int i = i0 + j * kGroups;
            acc[j] = own[j] = cx<T>{T(0), T(0)};
            gr[j] = gi[j] = T(0);
            if (on && i < nc) own[j] = M[(size_t)slot * plane + ((size_t)(c0 + i) * nz + z) * nbp + b];
        }
        Role cur, next;
        int k = find(0, cur), at = 0;
        if (k < roles) stage_in(buf, cur);
        asm volatile("cp.async.commit_group;" ::: "memory");
        while (k < roles) {
            const int kn = find(k + 1, next);
            if (stages == 2) {
                if (kn < roles) stage_in(buf + (at ^ 1) * stage_len, next);
                asm volatile("cp.async.commit_group;" ::: "memory");
                asm volatile("cp.async.wait_group 1;" ::: "memory");
            } else {
                asm volatile("cp.async.wait_group 0;" ::: "memory");
            }
            __syncthreads();
            const cx<T>* tab = buf + at * stage_len + b;
            const cx<T>* part = buf + at * stage_len + nbbp + i0 * nbp;
            cx<T> re[kPer], im[kPer];
#pragma unroll
            for (int j = 0; j < kPer; ++j) re[j] = im[j] = cx<T>{T(0), T(0)};
            int b2 = 0;
            for (; b2 + 1 < nb; b2 += 2) {
                const cx<T> t0 = tab[b2 * nb], t1 = tab[(b2 + 1) * nb];
#pragma unroll
                for (int j = 0; j < kPer; ++j) {
                    const cx<T>* y = part + j * kGroups * nbp + b2;
                    cx<T> y0, y1;
                    if constexpr (sizeof(T) == 4) {
                        const float4 v = *reinterpret_cast<const float4*>(y);  // nbp and b2 are even
                        y0 = cx<T>{v.x, v.y};
                        y1 = cx<T>{v.z, v.w};
                    } else {
                        y0 = y[0];
                        y1 = y[1];
                    }
                    mac_parts(re[j], im[j], t0, y0);
                    mac_parts(re[j], im[j], t1, y1);
                }
            }
            if (b2 < nb) {
                const cx<T> t = tab[b2 * nb];
#pragma unroll
                for (int j = 0; j < kPer; ++j) mac_parts(re[j], im[j], t, part[j * kGroups * nbp + b2]);
            }
#pragma unroll
            for (int j = 0; j < kPer; ++j) {
                const int i = i0 + j * kGroups;
                if (!on || s_z[i] != cur.z1) continue;
                // sum of the table and the conjugate of the partner as it enters the product
                const cx<T> s = cur.pconj ? cx<T>{re[j].x - im[j].y, re[j].y + im[j].x}
                                          : cx<T>{re[j].x + im[j].y, im[j].x - re[j].y};
                const cx<T> v = s_v[i];
                // times conj(coefficient): of w (kind 4), -conj(v) (kind 1) or -v
                const cx<T> cc = cur.kind == 4 ? cx<T>{s_w[i], T(0)} : cx<T>{-v.x, cur.kind == 1 ? -v.y : v.y};
                const cx<T> gx = cmul(s, cc);
                acc[j] = cadd(acc[j], cur.mconj ? cconj(gx) : gx);
                if (cur.is_x) {
                    const cx<T> p = cmul(cur.mconj ? own[j] : cconj(own[j]), s);
                    if (cur.kind == 4) {
                        gr[j] += p.x;  // c = w
                    } else {
                        gr[j] -= p.x;  // c = -v, or -conj(v): grad v = -conj(grad c)
                        gi[j] += cur.kind == 1 ? p.y : -p.y;
                    }
                }
            }
            __syncthreads();
            if (stages == 1) {
                if (kn < roles) stage_in(buf, next);
                asm volatile("cp.async.commit_group;" ::: "memory");
            } else {
                at ^= 1;
            }
            cur = next;
            k = kn;
        }
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();
        // the bins' parts of the coefficient's gradient through shared memory, added per centre (shared
        // atomics on one address by all bins cost more than the roles)
        T* red = reinterpret_cast<T*>(buf);
#pragma unroll
        for (int j = 0; j < kPer; ++j) {
            const int i = i0 + j * kGroups;
            if (on && i < nc) {
                out[((size_t)(c0 + i) * nz + z) * nbp + b] = acc[j];
                red[i * nb + b] = gr[j];
                if (isG) red[(kTileC + i) * nb + b] = gi[j];
            }
        }
        __syncthreads();
        for (int e = threadIdx.x; e < (isG ? 2 : 1) * kTileC; e += blockDim.x) {
            const int i = e % kTileC, first = (i % kGroups) * nb;  // the centre's first item
            if (i >= nc) continue;
            T sum = T(0);
            for (int b2 = max(0, it0 - first); b2 < min(nb, it0 + (int)blockDim.x - first); ++b2) sum += red[e * nb + b2];
            gc[3 * i + (isG ? e / kTileC : 2)] += sum;
        }
        __syncthreads();
    }
    __syncthreads();
    for (int i = threadIdx.x; i < 3 * nc; i += blockDim.x)
        if (gc[i] != T(0)) atomicAdd(&a.gvw[4 * (size_t)a.centre_idx[c0 + i / 3] + i % 3], gc[i]);
}

// ------------------------------------------------------------------ stage (a): pair loop

// adds (re grad v, im grad v, grad w) to a galaxy's 16-byte (FP32) or 32-byte (FP64) slot
__device__ __forceinline__ void atomic_add_vw(float* p, float vr, float vi, float w)
{
    atomicAdd(reinterpret_cast<float4*>(p), make_float4(vr, vi, w, 0.0f));
}
__device__ __forceinline__ void atomic_add_vw(double* p, double vr, double vi, double w)
{
    atomicAdd(p, vr);
    atomicAdd(p + 1, vi);
    atomicAdd(p + 2, w);
}

template <typename T>
__device__ __forceinline__ cx<T> unit_dir(float dx, float dy);
template <>
__device__ __forceinline__ cx<float> unit_dir<float>(float dx, float dy)
{
    const float ir = rsqrtf(dx * dx + dy * dy);
    return {dx * ir, dy * ir};
}
template <>
__device__ __forceinline__ cx<double> unit_dir<double>(float dx, float dy)
{
    const double fx = (double)dx, fy = (double)dy;
    const double ir = 1.0 / sqrt(fx * fx + fy * fy);
    return {fx * ir, fy * ir};
}

constexpr int kPairWarps = 4;

// one Horner step p <- p x + c in four fused multiply-adds
template <typename T>
__device__ __forceinline__ cx<T> horner_step(cx<T> p, cx<T> x, cx<T> c)
{
    return {fma(p.x, x.x, fma(-p.y, x.y, c.x)), fma(p.x, x.y, fma(p.y, x.x, c.y))};
}

constexpr int kList = 128;  // candidates listed at a time per warp

// Walks the candidates of redshift bin z around the centre at pc (from the grid's origin): the lanes find
// the one or two runs of cells of 32 cell rows at a time that meet bin b's annulus (annulus_runs), the
// candidates are listed in row order in the warp's list, and f(in, k, dx, dy) is called on every lane for
// 32 of them at a time (warp-uniform), with in = whether galaxy k is in the bin (decided on the integers
// near an edge). Must be called by the whole warp. A walk over one row at a time with 64-bit
// divisions took about 1500 instructions a row, most of the time of the narrow bins.
template <typename T, typename F>
__device__ __forceinline__ void for_each_in_annulus(const AdjArgs<T>& a, float2 pc, int b, int z, int lane, int* list, F&& f)
{
    constexpr unsigned FULL = 0xffffffffu;
    const BinGeom* bg = a.bins + b;
    SectorGeom g;
    g.gx = pc.x;
    g.gy = pc.y;
    g.hx = g.hy = 0.0f;
    g.Ri = bg->Ri;
    g.Ro = bg->Ro;
    g.S = (float)a.g.side;
    g.iS = 1.0f / g.S;
    g.ncx = a.g.ncx;
    g.ncy = a.g.ncy;
    const float mid = bg->mid, d_in = bg->d_in, d_out = bg->d_out;
    const int* row_start = a.cell_start + (size_t)z * a.g.ncells;
    const float ro = g.Ro + 8.0f;
    const float iy0 = fmaxf(floorf((g.gy - ro) * g.iS), 0.0f), iy1 = fminf(floorf((g.gy + ro) * g.iS), (float)(g.ncy - 1));
    for (float iy = iy0 + (float)lane; iy - (float)lane <= iy1; iy += 32.0f) {
        int st0 = 0, n0 = 0, st1 = 0, n1 = 0;
        if (iy <= iy1) annulus_runs(g, iy, (iy + 0.5f) * g.S - g.gy, 0, g.ncx - 1, row_start, st0, n0, st1, n1);
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
            const int off = incl - len, put = max(0, min(len, kList - off));
            for (int j = 0; j < put; ++j) list[off + j] = j < n0 ? st0 + j : st1 + (j - n0);
            const int t0 = min(put, n0);
            st0 += t0;
            n0 -= t0;
            st1 += put - t0;
            n1 -= put - t0;
            const int n = min(total, kList);
            __syncwarp();
            for (int t = lane; t < n + lane; t += 32) {
                const int k = list[min(t, n - 1)];
                const float2 p = a.posf[k];
                const float dx = p.x - pc.x, dy = p.y - pc.y;  // exact
                const float d = fabsf(fmaf(dx, dx, dy * dy) - mid);
                bool in = d < d_in;
                if (!in && d < d_out) {
                    const long long q2 = (long long)(int)dx * (int)dx + (long long)(int)dy * (int)dy;
                    in = q2 >= bg->e0 && q2 < bg->e1;
                }
                f(in && t < n, k, dx, dy);
            }
            __syncwarp();
            if (total <= kList) break;
        }
    }
}

// warp per centre (grid-stride); per bin the warp stages the centre's adjoint moments of every Z
// in shared memory and walks the annulus. The members found are queued (unit vector, galaxy) in
// the warp's shared-memory queue and evaluated 32 at a time, one per lane, so that no lane idles
// through the polynomial evaluations while others hold a member.
constexpr int kQueue = 64;

template <typename T>
__global__ void __launch_bounds__(kPairWarps * 32) moments_adjoint_pairs(const AdjArgs<T> a)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int nb = a.nb, nz = a.nz, nmax = a.n_max, nbp = nb_pad(nb);
    const int MG = 2 * nmax + 3, MW = 2 * nmax + 1, o = nmax + 3;
    __shared__ int list[kPairWarps][kList];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const unsigned lt_mask = (1u << lane) - 1u;
    cx<T>* co = reinterpret_cast<cx<T>*>(smem_raw) + (size_t)warp * nz * (MG + MW);  // [z][MG + MW]
    cx<T>* qz = reinterpret_cast<cx<T>*>(smem_raw) + (size_t)kPairWarps * nz * (MG + MW) + (size_t)warp * kQueue;
    int* qk = reinterpret_cast<int*>(reinterpret_cast<cx<T>*>(smem_raw) + (size_t)kPairWarps * nz * (MG + MW) +
                                     (size_t)kPairWarps * kQueue) + warp * kQueue;
    const size_t plane = (size_t)a.n_centres * nz * nbp;
    for (int c = blockIdx.x * kPairWarps + warp; c < a.n_centres; c += gridDim.x * kPairWarps) {
        const int d = a.centre_idx[c];
        const float2 p = a.posf[d];
        for (int b = 0; b < a.nb_pairs; ++b) {
            __syncwarp();
            for (int i = lane; i < nz * (MG + MW); i += 32) {
                const int z = i / (MG + MW), qq = i % (MG + MW);
                co[i] = qq < MG ? a.gG[(size_t)qq * plane + ((size_t)c * nz + z) * nbp + b]
                                : a.gW[(size_t)(qq - MG) * plane + ((size_t)c * nz + z) * nbp + b];
            }
            __syncwarp();
            for (int z = 0; z < nz; ++z) {
                const cx<T>* gg = co + (size_t)z * (MG + MW);
                const cx<T>* gw = gg + MG;
                // grad v_k += sum_m gG_m e^{-i m phi}, grad w_k += Re sum_m gW_m e^{-i m phi} for the
                // queued member e
                auto eval = [&](int e) {
                    const cx<T> zz = qz[e];
                    const int k = qk[e];
                    const cx<T> u{zz.x, -zz.y};
                    // m >= 0 part of sum_m gG_m u^m (Horner in u, P <- P u + c: four FMAs)
                    cx<T> P{T(0), T(0)};
#pragma unroll 4
                    for (int mm = nmax - 1; mm >= 0; --mm) P = horner_step(P, u, gg[o + mm]);
                    // m < 0 part: sum_{j >= 1} gG_{-j} z^j = z (gG_{-1} + z (gG_{-2} + ...))
                    cx<T> Q = gg[o - (nmax + 3)];
#pragma unroll 4
                    for (int j = nmax + 2; j >= 1; --j) Q = horner_step(Q, zz, gg[o - j]);
                    Q = cmul(Q, zz);
                    // W: sum_m gW_m u^m
                    cx<T> Rw{T(0), T(0)};
#pragma unroll 4
                    for (int mm = 2 * nmax; mm >= 0; --mm) Rw = horner_step(Rw, u, gw[mm]);
                    atomic_add_vw(a.gvw + 4 * (size_t)k, P.x + Q.x, P.y + Q.y, Rw.x);
                };
                int qn = 0;  // queued members (warp-uniform), < 32 between steps
                for_each_in_annulus(a, p, b, z, lane, list[warp],
                                    [&](bool in, int k, float dx, float dy) {
                    const unsigned m = __ballot_sync(0xffffffffu, in);
                    if (in) {
                        const int slot = qn + __popc(m & lt_mask);
                        qz[slot] = unit_dir<T>(dx, dy);
                        qk[slot] = k;
                    }
                    qn += __popc(m);
                    if (qn >= 32) {
                        __syncwarp();
                        eval(lane);
                        __syncwarp();
                        if (lane < qn - 32) {
                            qz[lane] = qz[32 + lane];
                            qk[lane] = qk[32 + lane];
                        }
                        __syncwarp();
                        qn -= 32;
                    }
                });
                __syncwarp();
                if (lane < qn) eval(lane);
                __syncwarp();
            }
        }
    }
}

// caller order, v = w (gamma_1 + i gamma_2): dL/dgamma_1 = w Re grad v, dL/dgamma_2 = w Im grad v,
// dL/dw = (direct) + Re grad v gamma_1 + Im grad v gamma_2; ADDS to the caller's arrays
template <typename T>
__global__ void adjoint_finish(int64_t n, const int* __restrict__ perm, const T* __restrict__ gvw,
                               const float* __restrict__ g1, const float* __restrict__ g2,
                               const float* __restrict__ w, float* __restrict__ dg1, float* __restrict__ dg2,
                               float* __restrict__ dw)
{
    for (int64_t d = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; d < n; d += (int64_t)gridDim.x * blockDim.x) {
        const int i = perm[d];
        const T vr = gvw[4 * d], vi = gvw[4 * d + 1];
        const T wi = (T)w[i];
        if (dg1) dg1[i] += (float)(wi * vr);
        if (dg2) dg2[i] += (float)(wi * vi);
        if (dw) dw[i] += (float)(gvw[4 * d + 2] + vr * (T)g1[i] + vi * (T)g2[i]);
    }
}

// ------------------------------------------------------------------ exclude_degenerate

template <typename T>
__device__ __forceinline__ T warp_sum(T v)
{
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Per (centre, z, bin) the sums over neighbours k of redshift bin z in the bin that the j = k
// triplets contribute (u = e^{-i phi}, v = w gamma): D6 = sum v^2 u^6, D2 = sum v^2 u^2,
// E2 = sum |v|^2 u^2, F = sum w^2, written as 4 complex values (F in the real part).
template <typename T>
__global__ void __launch_bounds__(kPairWarps * 32) degenerate_moments(const AdjArgs<T> a, cx<T>* __restrict__ out)
{
    const int nb = a.nb, nz = a.nz;
    __shared__ int list[kPairWarps][kList];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int c = blockIdx.x * kPairWarps + warp; c < a.n_centres; c += gridDim.x * kPairWarps) {
        const float2 p = a.posf[a.centre_idx[c]];
        for (int b = 0; b < nb; ++b)
            for (int z = 0; z < nz; ++z) {
                T s[7] = {T(0), T(0), T(0), T(0), T(0), T(0), T(0)};
                for_each_in_annulus(a, p, b, z, lane, list[warp],
                                    [&](bool in, int k, float dx, float dy) {
                    if (!in) return;
                    const cx<T> zz = unit_dir<T>(dx, dy);
                    const cx<T> u{zz.x, -zz.y};
                    const cx<T> u2 = cmul(u, u), u6 = cmul(cmul(u2, u2), u2);
                    const Pay<T> pk = a.pay[k];
                    const cx<T> v{pk.a, pk.b};
                    const cx<T> v2 = cmul(v, v);
                    const T vv = pk.a * pk.a + pk.b * pk.b;
                    const cx<T> d6 = cmul(v2, u6), d2 = cmul(v2, u2);
                    s[0] += d6.x;
                    s[1] += d6.y;
                    s[2] += d2.x;
                    s[3] += d2.y;
                    s[4] += vv * u2.x;
                    s[5] += vv * u2.y;
                    s[6] += pk.w * pk.w;
                });
                for (int i = 0; i < 7; ++i) s[i] = warp_sum(s[i]);
                if (lane == 0) {
                    cx<T>* o = out + (((size_t)c * nz + z) * nb + b) * 4;
                    o[0] = cx<T>{s[0], s[1]};
                    o[1] = cx<T>{s[2], s[3]};
                    o[2] = cx<T>{s[4], s[5]};
                    o[3] = cx<T>{s[6], T(0)};
                }
            }
    }
}

// Block per (z1, z, bin): S0 = sum_i v_i D6, S1 = sum_i conj(v_i) D2, S2 = sum_i v_i E2,
// SN = sum_i w_i F over the centres of redshift bin z1 (FP64, fixed order), then for the triplet
// (z1, z, z) and b1 = b2 = bin, every order: Upsilon_0 += S0, Upsilon_1 += S1, Upsilon_2,3 += S2,
// N -= SN (the j = k terms of the paper's sums, removed).
template <typename T>
__global__ void __launch_bounds__(256) degenerate_correct(const AdjArgs<T> a, const cx<T>* __restrict__ dm,
                                                         double* __restrict__ ups, double* __restrict__ norm)
{
    const int nb = a.nb, nz = a.nz, nmax = a.n_max, NN = nmax + 1, NW = 2 * nmax + 1;
    const int b = blockIdx.x % nb, z = (blockIdx.x / nb) % nz, z1 = blockIdx.x / (nb * nz);
    double s[7] = {0, 0, 0, 0, 0, 0, 0};
    for (int c = threadIdx.x; c < a.n_centres; c += blockDim.x) {
        const int d = a.centre_idx[c];
        if ((a.zs ? (int)a.zs[d] : 0) != z1) continue;
        const Pay<T> pv = a.pay[d];
        const cx<double> v{(double)pv.a, (double)pv.b};
        const cx<T>* m = dm + (((size_t)c * nz + z) * nb + b) * 4;
        const cx<double> d6{(double)m[0].x, (double)m[0].y}, d2{(double)m[1].x, (double)m[1].y};
        const cx<double> e2{(double)m[2].x, (double)m[2].y};
        const cx<double> t0 = cmul(v, d6), t1 = cmul(cconj(v), d2), t2 = cmul(v, e2);
        s[0] += t0.x; s[1] += t0.y; s[2] += t1.x; s[3] += t1.y; s[4] += t2.x; s[5] += t2.y;
        s[6] += (double)pv.w * (double)m[3].x;
    }
    __shared__ double red[7][256];
    for (int i = 0; i < 7; ++i) red[i][threadIdx.x] = s[i];
    __syncthreads();
    for (int h = blockDim.x / 2; h > 0; h >>= 1) {
        if ((int)threadIdx.x < h)
            for (int i = 0; i < 7; ++i) red[i][threadIdx.x] += red[i][threadIdx.x + h];
        __syncthreads();
    }
    const int zt = (z1 * nz + z) * nz + z;
    const size_t bb = (size_t)b * nb + b, nbb = (size_t)nb * nb;
    cx<double>* U = reinterpret_cast<cx<double>*>(ups);
    cx<double>* N = reinterpret_cast<cx<double>*>(norm);
    for (int n = threadIdx.x; n < NN; n += blockDim.x) {
        const cx<double> S0{red[0][0], red[1][0]}, S1{red[2][0], red[3][0]}, S2{red[4][0], red[5][0]};
        U[(((size_t)zt * 4 + 0) * NN + n) * nbb + bb] = cadd(U[(((size_t)zt * 4 + 0) * NN + n) * nbb + bb], S0);
        U[(((size_t)zt * 4 + 1) * NN + n) * nbb + bb] = cadd(U[(((size_t)zt * 4 + 1) * NN + n) * nbb + bb], S1);
        U[(((size_t)zt * 4 + 2) * NN + n) * nbb + bb] = cadd(U[(((size_t)zt * 4 + 2) * NN + n) * nbb + bb], S2);
        U[(((size_t)zt * 4 + 3) * NN + n) * nbb + bb] = cadd(U[(((size_t)zt * 4 + 3) * NN + n) * nbb + bb], S2);
    }
    for (int m = threadIdx.x; m < NW; m += blockDim.x) {
        cx<double>& e = N[((size_t)zt * NW + m) * nbb + bb];
        e.x -= red[6][0];
    }
}

// ---- adjoint of the exclude_degenerate correction. The forward adds S0 = sum_i v_i D6_i to every
// order of Upsilon_0, S1 = sum_i v_i^* D2_i to Upsilon_1, S2 = sum_i v_i E2_i to Upsilon_2 and
// Upsilon_3 and subtracts SN = sum_i w_i F_i from Re N (b1 = b2, Z2 = Z3). Block-free pass first:
// per (Z1, z, bin) gS0 = sum_n dL/dUpsilon_0,n, gS1, gS2 (Upsilon_2 and _3) and gSN = -sum_m
// Re dL/dN_m, stored as dgs[(z1 nz + z) nb + b][0..3] (gSN in the real part).
__global__ void degenerate_grad_sums(int nz, int nb, int n_max, const double* __restrict__ gups,
                                     const double* __restrict__ gnorm, cx<double>* __restrict__ dgs)
{
    const int NN = n_max + 1, NW = 2 * n_max + 1;
    const int total = nz * nz * nb;
    const size_t nbb = (size_t)nb * nb;
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < total; t += gridDim.x * blockDim.x) {
        const int b = t % nb, z = (t / nb) % nz, z1 = t / (nb * nz);
        const int zt = (z1 * nz + z) * nz + z;
        const size_t bb = (size_t)b * nb + b;
        cx<double> g[3] = {{0.0, 0.0}, {0.0, 0.0}, {0.0, 0.0}};
        for (int n = 0; n < NN; ++n)
            for (int mu = 0; mu < 4; ++mu) {
                const size_t i = 2 * ((((size_t)zt * 4 + mu) * NN + n) * nbb + bb);
                const int slot = mu < 3 ? mu : 2;
                g[slot].x += gups[i];
                g[slot].y += gups[i + 1];
            }
        double gn = 0.0;
        for (int m = 0; m < NW; ++m) gn -= gnorm[2 * (((size_t)zt * NW + m) * nbb + bb)];
        dgs[(size_t)t * 4 + 0] = g[0];
        dgs[(size_t)t * 4 + 1] = g[1];
        dgs[(size_t)t * 4 + 2] = g[2];
        dgs[(size_t)t * 4 + 3] = cx<double>{gn, 0.0};
    }
}

// Warp per centre i: per (bin, z) of the neighbours, with u = e^{-i phi_ij},
//   grad v_j += 2 v_j^* (u^6)^* gD6 + 2 v_j^* (u^2)^* gD2 + 2 v_j Re(gE2 (u^2)^*),
//   grad w_j += 2 w_j gF,   gD6 = v_i^* gS0, gD2 = v_i gS1, gE2 = v_i^* gS2, gF = w_i gSN,
// and, with the centre's own sums D6, D2, E2, F (re-formed in the same walk),
//   grad v_i += D6^* gS0 + D2 gS1^* + E2^* gS2,   grad w_i += F gSN.
template <typename T>
__global__ void __launch_bounds__(kPairWarps * 32) degenerate_adjoint_pairs(const AdjArgs<T> a)
{
    const int nb = a.nb, nz = a.nz;
    __shared__ int list[kPairWarps][kList];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int c = blockIdx.x * kPairWarps + warp; c < a.n_centres; c += gridDim.x * kPairWarps) {
        const int d = a.centre_idx[c];
        const float2 p = a.posf[d];
        const int z1 = a.zs ? (int)a.zs[d] : 0;
        const Pay<T> pv = a.pay[d];
        const cx<double> vi{(double)pv.a, (double)pv.b};
        const double wi = (double)pv.w;
        double cgr = 0.0, cgi = 0.0, cgw = 0.0;  // the centre's own gradient (lane 0 adds it)
        for (int b = 0; b < nb; ++b)
            for (int z = 0; z < nz; ++z) {
                const cx<double>* gs = a.dgs + ((size_t)(z1 * nz + z) * nb + b) * 4;
                const cx<double> gS0 = gs[0], gS1 = gs[1], gS2 = gs[2];
                const double gSN = gs[3].x;
                const cx<double> gD6 = cmul(cconj(vi), gS0), gD2 = cmul(vi, gS1), gE2 = cmul(cconj(vi), gS2);
                const double gF = wi * gSN;
                double sd[7] = {0, 0, 0, 0, 0, 0, 0};  // this lane's share of D6, D2, E2, F
                for_each_in_annulus(a, p, b, z, lane, list[warp],
                                    [&](bool in, int k, float dx, float dy) {
                    if (!in) return;
                    const cx<T> zz = unit_dir<T>(dx, dy);
                    const cx<double> u{(double)zz.x, -(double)zz.y};
                    const cx<double> u2 = cmul(u, u), u6 = cmul(cmul(u2, u2), u2);
                    const Pay<T> pk = a.pay[k];
                    const cx<double> vj{(double)pk.a, (double)pk.b};
                    const double wj = (double)pk.w;
                    const cx<double> vj2 = cmul(vj, vj);
                    const cx<double> d6 = cmul(vj2, u6), d2 = cmul(vj2, u2);
                    const double vv = vj.x * vj.x + vj.y * vj.y;
                    sd[0] += d6.x;
                    sd[1] += d6.y;
                    sd[2] += d2.x;
                    sd[3] += d2.y;
                    sd[4] += vv * u2.x;
                    sd[5] += vv * u2.y;
                    sd[6] += wj * wj;
                    const cx<double> t6 = cmul(cmul(cconj(vj), cconj(u6)), gD6);
                    const cx<double> t2 = cmul(cmul(cconj(vj), cconj(u2)), gD2);
                    const double re = cmul(gE2, cconj(u2)).x;
                    atomic_add_vw(a.gvw + 4 * (size_t)k, (T)(2.0 * (t6.x + t2.x + vj.x * re)),
                                  (T)(2.0 * (t6.y + t2.y + vj.y * re)), (T)(2.0 * wj * gF));
                });
                for (int i = 0; i < 7; ++i) sd[i] = warp_sum(sd[i]);
                const cx<double> D6{sd[0], sd[1]}, D2{sd[2], sd[3]}, E2{sd[4], sd[5]};
                const cx<double> gv = cadd(cadd(cmul(cconj(D6), gS0), cmul(D2, cconj(gS1))), cmul(cconj(E2), gS2));
                cgr += gv.x;
                cgi += gv.y;
                cgw += sd[6] * gSN;
            }
        if (lane == 0) atomic_add_vw(a.gvw + 4 * (size_t)d, (T)cgr, (T)cgi, (T)cgw);
    }
}

template <typename T>
static cudaError_t run_degenerate(const AdjArgs<T>& a, cx<T>* scratch, double* ups, double* norm, int n_sm,
                                  cudaStream_t st)
{
    if (a.n_centres <= 0) return cudaSuccess;
    const int blocks = (int)std::min<int64_t>((a.n_centres + kPairWarps - 1) / kPairWarps, (int64_t)n_sm * 32);
    degenerate_moments<T><<<blocks, kPairWarps * 32, 0, st>>>(a, scratch);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    degenerate_correct<T><<<a.nz * a.nz * a.nb, 256, 0, st>>>(a, scratch, ups, norm);
    return cudaGetLastError();
}

template <typename T>
static cudaError_t run(const AdjArgs<T>& a, int64_t n, const int* perm, const float* g1, const float* g2,
                       const float* w, float* dg1, float* dg2, float* dw, int n_sm, cudaStream_t st,
                       cudaError_t (*far)(void*) = nullptr, void* far_arg = nullptr)
{
    cudaError_t e = cudaMemsetAsync(a.gvw, 0, sizeof(T) * 4 * (size_t)n, st);
    if (e != cudaSuccess) return e;
    if (a.n_centres > 0) {
        const int MG = 2 * a.n_max + 3, MW = 2 * a.n_max + 1;
        const dim3 g1d((a.n_centres + kTileC - 1) / kTileC, MG + MW, a.nz);
        const int64_t z3 = (int64_t)a.nz * a.nz * a.nz, nbb = (int64_t)a.nb * a.nb;
        const int64_t nU = z3 * 4 * (a.n_max + 1), tot = (nU + z3 * (2 * a.n_max + 1)) * nbb;
        grad_tables<T><<<(unsigned)std::min<int64_t>((tot + 255) / 256, (int64_t)n_sm * 16), 256, 0, st>>>(a, nU, tot);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        // two stages where they leave room for two blocks on an SM
        const size_t stage = sizeof(cx<T>) * ((size_t)nbb + (nbb & 1) + (size_t)kTileC * nb_pad(a.nb));
        const int stages = stage <= 54 * 1024 ? 2 : 1;
        const size_t sm_mom = stages * stage;
        if ((e = set_smem_attr(contract_adjoint_moments<T>, sm_mom)) != cudaSuccess) return e;
        // threads: the items in as few, equally full passes as kAdjThreads allows
        const int items = kTileC / kPer * a.nb, passes = (items + kAdjThreads - 1) / kAdjThreads;
        const int threads = ((items + passes - 1) / passes + 31) / 32 * 32;
        contract_adjoint_moments<T><<<g1d, threads, sm_mom, st>>>(a, stages);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        const size_t sm_pair = sizeof(cx<T>) * (size_t)kPairWarps * (a.nz * (MG + MW) + kQueue) +
                               sizeof(int) * (size_t)kPairWarps * kQueue;
        e = set_smem_attr(moments_adjoint_pairs<T>, sm_pair);
        if (e != cudaSuccess) return e;
        const int blocks = (int)std::min<int64_t>((a.n_centres + kPairWarps - 1) / kPairWarps, (int64_t)n_sm * 32);
        if (a.nb_pairs > 0) moments_adjoint_pairs<T><<<blocks, kPairWarps * 32, sm_pair, st>>>(a);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        if (far && (e = far(far_arg)) != cudaSuccess) return e;
    }
    if (a.dgs && a.n_centres > 0) {
        // the j = k triplets left out of the forward (exclude_degenerate)
        const int total = a.nz * a.nz * a.nb;
        degenerate_grad_sums<<<(total + 127) / 128, 128, 0, st>>>(a.nz, a.nb, a.n_max, a.gups, a.gnorm, a.dgs);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        const int blocks = (int)std::min<int64_t>((a.n_centres + kPairWarps - 1) / kPairWarps, (int64_t)n_sm * 32);
        degenerate_adjoint_pairs<T><<<blocks, kPairWarps * 32, 0, st>>>(a);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    const unsigned gb = (unsigned)std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, (int64_t)n_sm * 16));
    adjoint_finish<T><<<gb, 256, 0, st>>>(n, perm, a.gvw, g1, g2, w, dg1, dg2, dw);
    return cudaGetLastError();
}

}  // namespace adj

cudaError_t launch_moments_adjoint_f32(const AdjArgs<float>& a, int64_t n, const int* perm, const float* g1,
                                       const float* g2, const float* w, float* dg1, float* dg2, float* dw,
                                       int n_sm, cudaStream_t st, cudaError_t (*far)(void*), void* far_arg)
{
    return adj::run<float>(a, n, perm, g1, g2, w, dg1, dg2, dw, n_sm, st, far, far_arg);
}

cudaError_t launch_moments_adjoint_f64(const AdjArgs<double>& a, int64_t n, const int* perm, const float* g1,
                                       const float* g2, const float* w, float* dg1, float* dg2, float* dw,
                                       int n_sm, cudaStream_t st)
{
    return adj::run<double>(a, n, perm, g1, g2, w, dg1, dg2, dw, n_sm, st);
}

}  // namespace mp3

namespace mp3 {

cudaError_t launch_degenerate_f32(const AdjArgs<float>& a, void* scratch, double* ups, double* norm, int n_sm,
                                  cudaStream_t st)
{
    return adj::run_degenerate<float>(a, reinterpret_cast<cx<float>*>(scratch), ups, norm, n_sm, st);
}

cudaError_t launch_degenerate_f64(const AdjArgs<double>& a, void* scratch, double* ups, double* norm, int n_sm,
                                  cudaStream_t st)
{
    return adj::run_degenerate<double>(a, reinterpret_cast<cx<double>*>(scratch), ups, norm, n_sm, st);
}

}  // namespace mp3
