// Gradient of J = sum_b <g_b, L r_b> with respect to the profile knots f_t.
//
// With rho_m(i,j) = sum_k c_k K_k cos(m x_k) (see contract.cu) the objective is
//     J = sum_{pairs (i,j)} sum_{m=0}^{N/2} rho_m(i,j) Q_m(i,j),
//     Q_m(i,j) = eta_m sum_b Re( w_j a_m(j,b) conj(g_m(i,b)) ),  eta = 1, 2, ..., 2, 1,
// where a and g are the (extended) ring spectra of the input maps and of the output
// gradients, so dJ/dK_k(i,j) = c_k sum_m cos(m x_k) Q_m(i,j), and K_k depends on the knots
// through the hat weights of the linear-in-u lookup.  N-S mirror pairs share their taps and
// contribute Q(i,j) + Q(R-1-i, R-1-j).  The pole rings add the derivative of their true-
// profile direct sum.  Every warp adds its deposits in a fixed order into bins of its own, a CTA's
// bins are summed in order, and the CTAs' rows too, so the result is bitwise reproducible.  Each
// launch serves several kernels.
#include <algorithm>

#include "fft_engine.cuh"

namespace arkcos {

namespace {

constexpr int kQRing = 8;  // representative rings per Q CTA


// Q[p][m] for all pairs p of a block of representative rings and 128 modes (grid x: mode
// blocks, y: ring blocks).  Q is written to global memory, pairs-major.
__global__ void __launch_bounds__(kModeBlock) k_knot_q(const __grid_constant__ KnotGradArgs a)
{
    chain_allow_next();
    chain_wait();
    const int kb = blockIdx.z;
    float *Q = a.Q + kb * a.qstride;
    const int tid = threadIdx.x;
    const int m = blockIdx.x * kModeBlock + tid;
    if (m >= a.NH) return;
    const int r0 = blockIdx.y * kQRing;
    const int nr = min(kQRing, a.nrep - r0);
    const KernDev &kd = a.kd[kb];
    const float eta = (m == 0 || 2 * m == a.N) ? 1.f : 2.f;
    for (int li = 0; li < nr; ++li) {
        const int i = r0 + li;
        const bool mirror = a.R - 1 - i != i;
        const bool pole = a.pole_fix && i == 0;  // ring 0 and R-1 carry no hybrid output
        const int p0 = kd.pstart[i], p1 = kd.pstart[i + 1], jl = kd.jlo[i];
        for (int p = p0; p < p1; ++p) {
            const int j = jl + (p - p0);
            float q = 0.f;
            if (!pole) {
                const int map0 = a.map0 + kb * a.per_map;
                for (int b = 0; b < a.nmaps; ++b) {
                    const float4 *sa = a.spec4 + (int64_t)(map0 + b) * a.nrep * a.NH;
                    const float4 *sg = a.gspec4 + (int64_t)(map0 + b) * a.nrep * a.NH;
                    const float4 x = paired_coeff(sa, j, a.R, a.NH, m);   // a(j), a(R-1-j)
                    const float4 y = paired_coeff(sg, i, a.R, a.NH, m);   // g(i), g(R-1-i)
                    q = fmaf(x.x, y.x, fmaf(x.y, y.y, q));
                    if (mirror) q = fmaf(x.z, y.z, fmaf(x.w, y.w, q));
                }
            }
            Q[(int64_t)p * a.NH + m] = eta * q;
        }
    }
}

// Q for bands of at most kQBand rings: thread = (mode, representative output ring i) with
// g(i) and g(R-1-i) in registers, the union band of the input spectra staged per map in
// shared memory (double-buffered cp.async), and one accumulator per ring pair of the band.
constexpr int kQBand = 32, kQModes = 64, kQRings = 8;

__global__ void __launch_bounds__(kQModes *kQRings, 2) k_knot_q_band(const __grid_constant__ KnotGradArgs a)
{
    chain_allow_next();
    chain_wait();
    const int kb = blockIdx.z;
    float *Q = a.Q + kb * a.qstride;
    extern __shared__ float4 qsh[];
    const int tm = threadIdx.x & (kQModes - 1);
    const int li = threadIdx.x / kQModes;
    const int m = blockIdx.x * kQModes + tm;
    const bool mv = m < a.NH;
    const int r0 = blockIdx.y * kQRings;
    const int nr = min(kQRings, a.nrep - r0);
    const bool lv = li < nr;
    const KernDev &kd = a.kd[kb];
    const int i = r0 + (lv ? li : 0);
    const int jl = kd.jlo[i], ps = kd.pstart[i];
    const int blen = lv ? kd.jhi[i] - jl + 1 : 0;
    const int ju0 = kd.jlo[r0];
    const int nu = kd.jhi[r0 + nr - 1] - ju0 + 1;
    const bool mirror = a.R - 1 - i != i;
    const bool pole = a.pole_fix && i == 0;  // ring 0 and R-1 carry no hybrid output
    const int mid = (a.R - 1) / 2;
    const bool crosses = ju0 + nu - 1 > mid;
    const int sstar = mid - jl + 1;
    const int joff = jl - ju0;
    const size_t bufsz = (size_t)nu * kQModes;
    const int m0 = blockIdx.x * kQModes;
    float q[kQBand];
#pragma unroll
    for (int s = 0; s < kQBand; ++s) q[s] = 0.f;
    const int b0 = a.map0 + kb * a.per_map, b1 = b0 + a.nmaps;
    if (b0 < b1) stage_band_async(qsh, a.spec4 + (int64_t)b0 * a.nrep * a.NH, ju0, nu, m0, kQModes, a.R, a.NH);
    for (int b = b0; b < b1; ++b) {
        const int cur = (b - b0) & 1;
        if (b + 1 < b1)
            stage_band_async(qsh + (cur ^ 1) * bufsz, a.spec4 + (int64_t)(b + 1) * a.nrep * a.NH, ju0, nu, m0,
                             kQModes, a.R, a.NH);
        else
            cp_async_commit();
        float4 g = make_float4(0.f, 0.f, 0.f, 0.f);  // (g(i), g(R-1-i))
        if (lv && mv) g = __ldg(&a.gspec4[((int64_t)b * a.nrep + i) * a.NH + m]);
        if (!mirror) g.z = g.w = 0.f;
        if (pole) g = make_float4(0.f, 0.f, 0.f, 0.f);
        cp_async_wait1();
        __syncthreads();
        if (lv && mv) {
            const float4 *col = qsh + cur * bufsz + joff * kQModes + tm;
#pragma unroll
            for (int s = 0; s < kQBand; ++s) {
                if (s < blen) {
                    float4 v = col[s * kQModes];
                    if (crosses && s >= sstar) v = make_float4(v.z, v.w, v.x, v.y);
                    q[s] = fmaf(v.x, g.x, fmaf(v.y, g.y, fmaf(v.z, g.z, fmaf(v.w, g.w, q[s]))));
                }
            }
        }
        __syncthreads();
    }
    if (lv && mv) {
        const float eta = (m == 0 || 2 * m == a.N) ? 1.f : 2.f;
#pragma unroll
        for (int s = 0; s < kQBand; ++s)
            if (s < blen) Q[(int64_t)(ps + s) * a.NH + m] = eta * q[s];
    }
}

// Q for bands whose every two consecutive rings have a union band of at most kQBand rings:
// thread = (mode, group of two output rings i0 = 2g, i1 = i0 + 1 of the block) over the common
// run of kQBand input rings from jlo(i0), so each staged value feeds both rings (twice the
// arithmetic per shared-memory load of k_knot_q_band).  Rows past the block's union band stay
// zero; products outside a ring's band are accumulated but never stored.
constexpr int kQGModes = 64, kQGGroups = 4;  // 8 rings per CTA

__global__ void __launch_bounds__(kQGModes *kQGGroups, 2) k_knot_q_g2(const __grid_constant__ KnotGradArgs a, int srows)
{
    chain_allow_next();
    chain_wait();
    const int kb = blockIdx.z;
    float *Q = a.Q + kb * a.qstride;
    extern __shared__ float4 qgs[];  // [2 buffers][srows][kQGModes]
    const int tm = threadIdx.x & (kQGModes - 1);
    const int grp = threadIdx.x / kQGModes;
    const int m = blockIdx.x * kQGModes + tm;
    const bool mv = m < a.NH;
    const int r0 = blockIdx.y * 2 * kQGGroups;
    const int nr = min(2 * kQGGroups, a.nrep - r0);
    const KernDev &kd = a.kd[kb];
    const int i0 = r0 + 2 * grp, i1 = i0 + 1;
    const bool v0 = 2 * grp < nr, v1 = 2 * grp + 1 < nr;  // warp-uniform (a warp is one group)
    const int jg0 = v0 ? kd.jlo[i0] : 0;
    const int ju0 = kd.jlo[r0];
    const int nu = kd.jhi[r0 + nr - 1] - ju0 + 1;
    const int joff = jg0 - ju0;
    const int mid = (a.R - 1) / 2;
    const bool crosses = ju0 + nu - 1 > mid;
    const int sstar = mid - jg0 + 1;  // first slot of the run that is a southern ring
    const size_t bufsz = (size_t)srows * kQGModes;
    const int m0 = blockIdx.x * kQGModes;
    for (size_t e = threadIdx.x; e < 2 * bufsz; e += blockDim.x) qgs[e] = make_float4(0.f, 0.f, 0.f, 0.f);
    __syncthreads();
    float q0[kQBand], q1[kQBand];
#pragma unroll
    for (int u = 0; u < kQBand; ++u) q0[u] = q1[u] = 0.f;
    // (g(i), g(R-1-i)) of a representative output ring, zero for the pole ring under the pole
    // fix (its hybrid output is replaced) and without the mirror term for the middle ring
    auto gload = [&](int b, int i, bool v) {
        float4 g = make_float4(0.f, 0.f, 0.f, 0.f);
        if (v && mv) g = __ldg(&a.gspec4[((int64_t)b * a.nrep + i) * a.NH + m]);
        if (a.R - 1 - i == i) g.z = g.w = 0.f;
        if (a.pole_fix && i == 0) g = make_float4(0.f, 0.f, 0.f, 0.f);
        return g;
    };
    const int b0 = a.map0 + kb * a.per_map, b1 = b0 + a.nmaps;
    if (b0 < b1) stage_band_async(qgs, a.spec4 + (int64_t)b0 * a.nrep * a.NH, ju0, nu, m0, kQGModes, a.R, a.NH);
    for (int b = b0; b < b1; ++b) {
        const int cur = (b - b0) & 1;
        if (b + 1 < b1)
            stage_band_async(qgs + (cur ^ 1) * bufsz, a.spec4 + (int64_t)(b + 1) * a.nrep * a.NH, ju0, nu, m0,
                             kQGModes, a.R, a.NH);
        else
            cp_async_commit();
        const float4 g0 = gload(b, i0, v0), g1 = gload(b, i1, v1);
        cp_async_wait1();
        __syncthreads();
        if (v0) {
            const float4 *col = qgs + cur * bufsz + joff * kQGModes + tm;
            if (!crosses) {
#pragma unroll
                for (int u = 0; u < kQBand; ++u) {
                    const float4 v = col[u * kQGModes];
                    q0[u] = fmaf(v.x, g0.x, fmaf(v.y, g0.y, fmaf(v.z, g0.z, fmaf(v.w, g0.w, q0[u]))));
                    q1[u] = fmaf(v.x, g1.x, fmaf(v.y, g1.y, fmaf(v.z, g1.z, fmaf(v.w, g1.w, q1[u]))));
                }
            } else {
#pragma unroll
                for (int u = 0; u < kQBand; ++u) {
                    float4 v = col[u * kQGModes];
                    if (u >= sstar) v = make_float4(v.z, v.w, v.x, v.y);
                    q0[u] = fmaf(v.x, g0.x, fmaf(v.y, g0.y, fmaf(v.z, g0.z, fmaf(v.w, g0.w, q0[u]))));
                    q1[u] = fmaf(v.x, g1.x, fmaf(v.y, g1.y, fmaf(v.z, g1.z, fmaf(v.w, g1.w, q1[u]))));
                }
            }
        }
        __syncthreads();
    }
    if (v0 && mv) {
        const float eta = (m == 0 || 2 * m == a.N) ? 1.f : 2.f;
        const int ps0 = kd.pstart[i0], len0 = kd.jhi[i0] - jg0 + 1;
#pragma unroll
        for (int u = 0; u < kQBand; ++u)
            if (u < len0) Q[(int64_t)(ps0 + u) * a.NH + m] = eta * q0[u];
        if (v1) {
            const int ps1 = kd.pstart[i1], d = kd.jlo[i1] - jg0, len1 = kd.jhi[i1] - kd.jlo[i1] + 1;
#pragma unroll
            for (int u = 0; u < kQBand; ++u)
                if (u >= d && u < d + len1) Q[(int64_t)(ps1 + u - d) * a.NH + m] = eta * q1[u];
        }
    }
}

// Adds w0 to bins[t0] and w1 to bins[t0 + 1] for every lane with t0 >= 0: the lanes of a warp, in
// its own bins, lane by lane only where they share a knot, so the order is fixed.
__device__ __forceinline__ void warp_deposit(double *bins, int t0, double w0, double w1)
{
    const unsigned same = __match_any_sync(0xffffffffu, t0);
    const int rank = __popc(same & ((1u << (threadIdx.x & 31)) - 1u));
    const int most = __reduce_max_sync(0xffffffffu, t0 >= 0 ? rank : -1);
    for (int q = 0; q <= most; ++q) {
        const bool mine = t0 >= 0 && rank == q;
        if (mine) bins[t0] += w0;
        __syncwarp();
        if (mine) bins[t0 + 1] += w1;
        __syncwarp();
    }
}

constexpr int kProjTaps = 8, kProjReseed = 16, kProjWarps = 8;  // k_knot_deposit, k_knot_proj

// Warps of a deposit CTA with bins of their own, and whether the table of reciprocal knot spacings has
// room beside them.
struct BinShape {
    int warps, table;
};

// Knot tables and per-warp bins of a deposit CTA in shared memory.
struct KnotBins {
    double *ut, *inv, *bins;  // [T] knots in u, [T] 1 / spacing (none: divided per sample), [warps][T]
    int T, warps;
    __device__ KnotBins(double *sm, const KernDev &kd, BinShape bs)
        : ut(sm), inv(bs.table ? sm + kd.T : nullptr), bins(sm + (1 + bs.table) * kd.T), T(kd.T), warps(bs.warps)
    {
        for (int t = threadIdx.x; t < T; t += blockDim.x) {
            ut[t] = kd.ut[t];
            if (inv) inv[t] = t < T - 1 ? 1.0 / (kd.ut[t + 1] - kd.ut[t]) : 0.0;
        }
        for (int t = threadIdx.x; t < warps * T; t += blockDim.x) bins[t] = 0.0;
        __syncthreads();
    }
    // 1 / spacing of segment t < T - 1
    __device__ __forceinline__ double spacing(int t) const { return inv ? inv[t] : 1.0 / (ut[t + 1] - ut[t]); }
    // the warps' bins summed in order into a row of partial sums
    __device__ void write(double *row)
    {
        __syncthreads();
        for (int t = threadIdx.x; t < T; t += blockDim.x) {
            double s = 0.0;
            for (int w = 0; w < warps; ++w) s += bins[w * T + t];
            row[t] = s;
        }
    }
};

// Deposit CTA of up to `most` warps with bins of their own beside `other` bytes, T up to 4096: as many
// as fit 200 KB with both tables, but one at least.  Beside the 16384-point transform of
// k_knot_proj_fft (139392 bytes) that one fits the 227 KB of a CTA with both tables up to T = 3877, and
// with the knots alone up to T = 4096.
BinShape bin_shape(int T, int most, size_t other)
{
    const int64_t row = (int64_t)T * (int64_t)sizeof(double);
    const int64_t rows = std::max<int64_t>(0, 200 * 1024 - (int64_t)other) / row;
    const int warps = (int)std::max<int64_t>(1, std::min<int64_t>(most, rows - 2));
    return BinShape{warps, (int64_t)other + (2 + warps) * row <= 227 * 1024};
}
// The same for k_knot_proj, whose warps all project: bins of their own or shared by turns, within a third
// of an SM, with the table where it fits beside them.
BinShape proj_shape(int T)
{
    int warps = kProjWarps;
    while (warps > 1 && (size_t)(1 + warps) * T * sizeof(double) > 74 * 1024) warps /= 2;
    return BinShape{warps, (size_t)(2 + warps) * T * sizeof(double) <= 74 * 1024};
}
size_t bin_bytes(int T, BinShape bs) { return (size_t)(1 + bs.table + bs.warps) * T * sizeof(double); }

// Hat weights of sample k of pair p: its knot segment and position in it.
__device__ __forceinline__ int sample_knot(const KnotGradArgs &a, const KernDev &kd, const KnotBins &kb, int p, int k, int f,
                                           double &lam)
{
    const int tt = 2 * k + f;
    const double u = fmin(4.0 * (kd.B[p] * a.s2[a.N - tt] + kd.A[p] * a.s2[tt]), kd.umax);
    const int t0 = knot_segment(u, kb.ut, kb.T, kd.gscale);
    lam = (u - kb.ut[t0]) * kb.spacing(t0);
    return t0;
}

// Plain FP32 projection by table: X[p][t] = sum_m Q_m(p) cos(pi m (2t + f) / N), a lane per tap
// t (32 at a time), a CTA for 16 consecutive pairs, whose taps share each cosine loaded (of
// either offset; the pairs' own by a uniform choice); its warps take every fourth 32 modes, and
// their sums (kept short: 128 modes at a time) are added in order.  Loads of the cosines through
// L1 bound it: 50 us per kernel at nside 256, 160 us with a phasor per pair, tap and mode.
constexpr int kXPairs = 16, kXWarps = 4;

__global__ void __launch_bounds__(kXWarps * 32) k_knot_proj_f32(const __grid_constant__ KnotGradArgs a,
                                                                const float *__restrict__ ctabP, int nmc)
{
    chain_allow_next();
    const int kb = blockIdx.z;
    const KernDev &kd = a.kd[kb];
    const int lane = threadIdx.x & 31, pf = a.fft_pairs[kb], NH = a.NH;
    const int p0 = pf + blockIdx.x * kXPairs, t = blockIdx.y * 32 + lane, wid = threadIdx.x >> 5;
    chain_wait();
    if (p0 >= kd.npairs) return;
    int most = 0;
    unsigned fm = 0;  // bit i: offset of pair p0 + i
    const float *q = a.Q + kb * a.qstride + (int64_t)p0 * NH;
#pragma unroll
    for (int i = 0; i < kXPairs; ++i) {
        const int p = min(p0 + i, kd.npairs - 1);
        const int f = a.shift_fix ? kd.fl[p] : 0;
        fm |= (unsigned)f << i;
        most = max(most, (f ? kd.S1[p] : kd.S0[p]) + 1);
    }
    if (blockIdx.y * 32 >= (unsigned)most) return;
    const bool any0 = fm != (1u << kXPairs) - 1u, any1 = fm != 0;
    const int np = min(kXPairs, kd.npairs - p0);
    // a chunk's Q values of the pairs, loaded a mode per lane
    __shared__ __align__(16) float qs_all[kXWarps][kXPairs][32];
    float (&qs)[kXPairs][32] = qs_all[wid];
    // rows t and 128 + t of the table tiles (32 modes: 8 x 16-byte pieces 128 bytes apart)
    const float4 *c0 = reinterpret_cast<const float4 *>(ctabP) + (t >> 3) * 64 + (t & 7), *c1 = c0 + 16 * 64;
    float acc[kXPairs], tot[kXPairs];
#pragma unroll
    for (int i = 0; i < kXPairs; ++i) acc[i] = tot[i] = 0.f;
    int since = 0;
    for (int c = wid; c < nmc; c += kXWarps) {
        __syncwarp();
#pragma unroll
        for (int i = 0; i < kXPairs; ++i) qs[i][lane] = i < np && 32 * c + lane < NH ? __ldg(&q[(int64_t)i * NH + 32 * c + lane]) : 0.f;
        __syncwarp();
#pragma unroll 2
        for (int j = 0; j < 8; ++j) {
            const int64_t o = (int64_t)c * 4096 + j * 8;
            const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
            const float4 h0 = any0 ? __ldg(&c0[o]) : z, l0 = any0 ? __ldg(&c0[o + 2048]) : z;
            const float4 h1 = any1 ? __ldg(&c1[o]) : z, l1 = any1 ? __ldg(&c1[o + 2048]) : z;
            const float x0[4] = {h0.x + l0.x, h0.y + l0.y, h0.z + l0.z, h0.w + l0.w};
            const float x1[4] = {h1.x + l1.x, h1.y + l1.y, h1.z + l1.z, h1.w + l1.w};
#pragma unroll
            for (int i = 0; i < kXPairs; ++i) {
                const float4 v = *reinterpret_cast<const float4 *>(&qs[i][4 * j]);
                acc[i] = fmaf(v.x, fm >> i & 1 ? x1[0] : x0[0], acc[i]);
                acc[i] = fmaf(v.y, fm >> i & 1 ? x1[1] : x0[1], acc[i]);
                acc[i] = fmaf(v.z, fm >> i & 1 ? x1[2] : x0[2], acc[i]);
                acc[i] = fmaf(v.w, fm >> i & 1 ? x1[3] : x0[3], acc[i]);
            }
        }
        if (++since == 4 || c + kXWarps >= nmc) {
            since = 0;
#pragma unroll
            for (int i = 0; i < kXPairs; ++i) {
                tot[i] += acc[i];
                acc[i] = 0.f;
            }
        }
    }
    // the warps' sums in order (their Q values are no longer needed)
    __syncthreads();
#pragma unroll
    for (int i = 0; i < kXPairs; ++i) qs[i][lane] = tot[i];
    __syncthreads();
    for (int i = wid; i < np; i += kXWarps) {
        float x = qs_all[0][i][lane];
#pragma unroll
        for (int w = 1; w < kXWarps; ++w) x += qs_all[w][i][lane];
        a.X[kb * a.xstride + (int64_t)(p0 + i - pf) * 128 + t] = x;
    }
}

// Hat-weight deposits of the projected pairs: c_k X_k goes to the knots of u(x_k) with weights
// 1 - lam and lam.  A warp takes four pairs at a time, eight lanes to a pair and its taps, and adds
// into its own bins; the CTA writes their sum as its row of partial sums.  FP64 bounds it: 0.08 ms
// for one nside-2048 kernel, 0.57 ms with a round's deposits staged for one thread to add.
__global__ void __launch_bounds__(kProjWarps * 32) k_knot_deposit(const __grid_constant__ KnotGradArgs a, BinShape bs)
{
    extern __shared__ double ksm[];
    const int kb = blockIdx.y;
    const KernDev &kd = a.kd[kb];
    KnotBins bn(ksm, kd, bs);
    const int nw = bs.warps;
    chain_wait();
    chain_allow_next();
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, pf = a.fft_pairs[kb];
    const double invN = 1.0 / (double)a.N;
    const float *X = a.X + kb * a.xstride;
    if (wid < nw) {
        for (int p4 = pf + 4 * (blockIdx.x * nw + wid); p4 < kd.npairs; p4 += 4 * gridDim.x * nw) {
            const int p = p4 + (lane >> 3);
            int f = 0, ntap = 0;
            if (p < kd.npairs) {
                f = a.shift_fix ? kd.fl[p] : 0;
                ntap = (f ? kd.S1[p] : kd.S0[p]) + 1;
            }
            const int most = __reduce_max_sync(0xffffffffu, ntap);
            for (int k0 = 0; k0 < most; k0 += 8) {
                const int k = k0 + (lane & 7);
                int t0 = -1;
                double w0 = 0.0, w1 = 0.0;
                if (k < ntap) {
                    const double mult = (f == 0 && (k == 0 || 2 * k == a.N)) ? 1.0 : 2.0;
                    const double x = (double)__ldg(&X[(int64_t)(p - pf) * 128 + k]) * mult * invN;
                    double lam;
                    t0 = sample_knot(a, kd, bn, p, k, f, lam);
                    w1 = lam * x;
                    w0 = x - w1;
                }
                warp_deposit(bn.bins + wid * bn.T, t0, w0, w1);
            }
        }
    }
    bn.write(a.partial + kb * a.pstride + (int64_t)blockIdx.x * bn.T);
}

// Projection and deposits of pairs of more than 128 samples without the FFT form: work unit =
// (pair, kProjTaps consecutive taps), from a table built with the kernel.  A warp takes one unit
// at a time with its lanes over the modes m = lane + 32 t (coalesced Q loads) and, per tap, the
// phasor z = exp(i m x_k) advanced by exp(i 32 x_k) each step and reseeded from computed ones every
// kProjReseed steps.  The lane sums are reduced by shuffles and deposited in the warp's bins; with many
// knots several warps share bins and deposit in turn, so that three CTAs (as many as the registers
// allow) still fit an SM: the phasors need the warps (nside 2000, 2048 knots, backward: 9.1 ms, 17.1 ms
// with bins for every warp and one CTA per SM; 4096 knots 9.2 and 29.7 ms).
template <bool SHARED>  // some bins belong to several warps
__global__ void __launch_bounds__(kProjWarps * 32) k_knot_proj(const __grid_constant__ KnotGradArgs a, BinShape bs)
{
    extern __shared__ double ksm[];
    const int kb = blockIdx.y;
    const KernDev &kd = a.kd[kb];
    KnotBins bn(ksm, kd, bs);
    chain_wait();
    chain_allow_next();
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int N = a.N, NH = a.NH;
    const double invN = 1.0 / (double)N;
    const int2 *units = a.shift_fix ? kd.unit_fix : kd.unit_nofix;
    const int nunits = a.shift_fix ? kd.nunit_fix : kd.nunit_nofix;
    for (int u0 = blockIdx.x * kProjWarps; u0 < nunits; u0 += gridDim.x * kProjWarps) {
        int t0 = -1;
        double w0 = 0.0, w1 = 0.0;
        if (u0 + wid < nunits) {
            const int2 un = __ldg(&units[u0 + wid]);
            const int p = un.x, k0 = un.y;
            const int f = a.shift_fix ? kd.fl[p] : 0;
            const int ntap = (f ? kd.S1[p] : kd.S0[p]) + 1;
            float mine = 0.f;
            const float *q = a.Q + kb * a.qstride + (int64_t)p * NH;
            float acc[kProjTaps], zr[kProjTaps], zi[kProjTaps], wr[kProjTaps], wi[kProjTaps];
#pragma unroll
            for (int j = 0; j < kProjTaps; ++j) {
                const int ang = 2 * (k0 + j) + f;  // x = pi ang / N
                const float2 w = expipi_ratio(32 * ang, N);
                wr[j] = w.x;
                wi[j] = w.y;
                acc[j] = 0.f;
                zr[j] = zi[j] = 0.f;
            }
            const int nsteps = (NH + 31) >> 5;
            for (int t = 0; t < nsteps; ++t) {
                const int m = lane + 32 * t;
                const float qm = m < NH ? __ldg(&q[m]) : 0.f;
                if (t % kProjReseed == 0) {
#pragma unroll
                    for (int j = 0; j < kProjTaps; ++j) {
                        const float2 z = expipi_ratio((2 * (k0 + j) + f) * m, N);
                        zr[j] = z.x;
                        zi[j] = z.y;
                    }
                }
#pragma unroll
                for (int j = 0; j < kProjTaps; ++j) {
                    acc[j] = fmaf(qm, zr[j], acc[j]);
                    const float r = fmaf(zr[j], wr[j], -zi[j] * wi[j]);
                    zi[j] = fmaf(zr[j], wi[j], zi[j] * wr[j]);
                    zr[j] = r;
                }
            }
#pragma unroll
            for (int j = 0; j < kProjTaps; ++j) {
                float v = acc[j];
                for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
                if (lane == j) mine = v;
            }
            const int k = k0 + lane;
            if (lane < kProjTaps && k < ntap) {
                const double mult = (f == 0 && (k == 0 || 2 * k == N)) ? 1.0 : 2.0;
                const double x = (double)mine * mult * invN;
                double lam;
                t0 = sample_knot(a, kd, bn, p, k, f, lam);
                w1 = lam * x;
                w0 = x - w1;
            }
        }
        if constexpr (SHARED) {
            for (int turn = 0; turn < kProjWarps / bs.warps; ++turn) {
                if (wid / bs.warps == turn) warp_deposit(bn.bins + wid % bs.warps * bn.T, t0, w0, w1);
                __syncthreads();
            }
        } else {
            warp_deposit(bn.bins + wid * bn.T, t0, w0, w1);
        }
    }
    bn.write(a.partial + kb * a.pstride + (int64_t)blockIdx.x * bn.T);
}

// The projection of the pairs next to the poles (up to N/2 + 1 samples each) by FFT.  The even
// extension of Q (half of Q_m at m and at N - m, with the phases exp(+-i pi m f / N)) has the real
// transform sum_m Q_m cos(m x_k), so one N-point inverse transform (the adjoint passes from
// digit-reversed input) projects two pairs, as its real and imaginary part.  Then the
// hat-weight deposits of every in-support sample, 32 consecutive samples to a warp and its bins; the
// CTA's sum is one row.  The 2297 pairs of one nside-2048 kernel take 0.22 ms, 0.76 ms
// with a transform per pair and one thread adding its samples.
template <int L>
struct ProjFft {
    const KnotGradArgs &a;
    const KernDev &kd;
    const float *Q;
    float2 *buf;
    KnotBins &bn;
    int p0, np;
    __device__ void run()
    {
        constexpr int N = 1 << L;
        const int NH = a.NH;
        const fft::Smem<L> sm{buf};
        int f[2], ntap[2];
        const float *q[2];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const int p = min(p0 + i, np - 1);
            f[i] = a.shift_fix ? kd.fl[p] : 0;
            ntap[i] = p0 + i < np ? (f[i] ? kd.S1[p] : kd.S0[p]) + 1 : 0;
            q[i] = Q + (int64_t)p * NH;
        }
        // the input of the pairs in `which` (bit i: pair p0 + i); whether some value is not finite
        auto fill = [&](int which) {
            bool bad = false;
            for (int m = threadIdx.x; m < NH; m += blockDim.x) {
                const bool edge = m == 0 || 2 * m == N;  // its own mirror
                const float2 ph = expipi_ratio(m, N);
                float2 e[2];  // Q_m exp(i pi m f / N), halved where the mirror holds the conjugate
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    const float v = (which >> i & 1) && ntap[i] > 0 ? __ldg(&q[i][m]) : 0.f, w = edge ? v : 0.5f * v;
                    bad |= !isfinite(v);
                    e[i] = f[i] ? make_float2(w * ph.x, edge ? 0.f : w * ph.y) : make_float2(w, 0.f);
                }
                // both pairs as real and imaginary part: e0 + i e1, and conj e0 + i conj e1 at N - m
                sm(fft::digitrev<L>(m), make_float2(e[0].x - e[1].y, e[0].y + e[1].x));
                if (!edge) sm(fft::digitrev<L>(N - m), make_float2(e[0].x + e[1].y, e[1].x - e[0].y));
            }
            return bad;
        };
        const double invN = 1.0 / (double)N;
        const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
        // a value that is not finite would reach the other pair's samples too: a transform each then
        const bool apart = __syncthreads_or(fill(3));
        for (int r = 0; r < (apart ? 2 : 1); ++r) {
            if (apart) {
                (void)fill(1 << r);
                __syncthreads();
            }
            fft::adj<L>(buf, a.tw, sm);
            if (wid < bn.warps) {
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    if (apart && i != r) continue;
                    for (int k0 = 32 * wid; k0 < ntap[i]; k0 += 32 * bn.warps) {
                        const int k = k0 + lane;
                        int t0 = -1;
                        double w0 = 0.0, w1 = 0.0;
                        if (k < ntap[i]) {
                            const float2 v = sm(k);
                            const double mult = (f[i] == 0 && (k == 0 || 2 * k == N)) ? 1.0 : 2.0;
                            const double x = (double)(i ? v.y : v.x) * mult * invN;
                            double lam;
                            t0 = sample_knot(a, kd, bn, p0 + i, k, f[i], lam);
                            w1 = lam * x;
                            w0 = x - w1;
                        }
                        warp_deposit(bn.bins + wid * bn.T, t0, w0, w1);
                    }
                }
            }
            if (apart) __syncthreads();
        }
    }
};

__global__ void __launch_bounds__(1024) k_knot_proj_fft(const __grid_constant__ KnotGradArgs a, int logN, BinShape bs)
{
    extern __shared__ float2 kbuf[];
    chain_allow_next();  // (the kernel before waited for Q)
    const int kb = blockIdx.y, p0 = 2 * blockIdx.x, np = a.fft_pairs[kb];
    if (p0 < np) {
        const KernDev &kd = a.kd[kb];
        KnotBins bn(reinterpret_cast<double *>(kbuf + fft::buffer_words(1 << logN)), kd, bs);
        const float *Q = a.Q + kb * a.qstride;
        switch (logN) {
        case 10: ProjFft<10>{a, kd, Q, kbuf, bn, p0, np}.run(); break;
        case 11: ProjFft<11>{a, kd, Q, kbuf, bn, p0, np}.run(); break;
        case 12: ProjFft<12>{a, kd, Q, kbuf, bn, p0, np}.run(); break;
        case 13: ProjFft<13>{a, kd, Q, kbuf, bn, p0, np}.run(); break;
        default: ProjFft<14>{a, kd, Q, kbuf, bn, p0, np}.run(); break;
        }
        bn.write(a.partial + kb * a.pstride + (int64_t)(a.row_fft + blockIdx.x) * bn.T);
    }
    chain_wait();
}

// Pole rings: d/df_t of sum_p g_p sum_q w_q K(u_pq) r_q: pole_split CTAs per (pole pixel, side,
// map) and kernel share the pixels of the band's rings (one run of the map), a row each.  Four
// kernels in one launch: 15 us; ring by ring with three FP64 sines per pixel and one thread adding
// a CTA's deposits: 154 us each.
constexpr int kPoleWarps = 8;

__global__ void __launch_bounds__(kPoleWarps * 32) k_knot_pole(const __grid_constant__ KnotGradArgs a, const float *map,
                                                               const float *gout, int64_t npix, BinShape bs)
{
    extern __shared__ double ksm[];
    chain_allow_next();
    const int kb = blockIdx.z / a.nmaps, b = blockIdx.z % a.nmaps, m = a.map0 + kb * a.per_map + b;
    const int C = a.pole_split[kb], p = blockIdx.x % 4, part = blockIdx.x / 4, e = blockIdx.y;
    if (part >= C) {
        chain_wait();
        return;
    }
    const KernDev &kd = a.kd[kb];
    const RingDev &rd = a.rd;
    KnotBins bn(ksm, kd, bs);
    const int nw = bs.warps;
    const int i = e == 0 ? 0 : a.R - 1, jh = kd.jhi[0], ja = e == 0 ? 0 : a.R - 1 - jh, jz = e == 0 ? jh : a.R - 1;
    const float *r = map + (int64_t)m * npix;
    const double gp = (double)gout[(int64_t)m * npix + rd.poff[i] + p];
    const int64_t q0 = rd.poff[ja], q1 = rd.poff[jz] + rd.n[jz];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (wid < nw) {
        for (int64_t q32 = q0 + 32 * (part * nw + wid); q32 < q1; q32 += 32 * C * nw) {
            const int64_t q = q32 + lane;
            int t0 = -1;
            double w0 = 0.0, w1 = 0.0;
            if (q < q1) {
                int j = ja, hi = jz;  // the pixel's ring
                while (j < hi) {
                    const int mid = (j + hi + 1) >> 1;
                    if (__ldg(&rd.poff[mid]) <= q) j = mid;
                    else hi = mid - 1;
                }
                // squared chord as in pole.cu
                const double y = (double)(2 * p + rd.hs[i]) / (2.0 * rd.n[i]) -
                                 (double)(2 * (int)(q - rd.poff[j]) + rd.hs[j]) / (2.0 * rd.n[j]);
                const int jj = e == 0 ? j : a.R - 1 - j;
                const double sy = sinpi(y), B = kd.B[jj], u = 4.0 * fma(kd.A[jj] - B, sy * sy, B);
                if (u <= kd.umax) {
                    t0 = knot_segment(u, bn.ut, bn.T, kd.gscale);
                    const double x = gp * (double)rd.w[j] * (double)__ldg(&r[q]);
                    w1 = (u - bn.ut[t0]) * bn.spacing(t0) * x;
                    w0 = x - w1;
                }
            }
            warp_deposit(bn.bins + wid * bn.T, t0, w0, w1);
        }
    }
    bn.write(a.partial + kb * a.pstride + (int64_t)(a.row_pole + ((b * 2 + e) * 4 + p) * C + part) * bn.T);
    chain_wait();
}

// One CTA per knot and kernel: each thread sums a strided subset of the rows in order, then a tree
// over the threads in a fixed pairing, so the result does not depend on scheduling.
// The rows of a kernel: deposit CTAs, then its FFT pairs (two to a row), then the pole rings from
// row_pole (a kernel with fewer FFT pairs than the longest of the call leaves rows unused).
__global__ void __launch_bounds__(256) k_knot_reduce(const __grid_constant__ KnotGradArgs a, int T, double *out)
{
    __shared__ double red[256];
    chain_wait();
    const int t = blockIdx.x, kb = blockIdx.y, head = a.row_fft + (a.fft_pairs[kb] + 1) / 2;
    const int pole_rows = a.pole_fix ? 8 * a.nmaps * a.pole_split[kb] : 0;
    const double *partial = a.partial + kb * a.pstride;
    double s = 0.0;
    for (int r = threadIdx.x; r < head + pole_rows; r += blockDim.x)
        s += partial[(int64_t)(r < head ? r : r - head + a.row_pole) * T + t];
    red[threadIdx.x] = s;
    __syncthreads();
    for (int h = blockDim.x / 2; h > 0; h >>= 1) {
        if (threadIdx.x < h) red[threadIdx.x] += red[threadIdx.x + h];
        __syncthreads();
    }
    if (threadIdx.x == 0) out[(int64_t)kb * T + t] = red[0];
}

}  // namespace

int knot_proj_blocks() { return device_sms() * 3; }
int knot_proj_taps() { return kProjTaps; }

int knot_q_form(int max_band, int max_union, int max_union2, int srows)
{
    if (max_union2 <= kQBand && 2 * (size_t)srows * kQGModes * sizeof(float4) <= 100 * 1024) return 0;
    return max_band <= kQBand && 2 * (size_t)max_union * kQModes * sizeof(float4) <= 200 * 1024 ? 1 : 2;
}

cudaError_t launch_knot_grad_q(const KnotGradArgs &a, int max_band, int max_union, int max_union2, int srows,
                               cudaStream_t st)
{
    const int form = knot_q_form(max_band, max_union, max_union2, srows);
    if (form == 0) {
        const size_t smem = 2 * (size_t)srows * kQGModes * sizeof(float4);
        cudaError_t e = cudaFuncSetAttribute((const void *)k_knot_q_g2,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        dim3 grid((a.NH + kQGModes - 1) / kQGModes, (a.nrep + 2 * kQGGroups - 1) / (2 * kQGGroups), a.nk);
        return launch_chained(k_knot_q_g2, grid, kQGModes * kQGGroups, smem, st, true, 1, a, srows);
    }
    if (form == 1) {
        const size_t smem = 2 * (size_t)max_union * kQModes * sizeof(float4);
        cudaError_t e = cudaFuncSetAttribute((const void *)k_knot_q_band,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        dim3 grid((a.NH + kQModes - 1) / kQModes, (a.nrep + kQRings - 1) / kQRings, a.nk);
        return launch_chained(k_knot_q_band, grid, kQModes * kQRings, smem, st, true, 1, a);
    }
    dim3 grid((a.NH + kModeBlock - 1) / kModeBlock, (a.nrep + kQRing - 1) / kQRing, a.nk);
    return launch_chained(k_knot_q, grid, kModeBlock, 0, st, true, 1, a);
}

cudaError_t launch_knot_proj_f32(const KnotGradArgs &a, const float *ctabP, int nmc, int maxpairs, int maxtaps,
                                 cudaStream_t st)
{
    if (maxpairs <= 0) return cudaSuccess;
    dim3 grid((maxpairs + kXPairs - 1) / kXPairs, (maxtaps + 31) / 32, a.nk);
    return launch_chained(k_knot_proj_f32, grid, kXWarps * 32, 0, st, true, 1, a, ctabP, nmc);
}

cudaError_t launch_knot_grad_proj(const KnotGradArgs &a, bool have_x, int T, cudaStream_t st)
{
    const BinShape bs = have_x ? bin_shape(T, kProjWarps, 0) : proj_shape(T);
    const size_t smem = bin_bytes(T, bs);
    const auto kernel = have_x ? k_knot_deposit : bs.warps < kProjWarps ? k_knot_proj<true> : k_knot_proj<false>;
    cudaError_t e = cudaFuncSetAttribute((const void *)kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    return launch_chained(kernel, dim3(knot_proj_blocks(), a.nk), kProjWarps * 32, smem, st, true, 1, a, bs);
}

// The kernels' FFT pairs (the caller checks that N is a power of two in [2^10, 2^14] and within
// the grid's twiddle table), two to a CTA and row.
cudaError_t launch_knot_grad_proj_fft(const KnotGradArgs &a, int maxpairs, int T, cudaStream_t st)
{
    if (maxpairs <= 0) return cudaSuccess;
    int logN = 0;
    while ((1 << logN) < a.N) ++logN;
    const size_t buf = (size_t)fft::buffer_words(a.N) * sizeof(float2);
    const BinShape bs = bin_shape(T, std::max(1, a.N / 16 / 32), buf);
    const size_t smem = buf + bin_bytes(T, bs);
    cudaError_t e = cudaFuncSetAttribute((const void *)k_knot_proj_fft,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    return launch_chained(k_knot_proj_fft, dim3((maxpairs + 1) / 2, a.nk), a.N / 16, smem, st, true, 1, a, logN, bs);
}

int knot_pole_split(int64_t band_pixels)
{
    int c = 1;
    while (c < 8 && 512 * (int64_t)c < band_pixels) c *= 2;
    return c;
}

cudaError_t launch_knot_grad_pole(const KnotGradArgs &a, const float *map, const float *gout, int64_t npix, int T,
                                  cudaStream_t st)
{
    const BinShape bs = bin_shape(T, kPoleWarps, 0);
    const size_t smem = bin_bytes(T, bs);
    cudaError_t e = cudaFuncSetAttribute((const void *)k_knot_pole,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    int split = 1;
    for (int k = 0; k < a.nk; ++k) split = std::max(split, a.pole_split[k]);
    return launch_chained(k_knot_pole, dim3(4 * split, 2, a.nmaps * a.nk), kPoleWarps * 32, smem, st, true, 1, a,
                          map, gout, npix, bs);
}

cudaError_t launch_knot_reduce(const KnotGradArgs &a, double *out, int T, cudaStream_t st)
{
    return launch_chained(k_knot_reduce, dim3(T, a.nk), 256, 0, st, true, 1, a, T, out);
}

}  // namespace arkcos
