// Kernel sampling (Sec. 4.1: kernel grid centred on each output ring) and the tabulated Fourier
// coefficients of the ring pairs next to the poles; the other pairs' coefficients are generated
// inside the contraction (contract_tc.cu).
//
// The kernel grid of ring pair (i, j) is sampled at longitudes x_k = pi (2k + f) / N with
// f = 1 when the shift fix applies to a pair of equal-length rings with different offsets
// (delta = +-pi/N) and f = 0 otherwise.  The samples are symmetric about x = 0, so the
// pair's Fourier coefficient including the offset phase is real:
//     rho_m(i,j) = sum_{k >= 0} c_k K(u(x_k)) cos(m x_k),   c_k = multiplicity(k) / N,
// and the contraction is c_m(i) = sum_j rho_m(i,j) w_j a_m(j) (w_j folded into a).
//
// k_taps evaluates c_k K(u) per sample (u is the squared chord of Eq. kernel_angle in the
// cancellation-free form 4[B cos^2(x/2) + A sin^2(x/2)]): the offset of u from its knot in FP64, the
// linear step from there in FP32.
#include <algorithm>

#include "fft_engine.cuh"

namespace arkcos {

namespace {

// Kernel samples K(u(x_k)) c_k / N.  u = 4 (B cos^2(x/2) + A sin^2(x/2)) is the haversine form
// of the squared chord, so the FP64 work per sample is the offset from the knot below it,
// u - u_t = 4B c2 + 4A s2 - u_t (two FMAs); the knot segment comes from an FP32 estimate of u
// (next to a knot the neighbouring segment's line differs by rounding only, the profile being
// continuous there) and the linear step runs in FP32 on tables pre-scaled by 1 / N.
//
// One launch serves every kernel of a call (blockIdx.y).  The pairs' slots are one array, so a
// warp takes a run of 128-slot tiles and a lane four slots of one pair, found by a binary search
// from the tile's first pair: most pairs have 6-24 samples, which left most lanes of a warp per
// pair idle (one 15' kernel at nside 2048 150 -> 40 us, at a degree of support 315 -> 268 us; 64
// kernels at nside 1024 in 64 launches 3.9 ms, now 0.55 ms).  FP64 bounds it (two FMAs and a
// conversion per sample at two per SM and clock: 30 us of the 40).  One CTA per SM, as each
// builds the knot tables with FP64 divisions (two of half the size: 50 us).
constexpr int kTapThreads = 1024;

__global__ void __launch_bounds__(kTapThreads) k_taps(const __grid_constant__ TapArgs a)
{
    extern __shared__ double tsm[];
    chain_allow_next();
    const int lane = threadIdx.x & 31;
    const KernDev &kb = a.kd[a.ksum > 0 ? a.kbase : blockIdx.y];  // whose pairs and slots are filled
    float *taps = a.taps[a.ksum > 0 ? a.kbase : blockIdx.y];
    const int slots = kb.toff[kb.npairs], tiles = (slots + 127) / 128;
    const int warps = gridDim.x * (kTapThreads / 32), per = (tiles + warps - 1) / warps;
    const int first = (blockIdx.x * (kTapThreads / 32) + (threadIdx.x >> 5)) * per, last = min(tiles, first + per);
    // last entry of tab[lo..hi] that is <= v (tab ascending, tab[lo] <= v)
    auto find = [](const int *__restrict__ tab, int lo, int hi, int v) {
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (__ldg(&tab[mid]) <= v) lo = mid;
            else hi = mid - 1;
        }
        return lo;
    };
    const int p0 = first < last ? find(kb.toff, 0, kb.npairs - 1, first * 128) : 0;
    const int nk = a.ksum > 0 ? a.ksum : 1;
    for (int q = 0; q < nk; ++q) {
        const KernDev &kd = a.kd[a.ksum > 0 ? q : blockIdx.y];
        const int T = kd.T;
        double *ut = tsm;                                  // [T] knots in u
        float *utf = reinterpret_cast<float *>(tsm + T);   // [T] the same in FP32
        float *f = utf + T, *slope = f + T, *span = slope + T;  // [T] profile / N, its slope, knot spacing
        const double invN = 1.0 / (double)a.N;
        if (q > 0) __syncthreads();
        for (int t = threadIdx.x; t < T; t += blockDim.x) {
            ut[t] = kd.ut[t];
            utf[t] = (float)kd.ut[t];
            f[t] = (float)(kd.knots[t] * invN);
            if (t < T - 1) {
                const double du = kd.ut[t + 1] - kd.ut[t];
                slope[t] = (float)((kd.knots[t + 1] - kd.knots[t]) / du * invN);
                span[t] = (float)du;
            }
        }
        __syncthreads();
        const float umaxf = (float)kd.umax;
        int p = p0;
        for (int tile = first; tile < last; ++tile) {
            const int s = tile * 128 + 4 * lane;
            // the pair of this lane's slots: at most 32 pairs with slots begin in a tile, but pairs
            // without any may lie between them, so the search ends at the last pair
            int hi = min(p + 32, kb.npairs - 1);
            if (__ldg(&kb.toff[hi + 1]) <= s) hi = kb.npairs - 1;
            p = find(kb.toff, p, hi, s);
            if (s < slots) {
                const int k0 = s - __ldg(&kb.toff[p]);
                int S = -1, fl = a.shift_fix ? __ldg(&kb.fl[p]) : 0;
                if (a.ksum > 0) {
                    // kernel q's own sample count for the pair's rings (i, j)
                    const int i = find(kb.pstart, 0, (int)kb.nrep - 1, p), j = __ldg(&kb.jlo[i]) + p - __ldg(&kb.pstart[i]);
                    const int jl = __ldg(&kd.jlo[i]);
                    if (j >= jl && j <= __ldg(&kd.jhi[i])) {
                        const int pq = __ldg(&kd.pstart[i]) + j - jl;
                        S = fl ? __ldg(&kd.S1[pq]) : __ldg(&kd.S0[pq]);
                    }
                } else {
                    S = fl ? __ldg(&kd.S1[p]) : __ldg(&kd.S0[p]);
                }
                const double A4 = 4.0 * __ldg(&kb.A[p]), B4 = 4.0 * __ldg(&kb.B[p]);
                const float A4f = (float)A4, B4f = (float)B4;
                float val[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int k = k0 + e;
                    val[e] = 0.f;
                    if (k <= S) {
                        const int t = 2 * k + fl;  // x_k / 2 = pi t / (2N)
                        const float uf = fminf(fmaf(B4f, __ldg(&a.s2f[a.N - t]), A4f * __ldg(&a.s2f[t])), umaxf);
                        const int sg = knot_segment_f(uf, utf, T, kd.gscale);
                        const double d = fma(B4, __ldg(&a.s2[a.N - t]), fma(A4, __ldg(&a.s2[t]), -ut[sg]));
                        // u is clamped to u_max: the last segment ends at its knot
                        const float df = fminf((float)d, span[sg]);
                        const float K = fmaf(df, slope[sg], f[sg]);
                        val[e] = (fl == 0 && (k == 0 || 2 * k == a.N)) ? K : 2.f * K;
                    }
                }
                float4 *out = reinterpret_cast<float4 *>(taps + s);
                if (a.ksum > 0) {
                    const float w = a.w[q];
                    float4 o = q > 0 ? *out : make_float4(0.f, 0.f, 0.f, 0.f);
                    if (k0 <= S) o = make_float4(fmaf(w, val[0], o.x), fmaf(w, val[1], o.y), fmaf(w, val[2], o.z), fmaf(w, val[3], o.w));
                    *out = o;
                } else {
                    *out = make_float4(val[0], val[1], val[2], val[3]);
                }
            }
            p = __shfl_sync(0xffffffffu, p, 31);
        }
    }
    chain_wait();
}

// Coefficients rho_m of the pairs next to the poles.  Those pairs have up to N/2 + 1 samples,
// so generating them inside the contraction would leave a few CTAs running long after the
// rest.  With x_k = pi (2k + f) / N,
//     rho_m = sum_k t_k cos(m x_k) = Re( exp(-i pi m f / N) T(m) ),  T(m) = sum_k t_k W_N^{mk},
// so for a power-of-two N one complex FFT of t_p + i t_{p+1} gives both pairs of a CTA:
// T_p(m) = (Z_m + conj Z_{N-m}) / 2 and T_{p+1}(m) = (Z_m - conj Z_{N-m}) / (2i).
template <int L>
struct PolarFft {
    const ContractArgs &a;
    float2 *buf;
    const float2 *tw;
    int kid, p0;
    __device__ void run()
    {
        constexpr int N = 1 << L;
        const KernDev &kd = a.kd[kid];
        const int np = kd.polar_pairs;
        int S[2], f[2];
        const float *tp[2];
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int p = p0 + q;
            S[q] = -1;
            f[q] = 0;
            tp[q] = a.taps[kid];
            if (p < np) {
                f[q] = a.shift_fix ? kd.fl[p] : 0;
                S[q] = f[q] ? kd.S1[p] : kd.S0[p];
                tp[q] = a.taps[kid] + kd.toff[p];
            }
        }
        auto ld = [&](int k) {
            return make_float2(k <= S[0] ? __ldg(&tp[0][k]) : 0.f, k <= S[1] ? __ldg(&tp[1][k]) : 0.f);
        };
        fft::dif<L>(buf, tw, ld);
        const fft::Smem<L> sm{buf};
        for (int m = threadIdx.x; m < a.NH; m += blockDim.x) {
            const float2 zm = sm(fft::digitrev<L>(m)), zn = sm(fft::digitrev<L>((N - m) & (N - 1)));
            const float2 t0 = make_float2(0.5f * (zm.x + zn.x), 0.5f * (zm.y - zn.y));
            const float2 t1 = make_float2(0.5f * (zm.y + zn.y), -0.5f * (zm.x - zn.x));
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                if (p0 + q >= np) continue;
                const float2 t = q ? t1 : t0;
                float r = t.x;  // f = 0
                if (f[q]) {
                    const float2 e = expipi_ratio(-m, N);  // exp(-i pi m / N)
                    r = e.x * t.x - e.y * t.y;
                }
                const_cast<float *>(a.prho[kid])[(int64_t)(p0 + q) * a.NH + m] = r;
            }
        }
    }
};

__global__ void __launch_bounds__(1024) k_polar_rho_fft(ContractArgs a, const float2 *tw, int logN)
{
    extern __shared__ float2 fbuf[];
    chain_allow_next();
    chain_wait();
    const int kid = blockIdx.y, p0 = 2 * blockIdx.x;
    if (p0 >= a.kd[kid].polar_pairs) return;
    switch (logN) {
    case 10: PolarFft<10>{a, fbuf, tw, kid, p0}.run(); break;
    case 11: PolarFft<11>{a, fbuf, tw, kid, p0}.run(); break;
    case 12: PolarFft<12>{a, fbuf, tw, kid, p0}.run(); break;
    case 13: PolarFft<13>{a, fbuf, tw, kid, p0}.run(); break;
    default: PolarFft<14>{a, fbuf, tw, kid, p0}.run(); break;
    }
}

// The same coefficients one thread per (pair, mode), for kernel grids without the FFT form.
__global__ void __launch_bounds__(256) k_polar_rho(const __grid_constant__ ContractArgs a, const float2 *__restrict__ cos2n)
{
    chain_allow_next();
    chain_wait();
    const int kid = blockIdx.z, p = blockIdx.y;
    const KernDev &kd = a.kd[kid];
    const int m = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= kd.polar_pairs || m >= a.NH) return;
    const int f = a.shift_fix ? kd.fl[p] : 0;
    const int S = f ? kd.S1[p] : kd.S0[p];
    const float4 *tp4 = reinterpret_cast<const float4 *>(a.taps[kid] + kd.toff[p]);
    const_cast<float *>(a.prho[kid])[(int64_t)p * a.NH + m] = gen_rho(tp4, S, f, m, a.N, cos2n);
}

}  // namespace

cudaError_t launch_polar_rho(const ContractArgs &a, int nk, int max_polar_pairs, const float2 *tw, int twM,
                             const float2 *cos2n, cudaStream_t st)
{
    if (max_polar_pairs <= 0 || nk <= 0) return cudaSuccess;
    int logN = 0;
    while ((1 << logN) < a.N) ++logN;
    if ((1 << logN) == a.N && logN >= 10 && logN <= 14 && a.N <= twM) {
        const size_t smem = (size_t)fft::buffer_words(a.N) * sizeof(float2);
        cudaError_t e = cudaFuncSetAttribute((const void *)k_polar_rho_fft,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        dim3 grid((max_polar_pairs + 1) / 2, nk);
        return launch_chained(k_polar_rho_fft, grid, a.N / 16, smem, st, true, 1, a, tw, logN);
    }
    dim3 grid((a.NH + 255) / 256, max_polar_pairs, nk);
    return launch_chained(k_polar_rho, grid, 256, 0, st, true, 1, a, cos2n);
}

cudaError_t launch_taps(const TapArgs &a, int nk, int64_t maxtaps, cudaStream_t st, bool after_prev)
{
    if (maxtaps <= 0) return cudaSuccess;
    int T = 0;
    for (int k = 0; k < std::max(nk, a.ksum); ++k) T = std::max(T, a.kd[k].T);
    const size_t smem = (size_t)T * (sizeof(double) + 4 * sizeof(float));
    cudaError_t e = cudaFuncSetAttribute((const void *)k_taps,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    // a warp per 128-slot tile while that fills at most one CTA per SM
    const int64_t want = (maxtaps + 128 * (kTapThreads / 32) - 1) / (128 * (kTapThreads / 32));
    const int blocks = (int)std::max<int64_t>(1, std::min<int64_t>(want, (device_sms() + nk - 1) / nk));
    return launch_chained(k_taps, dim3(blocks, nk), kTapThreads, smem, st, after_prev, 1, a);
}

}  // namespace arkcos
