// Forward ring transforms by the split Bluestein convolutions of ring_blu.cuh, and the chirp
// spectra they use.
#include "ring_blu.cuh"

namespace arkcos {

namespace {

using fft::cpair;
using ring::BluShape;
using ring::BluTables;

// The two spectra (even and odd frequencies of the 2M-point DFT, each in DIF order of M points,
// laid out as blu_convolve reads it) of the Bluestein sequence b_k = exp(+i pi k^2 / l), |k| < l, circular in 2M: once per grid.
template <int L>
__global__ void __launch_bounds__(BluShape<L>::kTeam) k_blu_spectra(RingDev rd, const int *reps, const float2 *tw,
                                                                    float2 *fb_all)
{
    extern __shared__ float2 cbuf[];
    constexpr int M = 1 << L;
    const int j = reps[blockIdx.x], h = rd.n[j] / 2, l = (h & 1) ? h : h / 2;
    auto b = [&](int k) {  // k < 2M
        const int kk = k < l ? k : (k > 2 * M - l ? 2 * M - k : -1);
        return kk < 0 ? make_float2(0.f, 0.f) : expipi_ratio(kk * kk, l);
    };
    for (int e = 0; e < 2; ++e) {
        fft::dif<L>(cbuf, tw, [&](int t) {
            const float2 u = b(t), v = b(t + M);
            return e ? cmulf(csubf(u, v), __ldg(&tw[M + t])) : caddf(u, v);
        });
        float2 *fb = fb_all + rd.fboff[j] + e * M;
        const fft::Smem<L> sm{cbuf};
        for (int p = threadIdx.x; p < M; p += blockDim.x)
            fb[2 * ((p >> 1 & 7) * (M / 16) + (p >> 4)) + (p & 1)] = sm(p);
        __syncthreads();
    }
}

// One ring pair: see ring_blu.cuh.  What bounds it: arithmetic and exchanges at 16 warps per SM
// (registers); the pixels, the next pass's twiddles and the chirp spectrum are asked for in whole
// batches, as latency, not arithmetic, took most of the time before.  The forward stage of 16
// nside-2048 maps 3.71 -> 3.06 ms (one long buffer per ring before), of six nside-4096 maps (rings
// up to 16380 pixels, four quarter transforms before) 7.8 -> 6.1 ms.
//
// BOTH (M <= 1024, rings of even h): four teams run both half sequences at once and the pixels are
// loaded once (12 nside-474 maps, forward stage 345 -> 274 us; at M = 2048, one CTA per SM, slower:
// eight nside-2048 maps 1.58 -> 1.62 ms).
template <int L, bool BOTH>
__global__ void __launch_bounds__(BluShape<L, BOTH>::kThreads, BluShape<L, BOTH>::kMinBlocks)
k_blu_fwd(const __grid_constant__ FftFwdArgs a)
{
    using Sh = BluShape<L, BOTH>;
    using namespace fft;
    constexpr int M = Sh::kM;
    // two buffers (four with BOTH: those of s = 1 behind those of s = 0) | twiddles | per-ring tables
    extern __shared__ float4 smem4[];
    chain_allow_next();
    cpair *buf0 = reinterpret_cast<cpair *>(smem4), *buf1 = buf0 + Sh::kBuf;
    const int j = a.reps[blockIdx.x], j2 = a.R - 1 - j, n = a.rd.n[j], h = n / 2, hs = a.rd.hs[j];
    float2 *twA = reinterpret_cast<float2 *>(buf0 + (BOTH ? 4 : 2) * Sh::kBuf), *twB = twA + M / 4;
    ring::blu_twiddles<L>(twA, a.tw);
    const BluTables tb = ring::blu_tables(twA + ring::blu_twiddle_words(M), h, n, -1);
    const int S = (h & 1) ? 1 : 2, l = h / S;
    const bool pair = j2 != j;
    const float wsc = a.weight ? a.rd.w[j] : 1.0f;
    const int team = threadIdx.x / Sh::kTeam, e = team & 1, tid = threadIdx.x % Sh::kTeam;
    const float2 *fb = a.rd.fb + a.rd.fboff[j] + e * M;
    const float inv = 0.5f / (float)M;
    __syncthreads();
    const int bend = min(a.B, (int)(blockIdx.y + 1) * a.mchunk);
    for (int b = blockIdx.y * a.mchunk; b < bend; ++b) {
        const float2 *m1 = reinterpret_cast<const float2 *>(a.map + (int64_t)b * a.npix + a.rd.poff[j]);
        const float2 *m2 = reinterpret_cast<const float2 *>(a.map + (int64_t)b * a.npix + a.rd.poff[j2]);
        if (b + 1 < bend) {
            // the next map's pixels of both rings into L2 while this map is transformed
            const char *p1 = reinterpret_cast<const char *>(m1 + a.npix / 2);
            const char *p2 = reinterpret_cast<const char *>(m2 + a.npix / 2);
            const int lines = (n * 4 + 127) / 128;
            for (int q = threadIdx.x; q < 2 * lines; q += Sh::kThreads)
                asm volatile("prefetch.global.L2 [%0];" ::"l"((q < lines ? p1 : p2) + 128 * (q % lines)));
        }
        for (int s0 = 0; s0 < (BOTH ? 1 : S); ++s0) {
            // input of the two convolutions: the radix-2 step and the chirp (with W^t for the odd
            // frequencies); z_t = x_2t + i x_2t+1 of both rings.  Both teams fill both buffers, the
            // loads of several elements in flight (each team loading its own elements into registers
            // one by one took twice as long as its transforms).
            const float2 *r1 = m1 + (h - l), *r2 = m2 + (h - l);
            const float f1 = !BOTH && S == 1 ? 0.f : (s0 ? -1.f : 1.f), g0 = pair ? 1.f : 0.f, g1 = pair ? f1 : 0.f;
            constexpr int kFill = M / Sh::kThreads;  // elements per thread
            float2 u0[kFill], w0[kFill], u1[kFill], w1[kFill], wt[kFill];
#pragma unroll
            for (int q = 0; q < kFill; ++q) {
                const int t = threadIdx.x + q * Sh::kThreads;
                wt[q] = __ldg(&a.tw[M + t]);
                u0[q] = w0[q] = u1[q] = w1[q] = make_float2(0.f, 0.f);
                if (t < l) {
                    u0[q] = __ldg(&m1[t]);
                    w0[q] = __ldg(&m2[t]);
                    u1[q] = __ldg(&r1[t]);
                    w1[q] = __ldg(&r2[t]);
                }
            }
#pragma unroll
            for (int q = 0; q < kFill; ++q) {
                const int t = threadIdx.x + q * Sh::kThreads;
                auto put = [&](cpair *b, int half, float c1, float d1) {
                    const cpair z{make_float2(fmaf(c1, u1[q].x, u0[q].x), fmaf(d1, w1[q].x, g0 * w0[q].x)),
                                  make_float2(fmaf(c1, u1[q].y, u0[q].y), fmaf(d1, w1[q].y, g0 * w0[q].y))};
                    const cpair z0 = e_mul(z, tb.chirp(half, t < l ? t : 0));  // (zero past the l points)
                    b[ring::bsp(t)] = z0;
                    b[Sh::kBuf + ring::bsp(t)] = e_mul(z0, wt[q]);
                };
                put(buf0, s0, f1, g1);
                if (BOTH) put(buf0 + 2 * Sh::kBuf, 1, -f1, -g1);
            }
            __syncthreads();
            cpair *x = buf0 + team * Sh::kBuf, v[16];
#pragma unroll
            for (int r = 0; r < 16; ++r) v[r] = x[ring::bsp(tid + r * Sh::kTeam)];
            ring::blu_convolve<L, false>(v, x, twA, twB, fb, tid, team);
            ring::blu_scale<L, true>(v, a.tw, l, tid, e, inv, [&](int t) { return tb.chirp0(t); });
#pragma unroll
            for (int r = 0; r < 16; ++r) x[ring::bsp(tid + r * Sh::kTeam)] = v[r];
            __syncthreads();
            for (int s = s0; s < (BOTH ? 2 : s0 + 1); ++s) {
                // DFT value k' (mode S k' + s of the h-point DFT)
                const cpair *bs = buf0 + (BOTH ? 2 * s : 0) * Sh::kBuf;
                auto y = [&](int k) { return e_add(bs[ring::bsp(k)], bs[Sh::kBuf + ring::bsp(k)]); };
                // X_k and X_{h-k} of both rings from Z_k and Z_{h-k}, times first-pixel phase and weight
                // (as FwdCta::split)
                auto split = [&](const cpair &zk, const cpair &zh, int k, cpair &xk, cpair &xhk) {
                    const float2 Er = pmul(bcast(0.5f), caddf(zk.re, zh.re)), Ei = pmul(bcast(0.5f), csubf(zk.im, zh.im));
                    const float2 Or = pmul(bcast(0.5f), caddf(zk.im, zh.im)), Oi = pmul(bcast(-0.5f), csubf(zk.re, zh.re));
                    const float2 w = tb.ph(2 * k);
                    const float2 Wr = pfma(Oi, bcast(-w.y), pmul(Or, bcast(w.x)));
                    const float2 Wi = pfma(Or, bcast(w.y), pmul(Oi, bcast(w.x)));
                    const cpair a0{caddf(Er, Wr), caddf(Ei, Wi)}, a1{csubf(Er, Wr), csubf(Wi, Ei)};
                    const float2 one = make_float2(1.f, 0.f);
                    xk = e_mul(a0, cscalef(hs ? tb.ph(k) : one, wsc));
                    xhk = e_mul(a1, cscalef(hs ? tb.ph(h - k) : one, wsc));
                };
                auto out4 = [&](const cpair &x) {
                    const float4 v = ring::lanes4(x);
                    return pair ? v : make_float4(v.x, v.y, v.x, v.y);
                };
                // the partner h - k of mode k = S q + s has index l - q (s = 0) or l - 1 - q (s = 1)
                const int last = s ? l - 1 : l;
                float2 *s1 = a.spec + (int64_t)b * a.nspec + a.rd.soff[j], *s2 = a.spec + (int64_t)b * a.nspec + a.rd.soff[j2];
                float4 *o4 = a.spec4 + ((int64_t)b * a.nrep + j) * a.NH;
                // every kernel-grid mode m <= N/2 that folds onto mode k <= h: the periodic extension
                // a_{k + qn} = exp(-i q n phi0) a_k and, conjugated, a_{(q+1)n - k} (ENHANCED), or a_k alone,
                // halved at the ring's Nyquist frequency (BASIC)
                auto extend = [&](int k, const cpair &x) {
                    const float4 v = out4(x);
                    const float first = a.basic && k == h && n < a.N ? 0.5f : 1.f;
                    for (int q = 0; k + q * n < a.NH; ++q) {
                        const float sg = a.basic && q > 0 ? 0.f : (hs && (q & 1)) ? -first : first;
                        o4[k + q * n] = make_float4(sg * v.x, sg * v.y, sg * v.z, sg * v.w);
                        const int m = (q + 1) * n - k;
                        if (k > 0 && k < h && m < a.NH) {
                            const float sn = a.basic ? 0.f : (hs && !(q & 1)) ? -1.f : 1.f;
                            o4[m] = make_float4(sn * v.x, -sn * v.y, sn * v.z, -sn * v.w);
                        }
                    }
                };
                for (int q = threadIdx.x; 2 * q <= last; q += Sh::kThreads) {
                    const int qp = last - q, k = S * q + s, kp = h - k;
                    cpair xk, xp;
                    const cpair zk = y(q), zp = q == 0 && s == 0 ? zk : y(qp);
                    split(zk, zp, k, xk, xp);
                    if (a.ext4) {
                        extend(k, xk);
                        if (q != qp) extend(kp, xp);
                    } else {
                        const float4 u = ring::lanes4(xk), v = ring::lanes4(xp);
                        s1[k] = make_float2(u.x, u.y);
                        if (pair) s2[k] = make_float2(u.z, u.w);
                        if (q != qp) {
                            s1[kp] = make_float2(v.x, v.y);
                            if (pair) s2[kp] = make_float2(v.z, v.w);
                        }
                    }
                }
            }
            __syncthreads();
        }
    }
    chain_wait();
}

template <int L, bool BOTH>
cudaError_t launch_fwd(const FftFwdArgs &a, int count, cudaStream_t st, bool after_prev)
{
    using Sh = BluShape<L, BOTH>;
    const size_t smem = ring::blu_smem_bytes(Sh::kM, a.tab, BOTH ? 4 : 2);
    cudaError_t e = cudaFuncSetAttribute((const void *)k_blu_fwd<L, BOTH>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    return launch_chained(k_blu_fwd<L, BOTH>, dim3(count, (a.B + a.mchunk - 1) / a.mchunk), Sh::kThreads, smem, st,
                          after_prev, 1, a);
}

template <int L>
cudaError_t launch_spectra(const FftFwdArgs &a, float2 *fb, int count, cudaStream_t st)
{
    k_blu_spectra<L><<<count, BluShape<L>::kTeam, fft::buffer_words(1 << L) * sizeof(float2), st>>>(a.rd, a.reps, a.tw, fb);
    return cudaGetLastError();
}

}  // namespace

int blu_table_words(int h) { return ring::blu_table_words(h); }
size_t blu_smem_bytes(int M, int tab) { return ring::blu_smem_bytes(M, tab); }

cudaError_t launch_blu_spectra(const FftFwdArgs &a, float2 *fb, int count, cudaStream_t st)
{
    if (count <= 0) return cudaSuccess;
    switch (a.logM) {
    case 9: return launch_spectra<9>(a, fb, count, st);
    case 10: return launch_spectra<10>(a, fb, count, st);
    case 11: return launch_spectra<11>(a, fb, count, st);
    default: return launch_spectra<12>(a, fb, count, st);
    }
}

// even_h: every ring of the class has an even h
cudaError_t launch_blu_fwd(const FftFwdArgs &a, bool even_h, int count, cudaStream_t st, bool after_prev)
{
    if (count <= 0) return cudaSuccess;
    switch (a.logM) {
    case 9: return even_h ? launch_fwd<9, true>(a, count, st, after_prev) : launch_fwd<9, false>(a, count, st, after_prev);
    case 10: return even_h ? launch_fwd<10, true>(a, count, st, after_prev) : launch_fwd<10, false>(a, count, st, after_prev);
    case 11: return launch_fwd<11, false>(a, count, st, after_prev);
    default: return launch_fwd<12, false>(a, count, st, after_prev);
    }
}

}  // namespace arkcos
