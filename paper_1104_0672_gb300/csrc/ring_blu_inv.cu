// Inverse ring transforms by the split Bluestein convolutions of ring_blu.cuh, with the Sec. 4.3
// fold of the kernel-grid modes onto each ring's own frequencies.
#include "ring_blu.cuh"

namespace arkcos {

namespace {

using fft::cpair;
using ring::BluShape;
using ring::BluTables;

// One ring pair: see ring_blu.cuh.  The two half sequences of a ring each take every folded
// coefficient; at M = 4096 and for odd h the fold runs once per half sequence rather than keep one
// of them in shared memory.  Bounds and batching as the forward kernel; the inverse stage of 16
// nside-2048 maps 4.28 -> 3.54 ms (one long buffer per ring before), of six nside-4096 maps
// 10.4 -> 6.9 ms (four quarter transforms before).
//
// BOTH (M <= 2048, rings of even h): four teams run both half sequences at once, with one fold for
// both -- short transforms leave room for the four buffers (12 nside-474 maps, inverse stage
// 485 -> 290 us, 64 nside-1024 maps 3.99 -> 3.54 ms; at M = 2048, where it leaves one CTA per SM,
// eight nside-2048 maps 1.86 -> 1.83 ms).
template <int L, bool BOTH>
__global__ void __launch_bounds__(BluShape<L, BOTH>::kThreads, BluShape<L, BOTH>::kMinBlocks)
k_blu_inv(const __grid_constant__ FftInvArgs a)
{
    using Sh = BluShape<L, BOTH>;
    using namespace fft;
    constexpr int M = Sh::kM;
    // two buffers (four with BOTH: those of s = 1 behind those of s = 0) | twiddles | per-ring tables
    extern __shared__ float4 smem4[];
    if (!a.first) chain_allow_next();
    cpair *buf0 = reinterpret_cast<cpair *>(smem4), *buf1 = buf0 + Sh::kBuf;
    const int i = a.reps[blockIdx.x], i2 = a.R - 1 - i, n = a.rd.n[i], h = n / 2, hs = a.rd.hs[i], nyq = a.N / 2;
    float2 *twA = reinterpret_cast<float2 *>(buf0 + (BOTH ? 4 : 2) * Sh::kBuf), *twB = twA + M / 4;
    ring::blu_twiddles<L>(twA, a.tw);
    const BluTables tb = ring::blu_tables(twA + ring::blu_twiddle_words(M), h, n, +1);
    const int S = (h & 1) ? 1 : 2, l = h / S;
    const bool pair = i2 != i;
    const float wsc = a.weight ? a.rd.w[i] : 1.0f, inv = 0.5f / (float)M;
    const int team = threadIdx.x / Sh::kTeam, e = team & 1, tid = threadIdx.x % Sh::kTeam;
    const float2 *fb = a.rd.fb + a.rd.fboff[i] + e * M;
    if (a.first) {
        // the first class of the stage starts beside the end of the contraction; the next class
        // may only follow its coefficients
        chain_wait();
        chain_allow_next();
    }
    __syncthreads();
    const int bend = min(a.B, (int)(blockIdx.y + 1) * a.mchunk);
    for (int b = blockIdx.y * a.mchunk; b < bend; ++b) {
        const float2 *c1 = a.c + ((int64_t)b * a.R + i) * a.NH;
        const float2 *c2 = a.c + ((int64_t)b * a.R + i2) * a.NH;
        if (b + 1 < bend) {
            // the next map's coefficient rows of both rings into L2 (128-byte lines)
            const char *p1 = reinterpret_cast<const char *>(c1 + (int64_t)a.R * a.NH);
            const char *p2 = reinterpret_cast<const char *>(c2 + (int64_t)a.R * a.NH);
            const int lines = (a.NH * 8 + 127) / 128;
            for (int q = threadIdx.x; q < 2 * lines; q += Sh::kThreads)
                asm volatile("prefetch.global.L2 [%0];" ::"l"((q < lines ? p1 : p2) + 128 * (q % lines)));
        }
        // The folded coefficients X_m of ring and mirror (lanes) for modes m in [0, h]: the
        // kernel-grid modes m + t n and (t + 1) n - m up to N/2, conjugated in the second case,
        // each with the reverse phase of the first pixel (as folded_coeff).  All loads of a round
        // t are issued together; rings longer than N/2 have one.
        const int rounds = a.basic ? 1 : nyq / n + 1;
        auto folded = [&](const auto &mm, auto &x) {
            constexpr int NX = sizeof(mm) / sizeof(mm[0]);
            const float2 zero = make_float2(0.f, 0.f);
            float2 p1[NX], p2[NX], g1[NX], g2[NX];
#pragma unroll
            for (int u = 0; u < NX; ++u) p1[u] = p2[u] = g1[u] = g2[u] = zero;
#pragma unroll 1
            for (int t = 0; t < rounds; ++t) {
                const float sg = hs && (t & 1) ? -1.f : 1.f;
                float2 d1[NX], d2[NX], f1[NX], f2[NX];
#pragma unroll
                for (int u = 0; u < NX; ++u) {
                    const int m = mm[u] + t * n, mn = (t + 1) * n - mm[u];
                    const bool pos = m <= nyq, neg = mn <= nyq && !a.basic;
                    d1[u] = pos ? __ldg(&c1[m]) : zero;
                    d2[u] = pos ? __ldg(&c2[m]) : zero;
                    f1[u] = neg ? __ldg(&c1[mn]) : zero;
                    f2[u] = neg ? __ldg(&c2[mn]) : zero;
                }
#pragma unroll
                for (int u = 0; u < NX; ++u) {
                    const int m = mm[u] + t * n, mn = (t + 1) * n - mm[u];
                    const float wp = m == nyq && !a.basic ? 0.5f * sg : sg, wn = (mn == nyq ? 0.5f : 1.f) * (hs ? -sg : 1.f);
                    if (m == 0) d1[u].y = d2[u].y = 0.f;  // the m = 0 term of a real ring
                    p1[u] = make_float2(fmaf(wp, d1[u].x, p1[u].x), fmaf(wp, d1[u].y, p1[u].y));
                    p2[u] = make_float2(fmaf(wp, d2[u].x, p2[u].x), fmaf(wp, d2[u].y, p2[u].y));
                    g1[u] = make_float2(fmaf(wn, f1[u].x, g1[u].x), fmaf(wn, f1[u].y, g1[u].y));
                    g2[u] = make_float2(fmaf(wn, f2[u].x, g2[u].x), fmaf(wn, f2[u].y, g2[u].y));
                }
            }
#pragma unroll
            for (int u = 0; u < NX; ++u) {
                const float2 p = hs ? tb.ph(mm[u]) : make_float2(1.f, 0.f);
                const float2 d1 = cmulf(p1[u], p), e1 = cmulf(g1[u], cconjf(p));
                const float2 d2 = cmulf(p2[u], p), e2 = cmulf(g2[u], cconjf(p));
                x[u].re = make_float2(d1.x + e1.x, pair ? d2.x + e2.x : 0.f);
                x[u].im = make_float2(d1.y - e1.y, pair ? d2.y - e2.y : 0.f);
                if (a.basic && mm[u] == h) x[u].im = zero;  // the ring's Nyquist term, (d + conj d) / 2
            }
        };
        // Z_k and Z_{h-k} (unnormalised) from X_k and X_{h-k}: Z_k = E + i O, E = X_k + conj X_{h-k},
        // O = (X_k - conj X_{h-k}) exp(2 pi i k / n), Z_{h-k} = conj E + i conj O
        auto unsplit = [&](const cpair &xk, const cpair &xh, int k, cpair &zk, cpair &zh) {
            const float2 Er = caddf(xk.re, xh.re), Ei = csubf(xk.im, xh.im);
            const float2 Fr = csubf(xk.re, xh.re), Fi = caddf(xk.im, xh.im);
            const float2 v = tb.ph(2 * k), ws = bcast(wsc);
            const float2 Or = pfma(Fi, bcast(-v.y), pmul(Fr, bcast(v.x)));
            const float2 Oi = pfma(Fi, bcast(v.x), pmul(Fr, bcast(v.y)));
            zk = cpair{pmul(csubf(Er, Oi), ws), pmul(caddf(Ei, Or), ws)};
            zh = cpair{pmul(caddf(Er, Oi), ws), pmul(csubf(Or, Ei), ws)};
        };
        float2 *o1 = reinterpret_cast<float2 *>(a.map + (int64_t)b * a.npix + a.rd.poff[i]);
        float2 *o2 = reinterpret_cast<float2 *>(a.map + (int64_t)b * a.npix + a.rd.poff[i2]);
        for (int s = 0; s < (BOTH ? 1 : S); ++s) {
            // input k of the convolutions from the two halves p, q of the radix-2 step: p + q (s = 0),
            // p - q (s = 1) times the chirp, and W^k for the odd frequencies
            auto put1 = [&](cpair *b, int half, int k, const cpair &v) {
                const cpair x = e_mul(v, tb.chirp(half, k));
                b[ring::bsp(k)] = x;
                b[Sh::kBuf + ring::bsp(k)] = e_mul(x, __ldg(&a.tw[M + k]));
            };
            auto put = [&](int k, const cpair &p, const cpair &q) {
                if (BOTH) {
                    put1(buf0, 0, k, e_add(p, q));
                    put1(buf0 + 2 * Sh::kBuf, 1, k, e_sub(p, q));
                } else {
                    put1(buf0, s, k, s ? e_sub(p, q) : e_add(p, q));
                }
            };
            if (BOTH || S == 2) {
                for (int k = threadIdx.x; 2 * k <= l; k += Sh::kThreads) {
                    // Z_k, Z_{h-k} and Z_{l-k}, Z_{l+k}: inputs k and l - k
                    cpair x[4], z0, z1, z2, z3;
                    const int mm[4] = {k, h - k, l - k, l + k};
                    folded(mm, x);
                    unsplit(x[0], x[1], k, z0, z1);
                    if (k == 0) {
                        unsplit(x[2], x[2], l, z2, z3);
                        put(0, z0, z2);
                    } else {
                        unsplit(x[2], x[3], l - k, z2, z3);
                        put(k, z0, z3);
                        if (2 * k != l) put(l - k, z2, z1);
                    }
                }
            } else {
                for (int k = threadIdx.x; 2 * k <= l; k += Sh::kThreads) {
                    cpair x[2], z0, z1;
                    const int mm[2] = {k, h - k};
                    folded(mm, x);
                    unsplit(x[0], x[1], k, z0, z1);
                    put1(buf0, 0, k, z0);
                    if (k > 0) put1(buf0, 0, h - k, z1);
                }
            }
            for (int k = l + threadIdx.x; k < M; k += Sh::kThreads) {
                buf0[ring::bsp(k)] = buf1[ring::bsp(k)] = e_zero(cpair{});
                if (BOTH) buf0[2 * Sh::kBuf + ring::bsp(k)] = buf1[2 * Sh::kBuf + ring::bsp(k)] = e_zero(cpair{});
            }
            __syncthreads();
            cpair *x = buf0 + team * Sh::kBuf, v[16];
#pragma unroll
            for (int r = 0; r < 16; ++r) v[r] = x[ring::bsp(tid + r * Sh::kTeam)];
            ring::blu_convolve<L, true>(v, x, twA, twB, fb, tid, team);
            ring::blu_scale<L, true>(v, a.tw, l, tid, e, inv, [&](int t) { return tb.chirp0(t); });
#pragma unroll
            for (int r = 0; r < 16; ++r) x[ring::bsp(tid + r * Sh::kTeam)] = v[r];
            __syncthreads();
#pragma unroll 4
            for (int t = threadIdx.x; t < l; t += Sh::kThreads) {
                const cpair z = e_add(buf0[ring::bsp(t)], buf1[ring::bsp(t)]);
                const int o = BOTH ? 2 * t : S * t + s;
                o1[o] = make_float2(z.re.x, z.im.x);
                if (pair) o2[o] = make_float2(z.re.y, z.im.y);
                if (BOTH) {
                    const cpair w = e_add(buf0[2 * Sh::kBuf + ring::bsp(t)], buf1[2 * Sh::kBuf + ring::bsp(t)]);
                    o1[o + 1] = make_float2(w.re.x, w.im.x);
                    if (pair) o2[o + 1] = make_float2(w.re.y, w.im.y);
                }
            }
            __syncthreads();
        }
    }
    chain_wait();
}

template <int L, bool BOTH>
cudaError_t launch_inv(const FftInvArgs &a, int count, cudaStream_t st, bool after_prev)
{
    using Sh = BluShape<L, BOTH>;
    const size_t smem = ring::blu_smem_bytes(Sh::kM, a.tab, BOTH ? 4 : 2);
    cudaError_t e = cudaFuncSetAttribute((const void *)k_blu_inv<L, BOTH>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    return launch_chained(k_blu_inv<L, BOTH>, dim3(count, (a.B + a.mchunk - 1) / a.mchunk), Sh::kThreads, smem, st,
                          after_prev, 1, a);
}

}  // namespace

// even_h: every ring of the class has an even h
cudaError_t launch_blu_inv(const FftInvArgs &a, bool even_h, int count, cudaStream_t st, bool after_prev)
{
    if (count <= 0) return cudaSuccess;
    switch (a.logM) {
    case 9: return even_h ? launch_inv<9, true>(a, count, st, after_prev) : launch_inv<9, false>(a, count, st, after_prev);
    case 10: return even_h ? launch_inv<10, true>(a, count, st, after_prev) : launch_inv<10, false>(a, count, st, after_prev);
    case 11: return even_h ? launch_inv<11, true>(a, count, st, after_prev) : launch_inv<11, false>(a, count, st, after_prev);
    default: return launch_inv<12, false>(a, count, st, after_prev);
    }
}

}  // namespace arkcos
