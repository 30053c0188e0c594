// Ring transforms whose length is no power of two and too long for one warp-sized buffer, by
// Bluestein's chirp-z algorithm (1970), split so that the convolution buffers stay small.
//
// A ring pair (two mirror rings as the lanes of a cpair, ring_common.cuh) of n pixels is the
// h = n/2-point complex sequence z of each ring.  For even h one radix-2 step first gives S = 2
// sequences of l = h/2 points (odd h: S = 1, l = h):
//     Z_{2k+s}  = DFT_l( (z_t + (-1)^s z_{t+l}) e^{-i pi s t / l} )_k         (forward),
//     z_{2t+s}  = IDFT_l( (Z_k + (-1)^s Z_{k+l}) e^{+i pi s k / l} )_t        (inverse),
// each independent of the other.  Its l-point DFT is a convolution with the chirp of length
// >= 2l - 1.  Zero-padding to 2M >= 2l points leaves the upper half of the input empty and only
// the lower half of the output is wanted, so the 2M-point convolution is two independent
// M-point ones, the even and the odd frequencies (e = 0, 1; W = e^{-i pi / M}):
//     y_t = ( y0_t + W^{-t} y1_t ) / 2M,   y_e = M IDFT_M( fb_e DFT_M( x_t W^{e t} ) ).
// A team of M / 16 threads with 16 elements apiece runs each (two teams, or four where the CTA takes
// both half sequences at once): three radix passes forward,
// the product and three back, of which the inner two on each side stay within a warp.
// Against one 2h - 1-point buffer per ring the same rings need half the buffer (so two CTAs fit
// an SM where one did, and one's loads and barriers overlap the other's arithmetic), four
// exchanges through it instead of five and the shuffles between them, and about a fifth less
// arithmetic (no first radix-2 level on zeros).
#pragma once
#include "ring_common.cuh"

namespace arkcos {
namespace ring {

using fft::cpair;

// CTA of the class of M = 2^L: two teams of M / 16 threads, or four that run both half sequences
// at once; 128 registers per thread.
template <int L, bool BOTH = false>
struct BluShape {
    static constexpr int kM = 1 << L, kTeam = kM / 16, kThreads = (BOTH ? 4 : 2) * kTeam;
    static constexpr int kMinBlocks = 512 / kThreads;
    static constexpr int kBuf = fft::buffer_words(kM);
};

// Place of element p in a buffer: one pad element per 16 keeps every access of this file free of
// bank conflicts (the engine's second term, for digit-reversed reads, would add some here).
__device__ __forceinline__ constexpr int bsp(int p) { return p + (p >> 4); }

// Words of the twiddle tables of the two radix-16 passes.
__host__ __device__ constexpr int blu_twiddle_words(int M) { return M / 4 + M / 64; }

// Shared memory of a class of lengths l <= lmax: two buffers, the chirps of s = 0 and 1 and the
// phase table.
inline size_t blu_smem_bytes(int M, int tab, int buffers = 2)
{
    return buffers * (size_t)fft::buffer_words(M) * sizeof(cpair) + (size_t)(tab + blu_twiddle_words(M)) * sizeof(float2);
}

// Words of the per-ring tables: chirp exp(-+ i pi t^2 / l) for t <= l/2, the same of t (t + 1)
// (S = 2), phase exp(-+ i pi m / n) for m <= h/2.
__host__ __device__ inline int blu_table_words(int h)
{
    const int l = (h & 1) ? h : h / 2;
    return l / 2 + 1 + ((h & 1) ? 0 : l / 2 + 1) + h / 2 + 1;
}

struct BluTables {
    const float2 *ca, *cb, *p;
    int l, h, sgn;
    // exp(sgn i pi t^2 / l), t < l
    __device__ __forceinline__ float2 chirp0(int t) const { return chirp_at(ca, t, l); }
    // exp(sgn i pi t (t + 1) / l), t < l: the value at l - 1 - t times (-1)^(l - 1)
    __device__ __forceinline__ float2 chirp1(int t) const
    {
        if (2 * t + 1 <= l) return cb[t];
        const float2 c = cb[l - 1 - t];
        return (l & 1) ? c : make_float2(-c.x, -c.y);
    }
    __device__ __forceinline__ float2 chirp(int s, int t) const { return s ? chirp1(t) : chirp0(t); }
    // exp(sgn i pi m / n), m <= h = n/2: past h/2 it is (sgn i) conj of the value at h - m
    __device__ __forceinline__ float2 ph(int m) const
    {
        if (2 * m <= h) return p[m];
        const float2 c = p[h - m];
        return sgn > 0 ? make_float2(c.y, c.x) : make_float2(-c.y, -c.x);
    }
};

// Copies the twiddles of the radix-16 passes to words[] (M / 4, then M / 64).
template <int L>
__device__ __forceinline__ void blu_twiddles(float2 *words, const float2 *__restrict__ tw)
{
    constexpr int M = 1 << L;
    for (int j = threadIdx.x; j < M / 4; j += blockDim.x) words[j] = __ldg(&tw[M / 2 + j]);
    for (int j = threadIdx.x; j < M / 64; j += blockDim.x) words[M / 4 + j] = __ldg(&tw[M / 32 + j]);
}

// Builds the tables in words[] (no barrier at the end).
__device__ __forceinline__ BluTables blu_tables(float2 *words, int h, int n, int sgn)
{
    const int l = (h & 1) ? h : h / 2;
    float2 *ca = words, *cb = ca + l / 2 + 1, *p = (h & 1) ? cb : cb + l / 2 + 1;
    for (int t = threadIdx.x; 2 * t <= l; t += blockDim.x) {
        ca[t] = expipi_ratio(sgn * t * t, l);
        if (!(h & 1)) cb[t] = expipi_ratio(sgn * t * (t + 1), l);
    }
    for (int m = threadIdx.x; 2 * m <= h; m += blockDim.x) p[m] = expipi_ratio(sgn * m, n);
    return BluTables{ca, cb, p, l, h, sgn};
}

// Barrier of the T threads of team e < 4 (a warp when T = 32).
template <int T>
__device__ __forceinline__ void team_sync(int e)
{
    if constexpr (T <= 32) __syncwarp();
    else if (e == 0) asm volatile("bar.sync 1, %0;" ::"n"(T) : "memory");
    else if (e == 1) asm volatile("bar.sync 2, %0;" ::"n"(T) : "memory");
    else if (e == 2) asm volatile("bar.sync 3, %0;" ::"n"(T) : "memory");
    else asm volatile("bar.sync 4, %0;" ::"n"(T) : "memory");
}

// v[k] *= w^k for k = 1..15 (conjugated when CONJ) from w, w^2, w^3 and w^4, as fft::twiddle.
template <bool CONJ>
__device__ __forceinline__ void twiddle16(cpair (&v)[16], float2 w1, float2 w2, float2 w3, float2 w4)
{
    if (CONJ) {
        w1.y = -w1.y;
        w2.y = -w2.y;
        w3.y = -w3.y;
        w4.y = -w4.y;
    }
    v[1] = fft::e_mul(v[1], w1);
    v[2] = fft::e_mul(v[2], w2);
    v[3] = fft::e_mul(v[3], w3);
    float2 wa = w4;
#pragma unroll
    for (int a = 4; a < 16; a += 4) {
        if (a > 4) wa = cmulf(wa, w4);
        v[a] = fft::e_mul(v[a], wa);
        v[a + 1] = fft::e_mul(v[a + 1], cmulf(wa, w1));
        v[a + 2] = fft::e_mul(v[a + 2], cmulf(wa, w2));
        v[a + 3] = fft::e_mul(v[a + 3], cmulf(wa, w3));
    }
}

// One team's M-point circular convolution (times M) of v, v[r] = input tid + r T of the thread,
// with the sequence of spectrum fb (DIF order, conjugated when CONJ); the result in natural order
// in v (same places), through the buffer x.  twA and twB: exp(-2 pi i j / M) for j < M / 4 and
// exp(-2 pi i j / (M / 16)) for j < M / 64, in shared memory.  fb holds the pairs of a thread's 16 values M / 16
// apart, so that a warp reads them in whole lines.  The passes of strides below M / 16 run on blocks
// of M / 16 elements that a run of neighbouring lanes holds, so only the two exchanges across the
// buffer need a team barrier.
template <int L, bool CONJ>
__device__ __forceinline__ void blu_convolve(cpair (&v)[16], cpair *x, const float2 *twA, const float2 *twB,
                                             const float2 *__restrict__ fb, int tid, int e)
{
    using G = fft::Geo<L>;
    static_assert(G::NP == 3, "three passes: 2^9 <= M <= 2^12");
    constexpr int T = G::M / 16, S1 = G::S(1), st0 = T + T / 16;
    fft::dft<16, false>(v);
    twiddle16<false>(v, twA[tid], twA[2 * tid], twA[3 * tid], twA[4 * tid]);
    cpair *p0 = x + bsp(tid);
#pragma unroll
    for (int r = 0; r < 16; ++r) p0[r * st0] = v[r];
    team_sync<T>(e);
    const int n2 = tid & (S1 - 1), base = (tid - n2) * 16 + n2;
#pragma unroll
    for (int r = 0; r < 16; ++r) v[r] = x[bsp(base + r * S1)];
    fft::dft<16, false>(v);
    twiddle16<false>(v, twB[n2], twB[2 * n2], twB[3 * n2], twB[4 * n2]);
#pragma unroll
    for (int r = 0; r < 16; ++r) x[bsp(base + r * S1)] = v[r];
    {
        constexpr int R = 1 << G::LAST;
        cpair *p1 = x + bsp(16 * tid);  // 16 consecutive elements share their padding
        float4 f[8];                      // the spectrum, on its way while the lanes exchange
        const float4 *f4 = reinterpret_cast<const float4 *>(fb) + tid;
#pragma unroll
        for (int r = 0; r < 8; ++r) f[r] = __ldg(&f4[r * T]);
        __syncwarp();
#pragma unroll
        for (int r = 0; r < 16; ++r) v[r] = p1[r];
#pragma unroll
        for (int q = 0; q < 16 / R; ++q) {
            cpair w[R];
#pragma unroll
            for (int r = 0; r < R; ++r) w[r] = v[q * R + r];
            fft::dft<R, false>(w);
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const float4 &g = f[(q * R + r) / 2];
                const float2 c = (r & 1) ? make_float2(g.z, g.w) : make_float2(g.x, g.y);
                w[r] = fft::e_mul(w[r], CONJ ? cconjf(c) : c);
            }
            fft::dft<R, true>(w);
#pragma unroll
            for (int r = 0; r < R; ++r) v[q * R + r] = w[r];
        }
#pragma unroll
        for (int r = 0; r < 16; ++r) p1[r] = v[r];
    }
    __syncwarp();
#pragma unroll
    for (int r = 0; r < 16; ++r) v[r] = x[bsp(base + r * S1)];
    twiddle16<true>(v, twB[n2], twB[2 * n2], twB[3 * n2], twB[4 * n2]);
    fft::dft<16, true>(v);
#pragma unroll
    for (int r = 0; r < 16; ++r) x[bsp(base + r * S1)] = v[r];
    team_sync<T>(e);
#pragma unroll
    for (int r = 0; r < 16; ++r) v[r] = p0[r * st0];
    twiddle16<true>(v, twA[tid], twA[2 * tid], twA[3 * tid], twA[4 * tid]);
    fft::dft<16, true>(v);
}

// Factors of the thread's elements t = tid + r T: c(t) = table(t) times sc, times W^t (conjugated
// after the convolution) for the odd frequencies; 1 past the ring's l points.
template <int L, bool POST, class C>
__device__ __forceinline__ void blu_scale(cpair (&v)[16], const float2 *__restrict__ tw, int l, int tid, int e, float sc,
                                          C table)
{
    constexpr int M = 1 << L, T = M / 16;
#pragma unroll
    for (int h = 0; h < 16; h += 4) {
        float2 w[4];
        if (e) {
#pragma unroll
            for (int r = 0; r < 4; ++r) w[r] = __ldg(&tw[M + tid + (h + r) * T]);
        }
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const int t = tid + (h + r) * T;
            float2 c = table(t < l ? t : 0);
            if (POST) c = cscalef(c, sc);
            if (e) c = cmulf(c, POST ? cconjf(w[r]) : w[r]);
            v[h + r] = fft::e_mul(v[h + r], c);
        }
    }
}

}  // namespace ring
}  // namespace arkcos
