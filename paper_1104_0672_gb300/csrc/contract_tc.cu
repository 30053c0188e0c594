// Tensor-core form of the ring-pair coefficient generation (3xTF32 on tcgen05), fused with
// the band contraction; and the tensor-core knot-gradient projection of the backward pass.
//
// For a block of RB (8 or 16) representative output rings x 128 modes the coefficients are a
// dense product  rho[m, col] = sum_k C_f[m, k] T[k, col]  with C_f[m, k] = cos(pi m (2k + f) / N)
// (f = the pair's sample offset, see contract.cu) and T the FP32 kernel samples.  The CTA
// stages C (cosines in FP64, split into TF32 hi + lo parts of together 22 to 23 bits, prepared per grid) and T (split
// into hi + lo on the fly) in shared memory, a pass of 16 samples at a time with the next pass's
// loads in flight, and one thread issues tcgen05.mma kind::tf32 with the accumulator in tensor
// memory:
//     D = C_hi T_hi + C_hi T_lo + C_lo T_hi      (3xTF32, FP32 accumulation).
// The plain FP32 form (F32) is the same kernel with the sums on the CUDA cores: the samples in
// shared memory, a thread's cosine times broadcast samples into 64 register sums by packed FMAs,
// and the coefficients stored to tensor memory (it replaces one recurrence per pair and mode; one
// nside-2048 map 2.52 -> 0.98 ms, six nside-4096 maps of an 8' support 15.0 -> 7.9 ms).
// The rings of the block go in groups of G (2 or 4) consecutive rings; slot u of ring l holds
// the pair of that ring with input ring jlo(first ring of its group) + u (zero when that ring is
// outside its band), so the rings of a group index one common run of 32 input rings.  On the
// equatorial belt the sample offset f alternates with the parity of i + j, so the 32 RB columns
// are split by the parity of u + l into two tiles: there each tile has one f, and one pass
// serves both with a cosine operand each (no products with the other offset's zeros); tiles
// that hold both offsets (blocks at the edge of the belt) take a pass for each.
// Each thread (mode, group) reads slices of its G x 32 coefficients of D with tcgen05.ld and
// contracts every staged input coefficient into all G rings' outputs.
//
// Bands wider than 32 rings take the 32 slots as a window that moves along the band, and pairs
// of more than 128 samples (untabulated rings next to the poles) are generated 128 samples at a
// time: the outputs are linear in the coefficients, so every (window, run of 128 samples) is
// generated, contracted and added in FP32.  No sum on the tensor core is longer than 128
// samples (its accumulator's additions do not round to nearest), and no table grows with the
// support.
//
// What bounds it: with many maps the contraction on the CUDA cores (0.155 ms per nside-2048
// map, issue); with one map per kernel the generation (tap loads, splits, one pass's round
// trip), which is why a pass stages no more samples and cosines than its K-steps read, serves
// both offsets and overlaps the copy of the first map: 64 nside-1024 maps with a beam each
// 9.05 -> 7.22 ms against passes of 32 samples per offset, one nside-2048 map 0.67 -> 0.51 ms,
// 16 maps with one beam 2.99 -> 2.94 ms.  Wide bands, one nside-2048 map at a degree of support
// (about 105 rings): 4.5 ms, against 77.1 ms generated and contracted on the CUDA cores.
// Waits on the MMA completion barriers are bounded: on expiry the kernel records an error
// (reported by arkcos_sync_status) and still frees its tensor memory.
#include <stdint.h>

#include <algorithm>

#include "tcgen05.cuh"

namespace arkcos {

__device__ int g_tc_error = 0;

namespace {

using namespace tc;

constexpr int kTcModes = 128;          // M of the MMA: modes per CTA (TMEM lanes)
constexpr int kTcBand = 32;            // input-ring slots per group (columns per ring)
constexpr int kTcK = 16;               // samples per pass (2 MMA K-steps of 8)
constexpr int kF32K = 32;              // samples per pass of the plain FP32 form
constexpr int kTcRun = 128;            // samples per generated run (longest tensor-core sum)
constexpr uint32_t kTcSBO = 4 * kLBO;  // row octets of an operand of 16 samples

// A CTA takes RB representative output rings (8 or 16) x kTcModes modes: RB / G ring groups
// of G (2 or 4) consecutive rings, one warp per group and lane quarter; RB x 32 tensor-memory
// columns in two tiles.  A stage holds the cosines of both tiles and the samples of every
// column for one pass; RB = 16 (one CTA per SM) has two stages, so that a pass is staged while
// the MMAs of the one before it run, RB = 8 has one (two CTAs per SM overlap instead).
template <int RB, int G>
struct TcShape {
    static constexpr int kGroups = RB / G, kThreads = kTcModes * kGroups;
    static constexpr int kN = RB * kTcBand, kTile = kN / 2, kTmemCols = kN;
    static constexpr uint32_t kA = kTcModes / 8 * kTcSBO;  // one cosine operand (hi or lo)
    static constexpr uint32_t kB = kN / 8 * kTcSBO;        // the samples (hi or lo) of every column
    static constexpr uint32_t kStage = 4 * kA + 2 * kB;
    static_assert((uint32_t)kF32K * kN * sizeof(float) <= kStage, "the FP32 form's samples fit a stage");
    static constexpr int kStages = RB / 8;
};

// (a, b) += c v, v as two packed pairs
__device__ __forceinline__ void fma4(float2 &a, float2 &b, float c, const float4 &v)
{
    const float2 cc = make_float2(c, c);
    a = __ffma2_rn(cc, make_float2(v.x, v.y), a);
    b = __ffma2_rn(cc, make_float2(v.z, v.w), b);
}

// acc += c v for the four lanes of v, as two packed two-lane FMAs (each lane rounds as fmaf)
__device__ __forceinline__ void fma4(float4 &acc, float c, const float4 &v)
{
    const float2 cc = make_float2(c, c);
    const float2 lo = __ffma2_rn(cc, make_float2(v.x, v.y), make_float2(acc.x, acc.y));
    const float2 hi = __ffma2_rn(cc, make_float2(v.z, v.w), make_float2(acc.z, acc.w));
    acc = make_float4(lo.x, lo.y, hi.x, hi.y);
}

// Issue the copies of input rings [j0, j0 + rows) x kTcModes modes from m0 (zero past N/2) into
// shared memory, raw paired rows: a thread keeps its mode.
template <int THREADS>
__device__ __forceinline__ void stage_rows(float4 *dst, const float4 *__restrict__ sp4b, int j0, int rows, int m0,
                                           int R, int NH)
{
    const int c = threadIdx.x % kTcModes, mm = m0 + c;
    const bool mv = mm < NH;
    if (m0 + (c & ~31) >= NH) rows = 0;  // nobody reads this warp's modes
    const float4 *src = sp4b + (mv ? mm : 0);
    for (int jj = threadIdx.x / kTcModes; jj < rows; jj += THREADS / kTcModes) {
        const int j = j0 + jj;
        cp_async16(&dst[jj * kTcModes + c], src + (mv ? (int64_t)min(j, R - 1 - j) * NH : 0), mv ? 16 : 0);
    }
    cp_async_commit();
}

// SLOTS: slots that the groups' bands reach (the plain form of narrow bands has one for 16 of the 32)
template <int RB, int G, bool WIDE, bool F32, int SLOTS = kTcBand>
__global__ void __launch_bounds__(TcShape<RB, G>::kThreads, 16 / RB)
k_contract_tc(ContractArgs a, const float *__restrict__ ctab, const float2 *__restrict__ cos2n, int nkc_tab, int srows,
              int nbuf, uint32_t rows0, uint32_t ctl)
{
    using Sh = TcShape<RB, G>;
    constexpr int kTcN = Sh::kN, kTile = Sh::kTile, NY = SLOTS / 8;  // NY: quads of columns per ring and tile
    static_assert(SLOTS == kTcBand || (F32 && !WIDE));
    extern __shared__ __align__(1024) unsigned char smem[];
    // per stage: cosines hi | lo of tile 0, of tile 1, samples hi | lo of every column; then
    // reused for the staged spectra; at ctl the MMA barriers and the tensor-memory address
    uint64_t *mbar = reinterpret_cast<uint64_t *>(smem + ctl);
    uint32_t *tslot = reinterpret_cast<uint32_t *>(smem + ctl + 16);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int q4 = warp & 3, grp = warp >> 2;  // lane quarter of TMEM, ring group
    const int mrow = q4 * 32 + lane;           // mode within the block
    const int m0 = blockIdx.x * kTcModes, m = m0 + mrow;
    const bool mv = m < a.NH;
    const int r0 = blockIdx.y * RB;
    const int nr = min(RB, a.nrep - r0);
    if (a.basic) {
        // BASIC variant: output ring i keeps only its modes m <= n_i / 2 (Sec. 4.1 truncation;
        // the inverse transform reads no others), so a block of modes above the Nyquist
        // frequency of every ring of the block (and of their mirrors) has nothing to compute
        int nmax = 0;
        for (int t = 0; t < nr; ++t) nmax = max(nmax, __ldg(&a.rd.n[r0 + t]));
        if (m0 > nmax / 2) {
            chain_wait();
            return;
        }
    }
    const int b0 = blockIdx.z * a.maps_per_chunk;
    const int b1 = min(a.B, b0 + a.maps_per_chunk);
    const int kid = a.per_map ? (b0 - a.map_base) : 0;
    const KernDev &kd = a.kd[kid];
    const float *taps = a.taps[kid];
    // this thread's rings i0 + t (t < G, valid while G grp + t < nr), i0 = r0 + G grp, whose
    // run starts at input ring jg0
    const int i0 = r0 + G * grp;
    const bool v0 = G * grp < nr;
    const bool wv = v0 && m0 + q4 * 32 < a.NH;  // some mode of the warp exists (N/2 + 1 modes: one in the last block)
    const int jg0 = v0 ? kd.jlo[i0] : 0;
    const int ju0 = kd.jlo[r0];
    const int jlast = kd.jhi[r0 + nr - 1];
    // the groups' common runs are covered by windows of 32 slots
    int nwin = 1;
    if constexpr (WIDE) {
        int len = 1;
        for (int g = 0; g < nr; g += G) len = max(len, kd.jhi[r0 + min(g + G, nr) - 1] - kd.jlo[r0 + g] + 1);
        nwin = (len + kTcBand - 1) / kTcBand;
    }

    // ---- tensor memory and the completion barriers
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"((uint32_t)__cvta_generic_to_shared(tslot)), "r"(Sh::kTmemCols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    if (tid == 0) {
        for (int q = 0; q < 2; ++q)
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;"
                         ::"r"((uint32_t)__cvta_generic_to_shared(mbar + q)));
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    // per column: sample offset in `taps`, last sample and offset flavour (S = -1: empty), and
    // the pair; the largest sample count per tile and flavour
    __shared__ int s_kmax[2][2];
    __shared__ int s_toff[kTcN], s_S[kTcN], s_p[kTcN];  // s_S = 2 S + f
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    if (tid < 4) s_kmax[tid >> 1][tid & 1] = 0;
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = *tslot;
    const uint32_t mbar_s = (uint32_t)__cvta_generic_to_shared(mbar);
    const uint32_t smem_s = (uint32_t)__cvta_generic_to_shared(smem);
    const uint32_t lane_base = tmem + ((uint32_t)(q4 * 32) << 16);

    // blocks whose pairs all have tabulated coefficients read them (whatever the block size,
    // so both block sizes give the same result)
    const bool tabulated = kd.pstart[r0 + nr] <= kd.polar_pairs;
    // once any CTA has seen an expired wait the results are invalid anyway: skip the MMAs
    bool ok = *((volatile int *)&g_tc_error) == 0;
    uint32_t ph = 0;  // bit s: parity of the next completion of stage s

    // ---- staged spectra: rows of the window's input rings, copied by 16-byte asynchronous
    // copies that every thread issues (the copy engine of one thread per CTA cannot keep enough
    // bytes in flight).  nbuf == 2: the next map is copied while this one is contracted;
    // nbuf == 1: one buffer.  Rows past the band read as zero, so every group runs its slots
    // unpredicated (its coefficients are zero there).  rows0 > 0: the first buffer lies past the
    // first stage of the operands, so that the first map is copied while a single pass generates
    // the coefficients.
    const int mid = (a.R - 1) / 2;
    const int row_bytes = kTcModes * (int)sizeof(float4);
    const uint32_t off0 = rows0, off1 = rows0 ? 0 : srows * row_bytes;
    auto issue = [&](int w, int bb, int q) {
        const int j0 = ju0 + w * kTcBand;
        stage_rows<Sh::kThreads>(reinterpret_cast<float4 *>(smem + (q ? off1 : off0)), map_spec4(a, bb), j0,
                                 min(srows, jlast - j0 + 1), m0, a.R, a.NH);
    };
    const int joff = jg0 - ju0;  // the group's first row within the staged rows
    // everything up to here is set up beside the end of the kernels before; the samples and the
    // spectra come from them
    chain_allow_next();
    chain_wait();
    float4 acc[G];
#pragma unroll
    for (int t = 0; t < G; ++t) acc[t] = make_float4(0.f, 0.f, 0.f, 0.f);
    bool fresh = true;  // nothing contracted yet
    auto put = [&](int b) {
        if (!mv) return;
        float2 *cb = a.c + (int64_t)b * a.R * a.NH + m;
#pragma unroll
        for (int t = 0; t < G; ++t) {
            const int i = i0 + t;
            if (G * grp + t < nr) {
                cb[(int64_t)i * a.NH] = make_float2(acc[t].x, acc[t].y);
                if (a.R - 1 - i != i) cb[(int64_t)(a.R - 1 - i) * a.NH] = make_float2(acc[t].z, acc[t].w);
            }
        }
    };

    for (int w = 0; w < nwin; ++w) {
        // ---- the window's columns
        for (int c = tid; c < kTcN; c += blockDim.x) {
            const int tile = c / kTile, l = c % kTile / 16, u = 2 * (c & 15) + ((tile + l) & 1);
            int toff = 0, S = -1, f = 0, p = 0;
            if constexpr (WIDE) {
                const int lg = l - l % G;
                if (l < nr) {
                    const int jl = kd.jlo[r0 + l], j = kd.jlo[r0 + lg] + w * kTcBand + u;
                    if (j >= jl && j <= kd.jhi[r0 + l]) {
                        p = kd.pstart[r0 + l] + j - jl;
                        toff = kd.toff[p];
                        f = a.shift_fix ? kd.fl[p] : 0;
                        S = f ? kd.S1[p] : kd.S0[p];
                    }
                }
            } else {
                // the table of columns is laid out per block of 8 rings
                const int blk8 = blockIdx.y * (RB / 8) + l / 8;
                const int4 *ct = G == 2 ? kd.coltab : kd.coltab4;
                const int4 e = 8 * blk8 < a.nrep ? __ldg(&ct[(size_t)blk8 * 256 + (l & 7) * kTcBand + u])
                                                 : make_int4(-1, 0, -1, -2);
                if (e.x >= 0) {
                    p = e.x;
                    toff = e.y;
                    f = a.shift_fix ? (e.w & 1) : 0;
                    S = f ? (e.w >> 1) : e.z;
                }
            }
            if (S >= 0) atomicMax(&s_kmax[tile][f], S + 1);
            s_toff[c] = toff;
            s_S[c] = 2 * S + f;
            s_p[c] = p;
        }
        __syncthreads();
        const int k00 = s_kmax[0][0], k01 = s_kmax[0][1], k10 = s_kmax[1][0], k11 = s_kmax[1][1];
        const int kall = max(max(k00, k01), max(k10, k11));
        // tiles of one offset each: one pass serves both
        const bool single = !(k00 && k01) && !(k10 && k11);
        const int f0s = k01 ? 1 : 0, f1s = k11 ? 1 : 0;
        // runs of up to 128 samples (0: no samples in the window; the narrow form is launched
        // with at most one)
        const int nrun = tabulated ? 1 : (WIDE ? (kall + kTcRun - 1) / kTcRun : min(kall, 1));
        bool early = false;
        for (int run = 0; run < nrun; ++run) {
            bool have = true;
            if (!tabulated) {
                // passes of this run: (first sample, offset of tile 0, offset of tile 1).  The
                // accumulator truncates each addition at the size of the running sum, so what is
                // small comes first: the last samples of a run (a beam's tail) before the first,
                // and the cross terms of a pass before its hi x hi products
                constexpr int kK = F32 ? kF32K : kTcK;
                const int kb = run * kTcRun;
                auto cap = [&](int k) { return max(0, min(kTcRun, k - kb)); };
                const int n0 = single ? (cap(kall) + kK - 1) / kK : (cap(max(k00, k10)) + kK - 1) / kK;
                const int np = single ? n0 : n0 + (cap(max(k01, k11)) + kK - 1) / kK;
                early = rows0 != 0 && np == 1 && b0 < b1;
                if constexpr (F32) {
                    // plain FP32 form: the samples of every column in shared memory, sample-major;
                    // a thread sums two of its rings at a time in registers (packed two-lane FMAs of
                    // its mode's cosine with broadcast samples), tensor memory holding the sums
                    float *ts = reinterpret_cast<float *>(smem);  // [kF32K][kTcN]
                    for (int i = 0; i < np; ++i) {
                        const bool second = !single && i >= n0;
                        const int k0 = kb + (second ? np - 1 - i : n0 - 1 - i) * kK;
                        const int fA = single ? f0s : (int)second, fB = single ? f1s : (int)second;
                        const int krem = (single ? kall : (second ? max(k01, k11) : max(k00, k10))) - k0;
                        const int nq = (min(kK, krem) + 3) / 4;  // groups of four samples
                        if (i > 0) __syncthreads();
                        for (int c = tid; c < kTcN; c += Sh::kThreads) {
                            const int sf = s_S[c], S = (sf & 1) == (c < kTile ? fA : fB) ? sf >> 1 : -1;
                            const float *tp = taps + s_toff[c] + k0;
                            for (int q = 0; q < nq; ++q) {
                                const float4 v = k0 + 4 * q <= S ? __ldg(reinterpret_cast<const float4 *>(tp + 4 * q))
                                                                 : make_float4(0.f, 0.f, 0.f, 0.f);
                                ts[(4 * q) * kTcN + c] = v.x;  // (slots past the last sample hold zeros)
                                ts[(4 * q + 1) * kTcN + c] = v.y;
                                ts[(4 * q + 2) * kTcN + c] = v.z;
                                ts[(4 * q + 3) * kTcN + c] = v.w;
                            }
                        }
                        if (early) issue(w, b0, 0);
                        __syncthreads();
                        // cosines of four samples from k for offset f (hi + lo of the tables: within
                        // one unit in the last place of the FP32 value)
                        auto cosines = [&](int k, int f, float (&c)[4]) {
                            if (!WIDE || k < nkc_tab * 32) {
                                const float4 *t4 = reinterpret_cast<const float4 *>(
                                    ctab + ((((size_t)blockIdx.x * 2 + f) * nkc_tab + (k >> 5)) * 2) * 4096) +
                                    (mrow >> 3) * 64 + ((k & 31) >> 2) * 8 + (mrow & 7);
                                const float4 h = __ldg(t4), l = __ldg(t4 + 1024);
                                c[0] = h.x + l.x;
                                c[1] = h.y + l.y;
                                c[2] = h.z + l.z;
                                c[3] = h.w + l.w;
                            } else {
#pragma unroll
                                for (int j = 0; j < 4; ++j) {
                                    const float2 v = __ldg(&cos2n[m * (2 * (k + j) + f) % (2 * a.N)]);
                                    c[j] = v.x + v.y;
                                }
                            }
                        };
#pragma unroll 1
                        for (int rp = 0; rp < (wv ? G / 2 : 0); ++rp) {
                            float2 sum[2][2][2 * NY];  // [ring][tile][column pair]
                            const int l0 = G * grp + 2 * rp;
#pragma unroll
                            for (int x = 0; x < 4; ++x) {
                                uint32_t old[4 * NY];
                                if (i > 0) {
                                    tmem_ld_async(lane_base + (uint32_t)((x & 1) * kTile + (l0 + x / 2) * 16), old);
                                    tmem_wait_ld();
                                }
#pragma unroll
                                for (int j = 0; j < 2 * NY; ++j)
                                    sum[x / 2][x & 1][j] = i > 0 ? make_float2(__uint_as_float(old[2 * j]), __uint_as_float(old[2 * j + 1]))
                                                                 : make_float2(0.f, 0.f);
                            }
#pragma unroll 1
                            for (int q = nq - 1; q >= 0; --q) {
                                float cA[4], cB[4];
                                cosines(k0 + 4 * q, fA, cA);
                                if (fA != fB) cosines(k0 + 4 * q, fB, cB);
                                else
#pragma unroll
                                    for (int j = 0; j < 4; ++j) cB[j] = cA[j];
#pragma unroll
                                for (int j = 3; j >= 0; --j) {
#pragma unroll
                                    for (int x = 0; x < 4; ++x) {
                                        const float c = x & 1 ? cB[j] : cA[j];
                                        const float4 *t4 = reinterpret_cast<const float4 *>(
                                            ts + (4 * q + j) * kTcN + (x & 1) * kTile + (l0 + x / 2) * 16);
#pragma unroll
                                        for (int y = 0; y < NY; ++y) fma4(sum[x / 2][x & 1][2 * y], sum[x / 2][x & 1][2 * y + 1], c, t4[y]);
                                    }
                                }
                            }
#pragma unroll
                            for (int x = 0; x < 4; ++x) {
                                float out[4 * NY];
#pragma unroll
                                for (int j = 0; j < 2 * NY; ++j) {
                                    out[2 * j] = sum[x / 2][x & 1][j].x;
                                    out[2 * j + 1] = sum[x / 2][x & 1][j].y;
                                }
                                tmem_st(lane_base + (uint32_t)((x & 1) * kTile + (l0 + x / 2) * 16), out);
                            }
                        }
                    }
                    __syncthreads();
                } else {
                // a thread takes 8 samples of a column, loaded four at a time (tap offsets are
                // multiples of 4 and each pair's slots are padded to 4, so a float4 that starts at
                // or before the last sample stays inside the pair); others read as zero
                constexpr int kUnits = 2 * kTcN / Sh::kThreads;
                float4 pre[kUnits][2];
                auto load_taps = [&](int i) {
                    const bool second = !single && i >= n0;
                    const int k0 = kb + (second ? np - 1 - i : n0 - 1 - i) * kTcK;
#pragma unroll
                    for (int u = 0; u < kUnits; ++u) {
                        const int e = tid + u * Sh::kThreads, c = e % kTcN, kk = k0 + 8 * (e / kTcN);
                        const int fp = single ? (c < kTile ? f0s : f1s) : (int)second;
                        const int sf = s_S[c], S = (sf & 1) == fp ? sf >> 1 : -1;
                        const float *tp = taps + s_toff[c] + kk;
#pragma unroll
                        for (int q = 0; q < 2; ++q)
                            pre[u][q] = kk + 4 * q <= S ? __ldg(reinterpret_cast<const float4 *>(tp + 4 * q))
                                                        : make_float4(0.f, 0.f, 0.f, 0.f);
                    }
                };
                uint32_t pend = 0;    // bit s: a pass of stage s not yet seen complete
                uint32_t issued = 0;  // bit s: its MMAs were issued
                auto await = [&](int st) {
                    if (pend >> st & 1) {
                        if (ok) {
                            bool done = mbar_wait(mbar_s + 8u * st, (ph >> st) & 1);
                            // an issued commit is waited for once more (bounded) before anything
                            // reuses the memory its MMAs use
                            if (!done && (issued >> st & 1)) done = mbar_wait(mbar_s + 8u * st, (ph >> st) & 1);
                            if (!done) atomicOr(&g_tc_error, 1);
                            ok = done;
                        } else if (issued >> st & 1) {
                            (void)mbar_wait(mbar_s + 8u * st, (ph >> st) & 1);
                        }
                        ph ^= 1u << st;
                        pend &= ~(1u << st);
                    }
                };
                bool first = true;
                load_taps(0);
                for (int i = 0; i < np; ++i) {
                    const int st = Sh::kStages == 2 ? (i & 1) : 0;
                    const bool second = !single && i >= n0;
                    const int k0 = kb + (second ? np - 1 - i : n0 - 1 - i) * kTcK;  // first sample of the pass
                    const int fA = single ? f0s : (int)second, fB = single ? f1s : (int)second;
                    const int krem = (single ? kall : (second ? max(k01, k11) : max(k00, k10))) - k0;
                    const int ksteps = krem > 8 ? 2 : 1;
                    unsigned char *A = smem + st * Sh::kStage, *Bh = A + 4 * Sh::kA, *Bl = Bh + Sh::kB;
                    await(st);  // the MMAs of the pass that used this stage
                    // A: this mode block's cosines of the pass (hi, lo), for tile 1 apart when its
                    // offset differs
                    const int ncos = fA == fB ? 1 : 2;
                    if (!WIDE || k0 < nkc_tab * 32) {
                        // prepared in the core layout, 32 samples to a tile
                        const int lp = 3 + ksteps;  // 16 or 32 16-byte units of a row octet
                        for (int e = tid; e < ncos << (lp + 5); e += Sh::kThreads) {
                            const int wi = e & ((1 << lp) - 1), oct = e >> lp & 15, part = e >> (lp + 4);  // 2 tile + lo
                            const float *src = ctab +
                                ((((size_t)blockIdx.x * 2 + (part >> 1 ? fB : fA)) * nkc_tab + (k0 >> 5)) * 2 + (part & 1)) * 4096;
                            cp_async16(A + part * Sh::kA + oct * kTcSBO + wi * 16,
                                       src + oct * 256 + (k0 & 16) * 8 + wi * 4, 16);
                        }
                    } else {
                        // past the tables: cos(pi t / N), t = m (2k + f) mod 2N, split as they are
                        const bool pow2 = (a.N & (a.N - 1)) == 0;
                        for (int e = tid; e < ncos * kTcModes * kTcK; e += Sh::kThreads) {
                            const int x = e % (kTcModes * kTcK), tl = e / (kTcModes * kTcK);
                            const int k = (x & 3) + 4 * (x >> 5 & 3), r = (x >> 2 & 7) + 8 * (x >> 7);
                            const int ang = (m0 + r) * (2 * (k0 + k) + (tl ? fB : fA));
                            const float2 v = __ldg(&cos2n[pow2 ? ang & (2 * a.N - 1) : ang % (2 * a.N)]);
                            const uint32_t off = (r >> 3) * kTcSBO + (k >> 2) * kLBO + (r & 7) * 16 + (k & 3) * 4;
                            *reinterpret_cast<float *>(A + 2 * tl * Sh::kA + off) = v.x;
                            *reinterpret_cast<float *>(A + (2 * tl + 1) * Sh::kA + off) = v.y;
                        }
                    }
                    cp_async_commit();
                    // B: the samples of every column for its tile's offset, split hi / lo
#pragma unroll
                    for (int u = 0; u < kUnits; ++u) {
                        const int e = tid + u * Sh::kThreads, c = e % kTcN, ks = e / kTcN;
                        if (ks >= ksteps) continue;
                        const int sf = s_S[c], kk = k0 + 8 * ks;
                        const uint32_t off = (c >> 3) * kTcSBO + 2 * ks * kLBO + (c & 7) * 16;
#pragma unroll
                        for (int q = 0; q < 2; ++q) {
                            const float v[4] = {pre[u][q].x, pre[u][q].y, pre[u][q].z, pre[u][q].w};
                            float4 hi4, lo4;
                            float *hp = &hi4.x, *lp = &lo4.x;
#pragma unroll
                            for (int j = 0; j < 4; ++j) {
                                const float x = kk + 4 * q + j <= (sf >> 1) ? v[j] : 0.f;
                                hp[j] = tf32_round(x);
                                lp[j] = tf32_round(x - hp[j]);
                            }
                            *reinterpret_cast<float4 *>(Bh + off + q * kLBO) = hi4;
                            *reinterpret_cast<float4 *>(Bl + off + q * kLBO) = lo4;
                        }
                    }
                    if (i + 1 < np) load_taps(i + 1);
                    if (early) issue(w, b0, 0);
                    else cp_async_commit();
                    cp_async_wait1();  // the cosines have landed (all but the newest group)
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                    ok = __syncthreads_and(ok);
                    // CTA-uniform: whether this pass's MMAs and their commit are issued (the test
                    // knob withholds them, so that the wait runs out)
                    const bool go = ok && !a.withhold_mma;
                    if (ok) pend |= 1u << st;
                    issued = go ? issued | (1u << st) : issued & ~(1u << st);
                    if (tid == 0 && go) {
                        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                        constexpr uint32_t idesc = tf32_idesc(kTcModes, kTile);
                        const uint32_t sa = smem_s + st * Sh::kStage, sb = sa + 4 * Sh::kA;
#pragma unroll 1
                        for (int x = 0; x < 3 * ksteps; ++x) {  // C_lo T_hi, C_hi T_lo, C_hi T_hi
                            const int prod = x / ksteps, ks = ksteps - 1 - x % ksteps;
                            const uint32_t o = ks * 2 * kLBO;  // 8 TF32 values = two core columns
#pragma unroll
                            for (int t = 0; t < 2; ++t) {
                                const uint32_t ca = sa + (t && ncos == 2 ? 2 * Sh::kA : 0) + (prod == 0 ? Sh::kA : 0) + o;
                                const uint32_t cb = sb + (uint32_t)t * (kTile / 8) * kTcSBO + (prod == 1 ? Sh::kB : 0) + o;
                                mma_tf32(tmem + (uint32_t)(t * kTile), smem_desc(ca, kTcSBO), smem_desc(cb, kTcSBO),
                                         idesc, first ? 0 : 1);
                            }
                            first = false;
                        }
                        mma_commit(mbar_s + 8u * st);
                    }
                }
                for (int st = 0; st < Sh::kStages; ++st) await((np + st) % Sh::kStages);
                ok = __syncthreads_and(ok);
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                have = ok;
                }
            } else {
                // blocks next to the poles have more samples per pair than the cosine tables hold:
                // their coefficients were tabulated before this launch; they go to the same
                // tensor-memory columns, a ring's 16 slots at a time
                const float *pr = a.prho[kid];
#pragma unroll 1
                for (int h = 0; h < G * 2; ++h) {
                    const int l = G * grp + h / 2, c0 = l * 16 + (h & 1) * 8;
#pragma unroll
                    for (int tile = 0; tile < 2; ++tile) {
                        float r[8];
#pragma unroll
                        for (int u = 0; u < 8; ++u) {
                            const int c = tile * kTile + c0 + u;
                            r[u] = mv && s_S[c] >= 0 ? __ldg(&pr[(int64_t)s_p[c] * a.NH + m]) : 0.f;
                        }
                        tmem_st(lane_base + (uint32_t)(tile * kTile + c0), r);
                    }
                }
                __syncthreads();
            }

            // ---- band contraction of the window's slots, for every map
            const int jw = jg0 + w * kTcBand;     // input ring of the group's first slot
            const int sstar = mid - jw + 1;       // first slot that is a southern ring
            const bool crosses = jlast > mid;
            // whole windows inside the band of every ring of the group run without a test; at the
            // ends of a wide band a slot outside a ring's band is left out (a non-finite input
            // ring reaches only outputs whose support holds it)
            int lo[G], hi[G];
            bool inner = true;
            if constexpr (WIDE) {
#pragma unroll
                for (int t = 0; t < G; ++t) {
                    const int i = r0 + min(G * grp + t, nr - 1);
                    lo[t] = kd.jlo[i] - jw;
                    hi[t] = kd.jhi[i] - jw;
                    inner = inner && lo[t] <= 0 && hi[t] >= kTcBand - 1;
                }
            }
            if (!early && b0 < b1) issue(w, b0, 0);
            // the rows past the band read as zero
            for (int e = min(srows, jlast - ju0 - w * kTcBand + 1) * kTcModes + tid; e < srows * kTcModes; e += Sh::kThreads) {
                reinterpret_cast<float4 *>(smem + off0)[e] = make_float4(0.f, 0.f, 0.f, 0.f);
                if (nbuf == 2) reinterpret_cast<float4 *>(smem + off1)[e] = make_float4(0.f, 0.f, 0.f, 0.f);
            }
            for (int b = b0; b < b1; ++b) {
                const int cur = nbuf == 2 ? (b - b0) & 1 : 0;
                if (nbuf == 2 && b + 1 < b1) {
                    issue(w, b + 1, cur ^ 1);
                    cp_async_wait1();  // this map's copies (all but the newest group) have landed
                } else {
                    asm volatile("cp.async.wait_all;" ::: "memory");
                }
                __syncthreads();
                // outputs of earlier windows and runs: in registers for one map, else written by
                // this thread before
                if (!WIDE || fresh) {
#pragma unroll
                    for (int t = 0; t < G; ++t) acc[t] = make_float4(0.f, 0.f, 0.f, 0.f);
                } else if (b1 - b0 > 1 && mv) {
                    const float2 *cb = a.c + (int64_t)b * a.R * a.NH + m;
#pragma unroll
                    for (int t = 0; t < G; ++t) {
                        const int i = i0 + t;
                        if (G * grp + t < nr) {
                            const float2 x = cb[(int64_t)i * a.NH], y = cb[(int64_t)(a.R - 1 - i) * a.NH];
                            acc[t] = make_float4(x.x, x.y, y.x, y.y);
                        }
                    }
                }
                if (wv && have) {  // warp-uniform: the tensor-memory loads are warp-collective
                    const float4 *col = reinterpret_cast<const float4 *>(smem + (cur ? off1 : off0)) + joff * kTcModes + mrow;
                    // CH slots at a time, in the order of the input rings (whatever the groups): the
                    // coefficients of the G rings (a ring's even and odd slots lie in different
                    // tiles), then the staged values, each used by all G rings
                    constexpr int CH = 8, UNROLL = WIDE ? 1 : SLOTS / CH;  // (wide: less code, 4.5 against 5.1 ms)
                    uint32_t cr[G][2][CH / 2];
                    auto coeffs = [&](int h) {
#pragma unroll
                        for (int t = 0; t < G; ++t)
#pragma unroll
                            for (int o = 0; o < 2; ++o)
                                tmem_ld_async(lane_base + (uint32_t)(((t + o) & 1) * kTile + (G * grp + t) * 16 + h / 2),
                                              cr[t][o]);
                        tmem_wait_ld();
                    };
#pragma unroll(UNROLL)
                    for (int h = 0; h < SLOTS; h += CH) {
                        coeffs(h);
                        if (!crosses && (!WIDE || inner)) {
#pragma unroll
                            for (int u = 0; u < CH; ++u) {
                                const float4 v = col[(h + u) * kTcModes];
#pragma unroll
                                for (int t = 0; t < G; ++t) fma4(acc[t], __uint_as_float(cr[t][u & 1][u >> 1]), v);
                            }
                        } else {
#pragma unroll
                            for (int u = 0; u < CH; ++u) {
                                float4 v = col[(h + u) * kTcModes];
                                if (h + u >= sstar) v = make_float4(v.z, v.w, v.x, v.y);
#pragma unroll
                                for (int t = 0; t < G; ++t)
                                    if (!WIDE || (h + u >= lo[t] && h + u <= hi[t]))
                                        fma4(acc[t], __uint_as_float(cr[t][u & 1][u >> 1]), v);
                            }
                        }
                    }
                    if constexpr (!WIDE) {
                        // a non-finite value of a staged ring times the zero coefficient of a ring
                        // whose band lacks it is NaN: a warp that finds such sums takes them again over
                        // the slots of each ring's own band (the same sums otherwise).  A test of the
                        // sums, as one of every slot costs more (one nside-256 map, plain FP32: 112 us
                        // without a test, 114 with this one, 122 with a test of the slots; 16
                        // nside-2048 maps, 3xTF32: 9.54, 9.55 and 9.74 ms)
                        float2 s = make_float2(0.f, 0.f);
#pragma unroll
                        for (int t = 0; t < G; ++t)
                            s = caddf(s, caddf(make_float2(acc[t].x, acc[t].y), make_float2(acc[t].z, acc[t].w)));
                        if (__any_sync(0xffffffffu, !isfinite(s.x + s.y))) {
                            uint32_t in[G];  // slots of the ring's band
#pragma unroll
                            for (int t = 0; t < G; ++t) {
                                const int i = r0 + min(G * grp + t, nr - 1), jl = kd.jlo[i];
                                in[t] = (0xffffffffu >> (kTcBand - 1 - (kd.jhi[i] - jl))) << (jl - jg0);
                                acc[t] = make_float4(0.f, 0.f, 0.f, 0.f);
                            }
#pragma unroll 1
                            for (int h = 0; h < SLOTS; h += CH) {
                                coeffs(h);
#pragma unroll
                                for (int u = 0; u < CH; ++u) {
                                    float4 v = col[(h + u) * kTcModes];
                                    if (h + u >= sstar) v = make_float4(v.z, v.w, v.x, v.y);
#pragma unroll
                                    for (int t = 0; t < G; ++t) {
                                        // (the plain form has no registers left for the masks)
                                        const int i = r0 + min(G * grp + t, nr - 1), j = jg0 + h + u;
                                        if (F32 ? j >= __ldg(&kd.jlo[i]) && j <= __ldg(&kd.jhi[i]) : in[t] >> (h + u) & 1)
                                            fma4(acc[t], __uint_as_float(cr[t][u & 1][u >> 1]), v);
                                    }
                                }
                            }
                        }
                    }
                }
                if (!WIDE || b1 - b0 > 1) put(b);
                __syncthreads();
                if (nbuf == 1 && b + 1 < b1) issue(w, b + 1, 0);
            }
            fresh = false;
        }
        if (WIDE && w + 1 < nwin) {
            if (tid < 4) s_kmax[tid >> 1][tid & 1] = 0;
            __syncthreads();
        }
    }
    // the wide form's sums of one map were kept in registers; no samples at all: zero outputs
    if (fresh || (WIDE && b1 - b0 == 1))
        for (int b = b0; b < b1; ++b) put(b);

    // ---- release tensor memory
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(Sh::kTmemCols));
}

// Knot-gradient projection on the tensor cores (the 3xTF32 form of the backward pass):
//     X[p][k] = sum_m Q_m(p) cos(pi m (2k + f) / N),   k < 128, f = 0 and 1,
// a dense product of the Q rows of 128 ring pairs (A, M = 128, split hi/lo on the fly) and a
// per-grid table of the cosines of NT taps of each flavour (B, N = 2 NT, K = 32 modes per
// chunk, hi/lo in the core layout), NT = 16, 32, 64 or 128 >= the most samples of a block's pairs
// (most blocks hold pairs of at most 16: one nside-2048 kernel 0.42 ms, the other classes beside
// it, bound by the loads of the Q rows; 1.14 ms with 128 for all, bound by the table copies and
// products).  The sum over the modes is long (N/2 + 1 terms) and the
// cosines make it cancel, so it is not left to the tensor core's accumulator, whose additions
// do not round to nearest: every chunk's twelve MMAs start from zero in one of two 2 NT-column
// accumulators, and once a chunk is complete its 128 x 2 NT partial sums are added in FP32
// (round to nearest) into registers of the epilogue threads while the next chunk's MMAs fill
// the other accumulator.  Two stages of shared memory: chunk c + 1 is staged while the MMAs of
// chunk c run, each stage (and its accumulator) released by its own completion barrier
// (bounded waits).  Each pair's row of its own flavour's NT values goes to X; the hat-weight
// deposits follow in k_knot_deposit.
constexpr int kPjPairs = 128, kPjThreads = 256;
constexpr uint32_t kPjA = 16384;
template <int NT>
struct PjShape {
    static constexpr uint32_t kB = 2 * NT * 128, kStage = 2 * kPjA + 2 * kB;  // 40 to 96 KiB per stage
    static constexpr uint32_t kCols = 2 * NT;                                 // per accumulator
    static constexpr uint32_t kAlloc = 2 * kCols < 32 ? 32 : 2 * kCols;
};

// cls: the class of blocks (KnotGradArgs::cut); first: the launch that follows the Q rows (the
// other classes start beside it and only end after it)
template <int NT>
__global__ void __launch_bounds__(kPjThreads, NT <= 32 ? 2 : 1)
k_knot_proj_tc(const __grid_constant__ KnotGradArgs a, const float *__restrict__ ctabP, int nmc, int cls, int first)
{
    using Sh = PjShape<NT>;
    constexpr uint32_t kPjStage = Sh::kStage, kPjB = Sh::kB, kPjCols = Sh::kCols;
    const int kb = blockIdx.y, blk = a.cut[kb][cls] + blockIdx.x;
    if (first) chain_wait();
    chain_allow_next();
    if (blk >= a.cut[kb][cls + 1]) {
        chain_wait();
        return;
    }
    const KernDev &kd = a.kd[kb];
    const float *Q = a.Q + kb * a.qstride;
    const int pfirst = a.fft_pairs[kb];
    float *X = a.X + kb * a.xstride;
    extern __shared__ __align__(1024) unsigned char smem[];
    uint64_t *bar = reinterpret_cast<uint64_t *>(smem + 2 * kPjStage);  // [2] stage barriers
    uint32_t *tslot = reinterpret_cast<uint32_t *>(smem + 2 * kPjStage + 16);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int pbase = pfirst + blk * kPjPairs;
    const int npairs = kd.npairs;
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"((uint32_t)__cvta_generic_to_shared(tslot)), "r"(Sh::kAlloc));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    if (tid == 0) {
        for (int q = 0; q < 2; ++q)
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;"
                         ::"r"((uint32_t)__cvta_generic_to_shared(bar + q)));
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = *tslot;
    const uint32_t bar_s = (uint32_t)__cvta_generic_to_shared(bar);
    bool ok = *((volatile int *)&g_tc_error) == 0;
    ok = __syncthreads_and(ok);
    uint32_t ph = 0;    // bit s: parity of the next completion of stage s
    uint32_t pend = 0;  // bit s: stage s has an issued commit not yet seen complete
    const uint32_t idesc = tf32_idesc(kTcModes, 2 * NT);
    // epilogue role of the thread: warp (lane quarter, column half), lane = pair, columns =
    // the half's NT taps; it sums every chunk's partials of those columns in registers
    const int er = (warp & 3) * 32 + lane, ehalf = warp >> 2;
    float acc[NT];
#pragma unroll
    for (int j = 0; j < NT; ++j) acc[j] = 0.f;
    // adds the completed partial sums of accumulator `buf` (after its completion wait)
    auto drain = [&](int buf) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t base = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)buf * kPjCols +
                              (uint32_t)(ehalf * NT);
#pragma unroll
        for (int h = 0; h < NT; h += 16) {
            uint32_t v[16];
            tmem_ld_async(base + (uint32_t)h, v);
            tmem_wait_ld();
#pragma unroll
            for (int j = 0; j < 16; ++j) acc[h + j] += __uint_as_float(v[j]);
        }
    };
    // A: a thread takes four units of (pair row r, 4 consecutive modes from k4); the eight
    // lanes of a quarter-warp hold eight consecutive rows, so their 16-byte stores land in
    // distinct bank groups of the core layout.  The next chunk's values are loaded into
    // registers while the current chunk's MMAs run.
    float pre[4][4];
    auto load_a = [&](int c) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int U = tid + kPjThreads * i;
            const int r = (U & 7) + 8 * (U >> 6), k4 = ((U >> 3) & 7) * 4;
            const int p = pbase + r;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int m = 32 * c + k4 + j;
                pre[i][j] = (p < npairs && m < a.NH) ? __ldg(&Q[(int64_t)p * a.NH + m]) : 0.f;
            }
        }
    };
    if (nmc > 0) load_a(0);
    for (int c = 0; c < nmc; ++c) {
        const int st = c & 1;
        unsigned char *Ahi = smem + st * kPjStage, *Alo = Ahi + kPjA, *Bhi = Ahi + 2 * kPjA, *Blo = Bhi + kPjB;
        if (c >= 2) {  // the MMAs of chunk c - 2 read this stage and wrote this accumulator
            if (ok) {
                ok = mbar_wait(bar_s + 8u * st, (ph >> st) & 1);
                if (ok) pend &= ~(1u << st);
            }
            ph ^= 1u << st;
            if (ok) drain(st);
        }
        // B: the first NT rows of each flavour of the chunk's cosine tile (hi then lo)
        const float *src = ctabP + (size_t)c * 2 * 8192;
        for (int e = tid; e < 4 * NT * 8; e += kPjThreads) {
            const int unit = e % (NT * 8), f = e / (NT * 8) & 1, part = e / (NT * 16);
            cp_async16(Bhi + part * kPjB + f * NT * 128 + unit * 16, src + part * 8192 + f * 4096 + unit * 4, 16);
        }
        cp_async_commit();
        // A: the Q rows of the block's pairs at the chunk's 32 modes, split hi / lo
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int U = tid + kPjThreads * i;
            const int r = (U & 7) + 8 * (U >> 6), k4 = ((U >> 3) & 7) * 4;
            float4 hi4, lo4;
            float *hp = &hi4.x, *lp = &lo4.x;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                hp[j] = tf32_round(pre[i][j]);
                lp[j] = tf32_round(pre[i][j] - hp[j]);
            }
            const uint32_t off = core_offset(r, k4);
            *reinterpret_cast<float4 *>(Ahi + off) = hi4;
            *reinterpret_cast<float4 *>(Alo + off) = lo4;
        }
        if (c + 1 < nmc) load_a(c + 1);
        asm volatile("cp.async.wait_all;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        // the accumulator's reads (drain) are ordered before the MMAs that overwrite it
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        ok = __syncthreads_and(ok);
        // CTA-uniform: the MMAs and commit of this chunk are issued (the test knob withholds
        // them, so that the completion wait runs out)
        const bool issued = ok && !a.withhold_mma;
        if (issued) pend |= 1u << st;
        if (tid == 0 && issued) {
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint32_t sa_hi = (uint32_t)__cvta_generic_to_shared(Ahi);
            const uint32_t sa_lo = (uint32_t)__cvta_generic_to_shared(Alo);
            const uint32_t sb_hi = (uint32_t)__cvta_generic_to_shared(Bhi);
            const uint32_t sb_lo = (uint32_t)__cvta_generic_to_shared(Blo);
            const uint32_t d = tmem + (uint32_t)st * kPjCols;
            for (int ks = 0; ks < 4; ++ks) {
                const uint32_t o = ks * 2 * kLBO;
                mma_tf32(d, smem_desc(sa_hi + o), smem_desc(sb_hi + o), idesc, ks == 0 ? 0 : 1);
                mma_tf32(d, smem_desc(sa_hi + o), smem_desc(sb_lo + o), idesc, 1);
                mma_tf32(d, smem_desc(sa_lo + o), smem_desc(sb_hi + o), idesc, 1);
            }
            mma_commit(bar_s + 8u * st);
        }
    }
    // the last (up to) two chunks
    for (int c = max(0, nmc - 2); c < nmc; ++c) {
        const int st = c & 1;
        if (ok) {
            ok = mbar_wait(bar_s + 8u * st, (ph >> st) & 1);
            if (ok) pend &= ~(1u << st);
        }
        ph ^= 1u << st;
        if (ok) drain(st);
    }
    ok = __syncthreads_and(ok);
    if (!ok && tid == 0) atomicOr(&g_tc_error, 4);
    // after an expired wait: every issued commit not yet seen complete is waited for once more
    // (bounded) before the tensor memory and shared memory its MMAs use are released; a
    // withheld issue left nothing in flight
    if (!ok)
        for (int st = 0; st < 2; ++st)
            if (pend & (1u << st)) (void)mbar_wait(bar_s + 8u * st, (ph >> st) & 1);
    // a pair keeps the half of its own flavour
    {
        const int p = pbase + er;
        const bool pv = ok && p < npairs;
        const int f = pv && a.shift_fix ? kd.fl[p] : 0;
        if (pv && f == ehalf) {
            float *xr = X + (int64_t)(p - pfirst) * 128;
#pragma unroll
            for (int j = 0; j < NT; j += 4)
                *reinterpret_cast<float4 *>(xr + j) = make_float4(acc[j], acc[j + 1], acc[j + 2], acc[j + 3]);
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(Sh::kAlloc));
    chain_wait();
}

}  // namespace

int contract_tc_modes() { return kTcModes; }

constexpr size_t kTcSmemLimit = 216 * 1024;  // dynamic shared memory of a one-CTA-per-SM launch
constexpr size_t kTcRow = (size_t)kTcModes * sizeof(float4);

// Staging buffers of srows rows for blocks of rb rings.  Two CTAs per SM
// (rb == 8): one, unless `want` == 2 and two fit in 200 KiB.  One CTA per SM (rb == 16): two when
// they fit.
int contract_tc_nbuf(int rb, int srows, int want)
{
    if (rb == 16) return 2 * srows * kTcRow + 32 <= kTcSmemLimit ? 2 : 1;
    return want == 2 && 2 * srows * kTcRow + 32 <= 200 * 1024 ? 2 : 1;
}

namespace {

// Offset of the first staging buffer: past the first operand stage where two buffers (the
// second over that stage) fit a CTA that has the SM to itself.
uint32_t tc_rows0(int rb, int srows)
{
    const uint32_t st = TcShape<16, 4>::kStage;
    return rb == 16 && srows * kTcRow <= st && st + srows * kTcRow + 32 <= kTcSmemLimit ? st : 0;
}

// Offset of the barriers behind the operand stages and the staging buffers.
size_t tc_ctl(int rb, int nbuf, int srows)
{
    const uint32_t rows0 = tc_rows0(rb, srows);
    const size_t stages = rb == 16 ? 2 * (size_t)TcShape<16, 4>::kStage : (size_t)TcShape<8, 4>::kStage;
    const size_t rows = rows0 ? rows0 + srows * kTcRow : nbuf * srows * kTcRow;
    return (std::max(stages, rows) + 15) & ~size_t(15);
}

}  // namespace

int contract_band_limit() { return kTcBand; }

namespace {

template <int RB, int G, bool WIDE, bool F32, int SLOTS = kTcBand>
cudaError_t launch_tc(const ContractArgs &a, int nchunks, const TcTables &tb, int srows, int nbuf, cudaStream_t st)
{
    const size_t ctl = tc_ctl(RB, nbuf, srows), smem = ctl + 32;
    cudaError_t e = cudaFuncSetAttribute((const void *)k_contract_tc<RB, G, WIDE, F32, SLOTS>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    dim3 grid((a.NH + kTcModes - 1) / kTcModes, (a.nrep + RB - 1) / RB, nchunks);
    return launch_chained(k_contract_tc<RB, G, WIDE, F32, SLOTS>, grid, TcShape<RB, G>::kThreads, smem, st, true, 1, a, tb.ctab,
                          tb.cos2n, tb.nkc, srows, nbuf, tc_rows0(RB, srows), (uint32_t)ctl);
}

}  // namespace

// union4: widest union band of a group of four.  Where it reaches 16 slots at most, the plain form sums no
// more: on few CTAs its sums are the longest part (one 90 x 180 map, supports of 4 and 10 degrees: 49.1 and
// 53.9 us, 65.5 and 70.0 with all 32 slots; five maps: 60.3 and 65 us, 77.4 and 82.3).
cudaError_t launch_contract_tc(const ContractArgs &a, int rb, int gs, bool f32, int union4, int nchunks,
                               const TcTables &tb, int srows, int want_nbuf, cudaStream_t st)
{
    const int nbuf = contract_tc_nbuf(rb, srows, want_nbuf);
    if (f32)
        return union4 <= 16 ? launch_tc<8, 4, false, true, 16>(a, nchunks, tb, srows, nbuf, st)
                            : launch_tc<8, 4, false, true>(a, nchunks, tb, srows, nbuf, st);
    if (rb == 16)
        return gs == 4 ? launch_tc<16, 4, false, false>(a, nchunks, tb, srows, nbuf, st)
                       : launch_tc<16, 2, false, false>(a, nchunks, tb, srows, nbuf, st);
    return gs == 4 ? launch_tc<8, 4, false, false>(a, nchunks, tb, srows, nbuf, st)
                   : launch_tc<8, 2, false, false>(a, nchunks, tb, srows, nbuf, st);
}

// Bands of any width: blocks of 16 rings in groups of four, the 32 slots moving along the band.
cudaError_t launch_contract_tc_wide(const ContractArgs &a, bool f32, int nchunks, const TcTables &tb, int srows,
                                    cudaStream_t st)
{
    const int nbuf = contract_tc_nbuf(16, srows, 0);
    return f32 ? launch_tc<16, 4, true, true>(a, nchunks, tb, srows, nbuf, st)
               : launch_tc<16, 4, true, false>(a, nchunks, tb, srows, nbuf, st);
}

namespace {

template <int NT>
cudaError_t launch_pj(const KnotGradArgs &a, const float *ctabP, int nmc, int cls, bool first, cudaStream_t st)
{
    int blocks = 0;
    for (int k = 0; k < a.nk; ++k) blocks = std::max(blocks, a.cut[k][cls + 1] - a.cut[k][cls]);
    if (blocks <= 0) return cudaSuccess;
    const size_t smem = 2 * (size_t)PjShape<NT>::kStage + 32;
    cudaError_t e = cudaFuncSetAttribute((const void *)k_knot_proj_tc<NT>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    return launch_chained(k_knot_proj_tc<NT>, dim3(blocks, a.nk), kPjThreads, smem, st, true, 1, a, ctabP, nmc, cls,
                          (int)first);
}

}  // namespace

// Knot-gradient projection of the pairs past the FFT ones into X (rows of 128 taps of each pair's
// own flavour); ctabP holds nmc chunks of 32 modes.
cudaError_t launch_knot_proj_tc(const KnotGradArgs &a, const float *ctabP, int nmc, int maxblocks, cudaStream_t st)
{
    if (maxblocks <= 0) return cudaSuccess;
    bool first = true;
    for (int cls = 3; cls >= 0; --cls) {
        int blocks = 0;
        for (int k = 0; k < a.nk; ++k) blocks = std::max(blocks, a.cut[k][cls + 1] - a.cut[k][cls]);
        if (blocks <= 0) continue;
        const cudaError_t e = cls == 3   ? launch_pj<16>(a, ctabP, nmc, cls, first, st)
                              : cls == 2 ? launch_pj<32>(a, ctabP, nmc, cls, first, st)
                              : cls == 1 ? launch_pj<64>(a, ctabP, nmc, cls, first, st)
                                         : launch_pj<128>(a, ctabP, nmc, cls, first, st);
        if (e != cudaSuccess) return e;
        first = false;
    }
    return cudaSuccess;
}

// Host-side reset/readout of the device error word (bounded waits that expired).
cudaError_t take_tc_error(int *out)
{
    int v = 0;
    cudaError_t e = cudaMemcpyFromSymbol(&v, g_tc_error, sizeof(int));
    if (e != cudaSuccess) return e;
    *out = v;
    if (v) {
        const int z = 0;
        e = cudaMemcpyToSymbol(g_tc_error, &z, sizeof(int));
    }
    return e;
}

}  // namespace arkcos
