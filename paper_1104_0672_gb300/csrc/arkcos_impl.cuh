// Internal declarations of libarkcos (not installed; the public ABI is include/arkcos.h).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <string>
#include <vector>

#include "arkcos.h"

namespace arkcos {

constexpr int kMaxKernelsPerLaunch = 32;  // per-map beams handled per contraction launch
constexpr int kMaxPolarPairs = 16384;      // most pairs whose coefficients are tabulated per call
constexpr int kModeBlock = 128;           // modes per CTA of the generic knot-gradient kernel
constexpr int kMaxFftM = 8192;            // largest in-shared-memory ring FFT buffer (complex pairs)
constexpr int kBluMin = 9, kBluMax = 12;  // log2 buffer of the split Bluestein classes (ring_blu.cuh)

// Ring table on the device (structure of arrays, R entries each).
struct RingDev {
    const int *n;         // pixels in the ring (even)
    const int *hs;        // 1: first pixel at phi0 = pi / n (half-pixel offset); 0: phi0 = 0
    const int64_t *poff;  // offset of the ring's first pixel in a map
    const int64_t *soff;  // offset of the ring's half spectrum (n/2 + 1 complex)
    const float *w;       // pixel solid-angle weight
    const double *theta;  // colatitude (FP64)
    const float2 *fb;     // Bluestein chirp spectra of the representative rings
    const int *fboff;     // [R] offset of a ring's chirp spectrum in fb (-1: power-of-two ring)
};

// One class of ring-pair representatives sharing an FFT buffer size M.
struct FftClass {
    int M = 0;            // largest buffer of the class (rings pick their own size <= M)
    int logM = 0;
    int threads = 0;
    int count = 0;
    int stage_c = 0;      // some ring of the class is shorter than N / 4
    int blu = 0;          // a split Bluestein class (ring_blu.cuh)
    int even_h = 1;       // ... whose rings all have a multiple of four pixels
    int tab = 0;          // largest chirp + phase table of the class (complex words)
    int *reps = nullptr;  // device array of representative (northern) ring indices
};

struct Grid {
    int kind = 0;  // 0 HEALPix, 1 ECP
    int64_t nside = 0, ntheta = 0, nphi = 0;
    int R = 0;         // rings
    int N = 0;         // kernel longitude grid length
    int nrep = 0;      // ring-pair representatives (northern rings incl. the middle one)
    int64_t npix = 0;  // pixels per map
    int64_t nspec = 0; // complex half-spectrum entries per map, sum (n/2 + 1)
    std::vector<double> theta, wgt;
    std::vector<int> n, hs;
    std::vector<int64_t> poff, soff;
    // device copies
    int *d_n = nullptr, *d_hs = nullptr;
    int64_t *d_poff = nullptr, *d_soff = nullptr;
    float *d_w = nullptr;
    double *d_theta = nullptr;
    float2 *d_tw = nullptr;     // stage twiddles: tw[h + p] = exp(-2 pi i p / (2h)), p < h
    int twM = 0;
    double *d_s2 = nullptr;     // sin^2(pi t / (2N)) for t = 0..N
    float *d_s2f = nullptr;     // the same rounded to FP32 (the knot-segment search)
    float *d_ctab = nullptr;    // tensor-core cosine table (TF32 hi/lo, core-matrix layout)
    int nkc_tab = 0;            // 32-sample chunks the cosine table covers
    float2 *d_cos2n = nullptr;  // cos(pi t / N), t < 2N, as TF32 (hi, lo): samples past that table
    float *d_ctabP = nullptr;   // knot-projection cosine table: per chunk of 32 modes, 128 taps of
                                // each flavour (TF32 hi/lo, core-matrix layout)
    int nmc_p = 0;              // its chunks of 32 modes
    std::vector<FftClass> fft;  // forward/inverse FFT launch classes
    int live_kernels = 0;
    float2 *d_fb = nullptr;     // Bluestein chirp spectra (DIF order) of the representative rings
    int *d_fboff = nullptr;
    RingDev dev() const { return RingDev{d_n, d_hs, d_poff, d_soff, d_w, d_theta, d_fb, d_fboff}; }
};

// Device view of one kernel's ring-pair tables.  Pairs are listed per representative
// output ring i (i <= R-1-i), with input rings j = jlo[i]..jhi[i] in order.
struct KernDev {
    const int *pstart;   // [nrep + 1] first pair of each representative
    const int *jlo;      // [nrep]
    const int *jhi;      // [nrep]
    const int *S0;       // [npairs] last in-support tap, integer-offset samples (-1 none)
    const int *S1;       // [npairs] last in-support tap, half-offset samples (-1 none)
    const int *fl;       // [npairs] 1 when the pair samples at half offsets (shift fix)
    const int *toff;     // [npairs + 1] tap offsets (multiples of 4)
    const double *A;     // [npairs] sin^2((theta_i + theta_j)/2)
    const double *B;     // [npairs] sin^2((theta_i - theta_j)/2)
    const double *knots; // [T]
    const double *ut;    // [T] u_t = 4 sin^2(gamma_t / 2)
    const int4 *coltab;  // [ceil(nrep / 8)][256] tensor-core columns of each block of 8 rings:
                         // (pair or -1, tap offset, S0, 2 S1 + fl), rings in groups of two
    const int4 *coltab4; // the same with the rings in groups of four
    const int2 *unit_fix;   // knot-gradient work units (pair, first tap), with the shift fix
    const int2 *unit_nofix; // ... and without it
    int nunit_fix, nunit_nofix;
    int T;
    int npairs;
    int nrep;            // representative output rings
    int polar_pairs;     // pairs [0, polar_pairs) (rings next to the poles with many samples)
                         // take their coefficients from a table computed before the contraction
    double umax;
    double gscale;       // (T - 1) / gamma_max, for the first guess of the knot segment
};

struct Kernel {
    Grid *g = nullptr;
    int T = 0;
    double gmax = 0, umax = 0;
    int npairs = 0;
    int64_t ntaps = 0;  // padded tap slots
    int maxband = 0;
    int pole_band = 0;         // input rings inside the support of ring 0
    int64_t pole_pixels = 0;   // their pixels
    int max_union8 = 0;        // largest union band of 8 consecutive representative rings
    int max_union2 = 0;        // largest union band of rings 2g, 2g+1 of those blocks of 8
    int max_stage_rows = 0;    // staged rows a tensor-core block of 8 rings needs: its union
                               // band, and every group's first ring + 32 slots
    int max_stage_rows16 = 0;  // the same for blocks of 16 rings
    int max_union4 = 0;        // largest union band of rings 4g .. 4g+3
    int max_stage_rows_g4 = 0, max_stage_rows16_g4 = 0;  // staged rows with groups of four
    int max_free_taps = 0;     // most samples of a pair whose coefficients are not tabulated
    int max_win_rows = 0;      // rows of a 32-slot window over a block of 16 in groups of four
    int polar_pairs = 0;       // leading pairs whose coefficients are tabulated per call
    int knot_fft_pairs = 0;    // leading pairs whose knot-gradient projection runs by FFT
    bool proj_tc_ok = false;   // the other pairs have at most 128 samples (projection by table)
    int proj_cut[5] = {};      // their blocks of 128 pairs by samples (KnotGradArgs::cut)
    int proj_taps = 0;         // most samples of one of them
    int64_t sum_taps_fix = 0;  // in-support tap count with the shift fix (for reporting)
    void *dmem = nullptr;      // one device allocation holding every table
    KernDev kd{};
};

// ------------------------------------------------------------------ launch arguments
struct TapArgs {
    KernDev kd[kMaxKernelsPerLaunch];
    float *taps[kMaxKernelsPerLaunch];  // [ntaps] of each kernel
    const double *s2;
    const float *s2f;
    int N;
    int shift_fix;
    // ksum > 0: the samples of sum_k w[k] K_k, k < ksum, over the pairs of kernel kbase (the widest)
    int ksum, kbase;
    float w[kMaxKernelsPerLaunch];
};

struct FftFwdArgs {
    RingDev rd;
    const float2 *tw;
    const float *map;   // [B][npix]
    float2 *spec;       // [B][nspec] half spectra (ext4 == 0)
    float4 *spec4;      // [B][nrep][NH] extended spectra of ring and mirror (ext4 == 1)
    int ext4, nrep, NH, basic;
    const int *reps;
    int M, logM, R, N, B;
    int mchunk;         // maps per CTA: CTA (ring pair, blockIdx.y) takes maps [y mchunk, ...)
    int64_t npix, nspec;
    int weight;         // multiply spectra by the ring weight
    int zero_poles;     // treat rings 0 and R-1 as zero (adjoint input)
    int tab;            // shared-memory words for the per-ring chirp and phase tables
};

struct FftInvArgs {
    RingDev rd;
    const float2 *tw;
    const float2 *c;    // [B][R][NH]
    float *map;         // [B][npix]
    const int *reps;
    int M, logM, R, N, NH, B;
    int mchunk;         // maps per CTA: CTA (ring pair, blockIdx.y) takes maps [y mchunk, ...)
    int64_t npix;
    int weight;         // multiply by the ring weight
    int basic;
    int skip_poles;     // leave rings 0 and R-1 untouched (written by the pole kernel)
    int stage_c;        // stage coefficients in shared memory for rings with 4 n < N
    int tab;            // shared-memory words for the per-ring chirp and phase tables
    int first;          // first class of the stage: its input comes from the kernel before it
};

struct ContractArgs {
    RingDev rd;
    KernDev kd[kMaxKernelsPerLaunch];
    const float *taps[kMaxKernelsPerLaunch];
    const float *prho[kMaxKernelsPerLaunch];  // [polar_pairs][NH] tabulated coefficients
    const float4 *spec4; // [B][nrep][NH]: (a_m(j), a_m(R-1-j)) for representative j
    float2 *c;          // [B][R][NH]
    int R, N, NH, nrep, B;
    int64_t nspec;
    int maps_per_chunk; // maps sharing one generation pass
    int per_map;        // 1: map b uses kd[b - map_base]
    int map_base;
    int basic, shift_fix;
    int withhold_mma;   // test knob: issue no tensor-core MMA, so the completion waits expire
    int vbase, vdiv;    // vdiv > 1 (several kernels on one input): map b of the launch reads the
                        // spectra of input (vbase + b) / vdiv of spec4; else those of map b
};

// Extended spectra of map b of a contraction launch.
__device__ __forceinline__ const float4 *map_spec4(const ContractArgs &a, int b)
{
    const int s = a.vdiv > 1 ? (a.vbase + b) / a.vdiv : b;
    return a.spec4 + (int64_t)s * a.nrep * a.NH;
}

struct PoleArgs {
    RingDev rd;
    KernDev kd[kMaxKernelsPerLaunch];
    const float *map;   // input (forward) or gradient (adjoint)
    float *out;
    int R, B, per_map, map_base;
    int64_t npix;
    int vbase, vdiv;    // vdiv > 1: output map b reads input map (vbase + b) / vdiv of `map`
    int nsum;           // > 0 (forward only): output map b is the sum over kernels k < nsum of
    double wsum[kMaxKernelsPerLaunch];  // wsum[k] x the direct sum of kd[k] over input map b
};

// Knot gradients of up to kMaxKernelsPerLaunch kernels (blockIdx.z or .y of the launches): kernel
// b of the batch has its own Q rows, projections and partial sums.
struct KnotGradArgs {
    RingDev rd;
    KernDev kd[kMaxKernelsPerLaunch];
    int fft_pairs[kMaxKernelsPerLaunch];  // leading pairs projected by FFT
    int cut[kMaxKernelsPerLaunch][5];     // tensor-core projection: first block of 128 pairs (past those) of
                                          // at most 128, 64, 32 and 16 samples, and their number
    const float4 *spec4;  // weighted extended spectra of the input maps [B][nrep][NH]
    const float4 *gspec4; // extended spectra of the output gradients [B][nrep][NH]
    const double *s2;
    const float2 *tw;    // stage twiddles of the grid (FFT projection of the polar pairs)
    float *Q, *X;        // [pairs][NH] and [pairs past the FFT ones][128] per kernel
    double *partial;     // [rows][T] partial sums per kernel: deposit CTAs, FFT pairs, pole rings
    int64_t qstride, xstride, pstride;  // elements from a kernel to the next
    int nk;              // kernels of the launch
    int row_fft, row_pole;              // first rows of the FFT pairs and the pole rings
    int pole_split[kMaxKernelsPerLaunch];  // CTAs sharing a pole pixel's sum
    int R, N, NH, nrep, B, map0, nmaps; // kernel b sums maps [map0 + b * per_map, + nmaps)
    int per_map;
    int64_t nspec;
    int basic, shift_fix;
    int pole_fix;        // pole rings' hybrid outputs are replaced (skip their g)
    int withhold_mma;    // test knob: issue no tensor-core MMA, so the completion waits expire
};

// Extended spectrum of ring j at mode m from the paired layout: the representative row of j
// holds (a(rep), a(R-1-rep)); swap the halves for rings of the southern half.
__device__ __forceinline__ float4 paired_coeff(const float4 *__restrict__ sp4, int j, int R, int NH, int m)
{
    const int jm = R - 1 - j;
    const bool south = j > jm;
    float4 v = __ldg(&sp4[(int64_t)(south ? jm : j) * NH + m]);
    if (south) v = make_float4(v.z, v.w, v.x, v.y);
    return v;
}

// ------------------------------------------------------------------ launchers (return cuda error)
// Kernel samples of nk kernels (or the weighted sum, a.ksum); maxtaps: most tap slots of one.
// after_prev: may begin while the kernel before it on the stream still runs.
cudaError_t launch_taps(const TapArgs &a, int nk, int64_t maxtaps, cudaStream_t st, bool after_prev);
cudaError_t launch_polar_rho(const ContractArgs &a, int nk, int max_polar_pairs, const float2 *tw, int twM,
                             const float2 *cos2n, cudaStream_t st);
size_t fft_smem_bytes(int M, int N, bool stage_c, int tab, int threads);  // shared memory of a ring FFT class
cudaError_t launch_chirp_spectra(const FftFwdArgs &a, float2 *fb, int count, int threads, cudaStream_t st);
// Ring FFT class launches.  after_prev: the previous kernel on the stream is the previous class
// of the same stage (or the kernel of the call before an inverse stage), and this launch may begin
// while it still runs (launch_chained): the classes of a stage write disjoint rings and read only
// what earlier stages wrote, so later ones fill the SMs that the last wave of one leaves idle.
cudaError_t launch_fft_fwd(const FftFwdArgs &a, int count, cudaStream_t st, bool after_prev);
cudaError_t launch_blu_fwd(const FftFwdArgs &a, bool even_h, int count, cudaStream_t st, bool after_prev);
cudaError_t launch_blu_inv(const FftInvArgs &a, bool even_h, int count, cudaStream_t st, bool after_prev);
cudaError_t launch_blu_spectra(const FftFwdArgs &a, float2 *fb, int count, cudaStream_t st);  // a.logM, rd, reps, tw
int blu_table_words(int h);                // words of the per-ring tables of a ring of n = 2h pixels
size_t blu_smem_bytes(int M, int tab);
int fft_map_chunk(int count, int nmaps, int split_mult);  // maps per CTA of a ring FFT launch over `count` ring pairs
cudaError_t launch_fft_inv(const FftInvArgs &a, int count, cudaStream_t st, bool after_prev);

// Launch of kernel(args...) in clusters of `cluster` CTAs along x, with the
// programmatic-serialization attribute when after_prev: the kernel may then begin while the
// kernel before it on the stream still runs, once all CTAs of that one have started and allowed
// it, and waits for it (chain_wait) before it reads its results and before it ends, so that the
// end of every kernel of a chain is the end of all before it.
template <class... P, class... A>
cudaError_t launch_chained(void (*kernel)(P...), dim3 grid, int threads, size_t smem, cudaStream_t st,
                           bool after_prev, int cluster, const A &...args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[2];
    int n = 0;
    if (after_prev) {
        at[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        at[n++].val.programmaticStreamSerializationAllowed = 1;
    }
    if (cluster > 1) {
        at[n].id = cudaLaunchAttributeClusterDimension;
        at[n].val.clusterDim.x = (unsigned)cluster;
        at[n].val.clusterDim.y = 1;
        at[n++].val.clusterDim.z = 1;
    }
    cfg.attrs = at;
    cfg.numAttrs = n;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}
// band_pixels: pixels of the rings inside the support of a pole
cudaError_t launch_pole_fwd(const PoleArgs &a, int64_t band_pixels, cudaStream_t st, bool after_prev);
cudaError_t launch_pole_adj(const PoleArgs &a, int max_band_rings, cudaStream_t st);
cudaError_t launch_knot_grad_q(const KnotGradArgs &a, int max_band, int max_union, int max_union2, int srows,
                               cudaStream_t st);
// The cosine sums of the pairs past the FFT ones into X (all of at most 128 samples): tensor cores
// or plain FP32
cudaError_t launch_knot_proj_tc(const KnotGradArgs &a, const float *ctabP, int nmc, int maxblocks, cudaStream_t st);
cudaError_t launch_knot_proj_f32(const KnotGradArgs &a, const float *ctabP, int nmc, int maxpairs, int maxtaps,
                                 cudaStream_t st);
// Deposits of those pairs (have_x), or projection and deposits where a pair has more samples
cudaError_t launch_knot_grad_proj(const KnotGradArgs &a, bool have_x, int T, cudaStream_t st);
cudaError_t launch_knot_grad_proj_fft(const KnotGradArgs &a, int maxpairs, int T, cudaStream_t st);
cudaError_t launch_knot_grad_pole(const KnotGradArgs &a, const float *map, const float *gout, int64_t npix, int T,
                                  cudaStream_t st);
int knot_proj_blocks();
int knot_proj_taps();
int knot_pole_split(int64_t band_pixels);  // CTAs sharing a pole pixel's sum
cudaError_t launch_knot_reduce(const KnotGradArgs &a, double *out, int T, cudaStream_t st);
// Which of the Q kernels serves bands like these (kernels of one launch agree on it)
int knot_q_form(int max_band, int max_union, int max_union2, int srows);
void set_last_error(const char *msg);  // sets the message arkcos_last_error() returns
int contract_band_limit();
// tensor-core contraction over blocks of rb (8 or 16) representative rings, a thread taking
// a group of gs (2 or 4) rings; the wide form takes bands of any width
struct TcTables {
    const float *ctab;    // cosines of the first 32 nkc samples in the operand layout
    const float2 *cos2n;  // cos(pi t / N), t < 2N (hi, lo)
    int nkc;
};
cudaError_t launch_contract_tc(const ContractArgs &a, int rb, int gs, bool f32, int union4, int nchunks,
                               const TcTables &tb, int srows, int want_nbuf, cudaStream_t st);
cudaError_t launch_contract_tc_wide(const ContractArgs &a, bool f32, int nchunks, const TcTables &tb, int srows,
                                    cudaStream_t st);
int contract_tc_nbuf(int rb, int srows, int want_nbuf);
int contract_tc_modes();
cudaError_t take_tc_error(int *out);
// Failure-detection test knob, read on every call: when the environment variable
// ARKCOS_TEST_WITHHOLD_MMA is set to a non-zero integer, the tensor-core kernels issue no MMA,
// so their bounded completion waits run out and the call reports ETIMEOUT through
// arkcos_sync_status.  Nothing is in flight when the waits give up.
int test_withhold_mma();
// Streaming multiprocessors of the current device (queried once per device; 152 if the query
// fails), for grid sizes that cover the GPU.
int device_sms();

}  // namespace arkcos
