// Pole-ring correction (Sec. 4.2, last paragraph): the first and last HEALPix ring (4 pixels
// each) are recomputed by the true-profile direct sum s_p = sum_q w_q f(gamma_pq) r_q over
// the input rings inside the support, and the adjoint adds the transposed sum.  FP64 squared
// chords and profile values, FP64 accumulation, deterministic block reductions.
#include <cooperative_groups.h>

#include "device_common.cuh"

namespace arkcos {

namespace {

// Half of the longitude difference (over pi) between pixel p of ring i and pixel q of ring j
// (pixels at longitudes pi (2p + hs) / n).
__device__ __forceinline__ double half_lon(const RingDev &rd, int i, int p, int j, int q)
{
    return (double)(2 * p + rd.hs[i]) / (2.0 * rd.n[i]) - (double)(2 * q + rd.hs[j]) / (2.0 * rd.n[j]);
}

// Squared chord between a pixel of the pole ring and one of the jj-th ring from that pole:
// u = 4 (B cos^2(x/2) + A sin^2(x/2)) = 4 (B + (A - B) sin^2(x/2)), A - B = sin(theta_i)
// sin(theta_j) >= 0, with the band table's A = sin^2 and B = sin^2 of the half sum and difference
// of the colatitudes (the mirror pairs of the south pole share them).
__device__ __forceinline__ double pole_chord2(const KernDev &kd, int jj, double y)
{
    const double s = sinpi(y), B = kd.B[jj];
    return 4.0 * fma(kd.A[jj] - B, s * s, B);
}

__device__ double block_sum(double v, double *red)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if (lane == 0) red[wid] = v;
    __syncthreads();
    double s = 0.0;
    if (threadIdx.x == 0)
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += red[w];
    __syncthreads();
    return s;
}

// A pixel's sum is taken in slices, each by the threads of one CTA and added in order, as many as its
// kernel's band has blocks of pixels (a power of two up to kPoleSlices): the order of the sum
// depends on the kernel alone, not on how many maps or other kernels share the launch.
constexpr int kPoleThreads = 256, kPoleSlices = 8;

__host__ __device__ inline int pole_slices(int64_t band_pixels)
{
    int s = 1;
    while (s < kPoleSlices && kPoleThreads * (int64_t)s < band_pixels) s *= 2;
    return s;
}

// Pixels of the rings of kernel kd's band about a pole.
__device__ __forceinline__ int64_t band_pixels(const RingDev &rd, const KernDev &kd)
{
    const int jh = kd.jhi[0];
    return rd.poff[jh] + rd.n[jh];
}

// Direct sum of kernel kd at pixel p of the pole ring over input map mp: this thread's share of slice
// `slice` (the slices take the pixels of the band's rings, one run of the map, in turn).
__device__ double pole_sum(const PoleArgs &a, const KernDev &kd, const float *mp, int p, int e, int slice, int slices)
{
    const int jh = kd.jhi[0], ja = e == 0 ? 0 : a.R - 1 - jh, jz = e == 0 ? jh : a.R - 1;
    const int i = e == 0 ? 0 : a.R - 1;
    const int64_t q0 = a.rd.poff[ja], q1 = a.rd.poff[jz] + a.rd.n[jz];
    double acc = 0.0;
    for (int64_t q = q0 + slice * kPoleThreads + threadIdx.x; q < q1; q += slices * kPoleThreads) {
        int j = ja, hi = jz;  // the pixel's ring
        while (j < hi) {
            const int mid = (j + hi + 1) >> 1;
            if (__ldg(&a.rd.poff[mid]) <= q) j = mid;
            else hi = mid - 1;
        }
        const double u = pole_chord2(kd, e == 0 ? j : a.R - 1 - j, half_lon(a.rd, i, p, j, (int)(q - a.rd.poff[j])));
        if (u <= kd.umax)
            acc += (double)a.rd.w[j] * profile_eval(u, kd.ut, kd.knots, kd.T, kd.gscale) * (double)__ldg(&mp[q]);
    }
    return acc;
}

// One cluster per (pixel p of the pole ring, pole e in {0: ring 0, 1: ring R-1}, map b), whose CTAs
// take its slices in turn.  It reads only the input maps and the inverse transforms leave these
// rings alone, so it runs beside their end.  FP64 arithmetic (two FMAs per SM and clock) bounds
// it: the chord from the band table and one sine per pixel, spread over more SMs, 14 us for one
// nside-2048 map with a 15' support and 21 us at a degree, launch included, against 60 and 224 us
// with three sines per pixel and a CTA per output pixel going ring by ring.
__global__ void __launch_bounds__(kPoleThreads) k_pole_fwd(const __grid_constant__ PoleArgs a)
{
    namespace cg = cooperative_groups;
    __shared__ double red[kPoleThreads / 32], part[kPoleSlices];
    auto cluster = cg::this_cluster();
    const int ranks = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
    const int p = blockIdx.x / ranks, e = blockIdx.y, b = blockIdx.z;
    const int src = a.vdiv > 1 ? (a.vbase + b) / a.vdiv : b;
    const float *mp = a.map + (int64_t)src * a.npix;
    const int kid = a.nsum > 0 || !a.per_map ? 0 : b - a.map_base;
    int64_t pixels = band_pixels(a.rd, a.kd[kid]);
    for (int k = 1; k < a.nsum; ++k) pixels = max(pixels, band_pixels(a.rd, a.kd[k]));
    const int slices = pole_slices(pixels);
    for (int s = rank; s < slices; s += ranks) {
        double acc = 0.0;
        if (a.nsum > 0) {
            // the weighted sum over several kernels of one input map, in kernel order
            for (int k = 0; k < a.nsum; ++k) acc += a.wsum[k] * pole_sum(a, a.kd[k], mp, p, e, s, slices);
        } else {
            acc = pole_sum(a, a.kd[kid], mp, p, e, s, slices);
        }
        acc = block_sum(acc, red);
        if (threadIdx.x == 0) part[s] = acc;
    }
    cluster.sync();
    if (rank == 0 && threadIdx.x == 0) {
        double acc = part[0];
        for (int s = 1; s < slices; ++s) acc += *cluster.map_shared_rank(&part[s], s % ranks);
        a.out[(int64_t)b * a.npix + a.rd.poff[e == 0 ? 0 : a.R - 1] + p] = (float)acc;
    }
    cluster.sync();
    chain_wait();
}

// grid: (ring index within the pole band, side e, map b); adds the transposed direct sum of
// both pole rings to every pixel of the band rings.
__global__ void __launch_bounds__(256) k_pole_adj(PoleArgs a)
{
    const int jj = blockIdx.x, e = blockIdx.y, b = blockIdx.z;
    const KernDev &kd = a.kd[a.per_map ? b - a.map_base : 0];
    const int jl = kd.jlo[0], jh = kd.jhi[0];
    if (jj > jh - jl) return;
    const int j = e == 0 ? jl + jj : a.R - 1 - (jl + jj);
    // a ring inside both pole bands (tiny grids) is handled once, from the north side
    if (e == 1 && a.R - 1 - j <= jh && j <= jh) return;
    const int nj = a.rd.n[j];
    const double wj = (double)a.rd.w[j];
    const float *g = a.map + (int64_t)b * a.npix;
    float *o = a.out + (int64_t)b * a.npix + a.rd.poff[j];
    for (int q = threadIdx.x; q < nj; q += blockDim.x) {
        double acc = 0.0;
        for (int side = 0; side < 2; ++side) {
            const int i = side == 0 ? 0 : a.R - 1;
            const int jn = side == 0 ? j : a.R - 1 - j;  // distance in rings from that pole
            if (jn < jl || jn > jh) continue;
            for (int p = 0; p < a.rd.n[i]; ++p) {
                const double u = pole_chord2(kd, jn, half_lon(a.rd, i, p, j, q));
                if (u <= kd.umax)
                    acc += wj * profile_eval(u, kd.ut, kd.knots, kd.T, kd.gscale) *
                           (double)__ldg(&g[a.rd.poff[i] + p]);
            }
        }
        o[q] += (float)acc;
    }
}

}  // namespace

cudaError_t launch_pole_fwd(const PoleArgs &a, int64_t band_pixels, cudaStream_t st, bool after_prev)
{
    // CTAs per cluster: one per slice, while the launch is not already some CTAs per SM
    int c = 1;
    while (c < pole_slices(band_pixels) && 16 * (int64_t)c * a.B <= 4 * device_sms()) c *= 2;
    return launch_chained(k_pole_fwd, dim3(4 * c, 2, a.B), kPoleThreads, 0, st, after_prev, c, a);
}

cudaError_t launch_pole_adj(const PoleArgs &a, int max_band_rings, cudaStream_t st)
{
    dim3 grid(max_band_rings, 2, a.B);
    k_pole_adj<<<grid, 256, 0, st>>>(a);
    return cudaGetLastError();
}

}  // namespace arkcos
