// tk_layout.cu -- moves the state between the ABI's planes [Ntheta][Nr] (the
// paper's idx(b,a) = N*b + a layout) and the device-resident column layout
// u[i][c][jp]; sets the initial momentum; finite check; waveform sums.
#include <math.h>

#include "tk_internal.h"

namespace tk {
namespace {

// The planes [Ntheta][Nr] and the state [i][c][jp] are each other's transpose:
// tiles of 32 rows by TI columns (tile_columns) go through shared memory, so that
// both sides are read and written in runs (a thread per point, one side strided,
// and a division per derived momentum took: import 125 us at 16001 x 128, 15 at
// 4001 x 64, 6.2 at 1601 x 32; now 33, 8.5, 5.2).

// Initial data (Sec. 3.2).  Pi is either given or, for zero time derivative,
// Pi = b d_* Phi with the centred difference (Phi_{i+1} - Phi_{i-1})/(2 dr*).
// Both fields vanish on the radial edges; padding rows are zero.
template <typename T, int TI>
__global__ void __launch_bounds__(kTileThreads)
import_kernel(int Nr, int Nth, int NP, Divisor d, const double *__restrict__ phr,
              const double *__restrict__ phi, const double *__restrict__ pir, const double *__restrict__ pii,
              const double *__restrict__ b_node, T *__restrict__ u)
{
    __shared__ double f[2][32][TI + 3];   // Phi of columns i0 - 1 .. i0 + TI
    __shared__ double g[2][32][TI + 1];
    const int j0 = blockIdx.x * 32, i0 = blockIdx.y * TI;
    for (int q = threadIdx.x; q < 32 * (TI + 2); q += kTileThreads) {
        const int r = q / (TI + 2), x = q % (TI + 2), jp = j0 + r, i = i0 - 1 + x;
        const bool in = jp < Nth && i >= 0 && i < Nr;
        const size_t k = (size_t)jp * Nr + i;
        f[0][r][x] = in ? phr[k] : 0.0;
        f[1][r][x] = in ? phi[k] : 0.0;
    }
    if (pir)
        for (int q = threadIdx.x; q < 32 * TI; q += kTileThreads) {
            const int r = q / TI, x = q % TI, jp = j0 + r, i = i0 + x;
            const bool in = jp < Nth && i < Nr;
            const size_t k = (size_t)jp * Nr + i;
            g[0][r][x] = in ? pir[k] : 0.0;
            g[1][r][x] = in ? pii[k] : 0.0;
        }
    __syncthreads();
    const int r = threadIdx.x & 31, jp = j0 + r;
    for (int x = threadIdx.x >> 5; x < TI; x += kTileThreads / 32) {
        const int i = i0 + x;
        if (i >= Nr) break;
        double v[4] = {0.0, 0.0, 0.0, 0.0};
        if (jp < Nth && i > 0 && i < Nr - 1) {
            v[0] = f[0][r][x + 1];
            v[1] = f[1][r][x + 1];
            if (pir) {
                v[2] = g[0][r][x];
                v[3] = g[1][r][x];
            } else {
                const double b = b_node[(size_t)i * NP + jp];
                v[2] = d.under(b * (f[0][r][x + 2] - f[0][r][x]));
                v[3] = d.under(b * (f[1][r][x + 2] - f[1][r][x]));
            }
        }
        T *col = u + (size_t)i * 4 * NP + jp;
#pragma unroll
        for (int c = 0; c < 4; ++c) col[(size_t)c * NP] = (T)v[c];
    }
}

template <typename T, int TI>
__global__ void __launch_bounds__(kTileThreads)
export_kernel(int Nr, int Nth, int NP, const T *__restrict__ u, double *__restrict__ out)
{
    __shared__ T f[4][32][TI + 1];
    const int j0 = blockIdx.x * 32, i0 = blockIdx.y * TI, lane = threadIdx.x & 31;
    for (int x = threadIdx.x >> 5; x < TI; x += kTileThreads / 32) {
        const int i = i0 + x;
        if (i >= Nr) break;
        const T *col = u + (size_t)i * 4 * NP + j0 + lane;
#pragma unroll
        for (int c = 0; c < 4; ++c) f[c][lane][x] = col[(size_t)c * NP];
    }
    __syncthreads();
    const size_t plane = (size_t)Nth * Nr;
    for (int q = threadIdx.x; q < 32 * TI; q += kTileThreads) {
        const int r = q / TI, x = q % TI, jp = j0 + r, i = i0 + x;
        if (jp >= Nth || i >= Nr) continue;
#pragma unroll
        for (int c = 0; c < 4; ++c) out[c * plane + (size_t)jp * Nr + i] = (double)f[c][r][x];
    }
}

template <typename T>
__global__ void finite_kernel(size_t n, const T *__restrict__ u, int *flag)
{
    int bad = 0;
    for (size_t k = blockIdx.x * (size_t)blockDim.x + threadIdx.x; k < n;
         k += (size_t)gridDim.x * blockDim.x)
        bad |= !isfinite((double)u[k]);
    if (__syncthreads_or(bad) && threadIdx.x == 0) atomicOr(flag, 1);
}

// Waveform read-out (the bilinear sample of Phi = w Phi^ in r* and theta).
// FP64 entries are two weighted partial sums: the sample is their sum.  FP32
// entries are the state values of the interpolation cell (WaveRead): the
// sample is formed here in FP64 by the FP64 path's own expression,
//   slot s = wr_s [(1 - fth) w_j0 Phi_{s,j0} + fth w_j0+1 Phi_{s,j0+1}],
// on the exactly converted values.
__global__ void wave_sum_kernel(const double *__restrict__ w, int64_t first, int64_t count,
                                const WaveRead r, double *__restrict__ re, double *__restrict__ im)
{
    const int64_t n = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (n >= count) return;
    const double *p = w + 4 * (first + n);
    if (r.precision == 0) {
        re[n] = p[0] + p[2];
        im[n] = p[1] + p[3];
        return;
    }
    const float4 *f = reinterpret_cast<const float4 *>(p);
    const double w0 = (1.0 - r.ft) * r.w_row[r.j0];
    const double w1 = r.ft * r.w_row[r.j0 + 1];
    double sr[2], si[2];
#pragma unroll
    for (int s = 0; s < 2; ++s) {
        const float4 v = f[s];   // Phi_R, Phi_I at row j0, then at row j0 + 1
        const double cr = w0 * (double)v.x + w1 * (double)v.z;
        const double ci = w0 * (double)v.y + w1 * (double)v.w;
        const double wr = s ? r.wr1 : r.wr0;
        sr[s] = wr * cr;
        si[s] = wr * ci;
    }
    re[n] = sr[0] + sr[1];
    im[n] = si[0] + si[1];
}

// SplitMix64 (G. L. Steele, D. Lea, C. H. Flood, "Fast splittable
// pseudorandom number generators", OOPSLA 2014) in its counter form: output k
// (k = 0, 1, ...) of seed S is the 64-bit finaliser applied to
// S + (k + 1) * 0x9E3779B97F4A7C15; a uniform double in [0, 1) is the top 53
// bits times 2^-53.
__device__ __forceinline__ double splitmix64_uniform(unsigned long long seed, unsigned long long k)
{
    unsigned long long z = seed + (k + 1ull) * 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    z ^= z >> 31;
    return (double)(z >> 11) * 0x1.0p-53;
}

// Gaussian pulse with the sin^2(theta) profile plus uniform noise, planes
// [Ntheta][Nr]: re = sin^2(theta_j) * amp * exp(-(r*_i - c)^2 / (2 w^2))
// + noise * (2 u - 1), im = noise * (2 u' - 1), with u the SplitMix64 output
// j Nr + i and u' the output Nr Ntheta + j Nr + i.  Every operation is rounded
// on its own (no contraction), so the planes agree with the same formula
// evaluated one IEEE operation at a time up to the last bits of exp and sin.
// A block takes 32 rows by 32 columns and forms the exponential once per column
// and the sine once per row (both at every point, 60 FP64 instructions, took 33
// us at 4001 x 64, now 9).
__global__ void __launch_bounds__(256)
gaussian_kernel(int Nr, int Nth, double rs_min, double drs, double dth, double amp,
                double center, double two_w2, double noise,
                unsigned long long seed, double *__restrict__ re,
                double *__restrict__ im)
{
    __shared__ double s2[32], gr[32];
    const long long P = (long long)Nr * Nth;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, i = blockIdx.x * 32 + lane, j0 = blockIdx.y * 32;
    if (w == 0) {
        const double rs = __dadd_rn(rs_min, __dmul_rn((double)i, drs));
        const double d = __dsub_rn(rs, center);
        gr[lane] = __dmul_rn(amp, exp(-__ddiv_rn(__dmul_rn(d, d), two_w2)));
    } else if (w == 1) {
        const double sn = sin(__dmul_rn(__dadd_rn((double)(j0 + lane), 0.5), dth));
        s2[lane] = __dmul_rn(sn, sn);
    }
    __syncthreads();
    if (i >= Nr) return;
    for (int r = w; r < 32 && j0 + r < Nth; r += 8) {
        const long long k = (long long)(j0 + r) * Nr + i;
        double vr = __dmul_rn(s2[r], gr[lane]), vi = 0.0;
        if (noise > 0.0) {
            const double ur = splitmix64_uniform(seed, (unsigned long long)k);
            const double ui = splitmix64_uniform(seed, (unsigned long long)(P + k));
            vr = __dadd_rn(vr, __dmul_rn(noise, __dsub_rn(__dmul_rn(2.0, ur), 1.0)));
            vi = __dmul_rn(noise, __dsub_rn(__dmul_rn(2.0, ui), 1.0));
        }
        re[k] = vr;
        im[k] = vi;
    }
}

}  // namespace

cudaError_t launch_import_state(int precision, int Nr, int Ntheta, int NP, double drs,
                                const double *phi_re, const double *phi_im, const double *pi_re,
                                const double *pi_im, const double *b_node, void *u, int num_sms,
                                cudaStream_t st)
{
    const int ti = tile_columns(Nr, NP, num_sms);
    const dim3 grid(NP / 32, (Nr + ti - 1) / ti);
    const Divisor d = divisor(2.0 * drs);
    auto go = [&](auto kern, auto *w) {
        kern<<<grid, kTileThreads, 0, st>>>(Nr, Ntheta, NP, d, phi_re, phi_im, pi_re, pi_im, b_node, w);
    };
    if (precision == 0) go(ti == 8 ? import_kernel<double, 8> : import_kernel<double, 32>, (double *)u);
    else go(ti == 8 ? import_kernel<float, 8> : import_kernel<float, 32>, (float *)u);
    return cudaGetLastError();
}

cudaError_t launch_export_state(int precision, int Nr, int Ntheta, int NP, const void *u,
                                double *planes4, int num_sms, cudaStream_t st)
{
    const int ti = tile_columns(Nr, NP, num_sms);
    const dim3 grid(NP / 32, (Nr + ti - 1) / ti);
    auto go = [&](auto kern, auto *w) { kern<<<grid, kTileThreads, 0, st>>>(Nr, Ntheta, NP, w, planes4); };
    if (precision == 0) go(ti == 8 ? export_kernel<double, 8> : export_kernel<double, 32>, (const double *)u);
    else go(ti == 8 ? export_kernel<float, 8> : export_kernel<float, 32>, (const float *)u);
    return cudaGetLastError();
}

cudaError_t launch_finite_check(int precision, size_t n, const void *u, int *flag, cudaStream_t st)
{
    const int blocks = 304, threads = 256;
    if (precision == 0)
        finite_kernel<double><<<blocks, threads, 0, st>>>(n, (const double *)u, flag);
    else
        finite_kernel<float><<<blocks, threads, 0, st>>>(n, (const float *)u, flag);
    return cudaGetLastError();
}

cudaError_t launch_wave_sum(const double *wave_obs, int64_t first, int64_t count, const WaveRead &r,
                            double *re, double *im, cudaStream_t st)
{
    if (count <= 0) return cudaSuccess;
    const int threads = 256;
    const int64_t blocks = (count + threads - 1) / threads;
    wave_sum_kernel<<<(unsigned)blocks, threads, 0, st>>>(wave_obs, first, count, r, re, im);
    return cudaGetLastError();
}

cudaError_t launch_gaussian(int Nr, int Ntheta, double rs_min, double drs, double amp,
                            double center, double width, double noise, unsigned long long seed,
                            double *re, double *im, cudaStream_t st)
{
    const dim3 grid((Nr + 31) / 32, (Ntheta + 31) / 32);
    gaussian_kernel<<<grid, 256, 0, st>>>(Nr, Ntheta, rs_min, drs, M_PI / Ntheta, amp,
                                                      center, 2.0 * (width * width), noise, seed,
                                                      re, im);
    return cudaGetLastError();
}

}  // namespace tk
