// tk_adjoint.cu -- the transpose of the fused Lax-Wendroff step, for
// gradients of waveform losses with respect to the initial data.
//
// One inner step is linear and time-invariant: u^{n+1} = A u^n, with
//   h_{i+1/2} = H(u_i, u_{i+1})                        (Eq. lw1, folded tables "half")
//   u^{n+1}_i = u^n_i + N(h_{i-1/2}, h_{i+1/2})        (Eq. lw2, folded tables "node")
// and u^{n+1} = 0 on the two radial edges.  Its transpose maps an adjoint
// state lam (dL/du^{n+1}) to mu = A^T lam (dL/du^n):
//   lam~ = lam with the edge columns set to 0,
//   eta_{i+1/2} = (dN_i/dh_{i+1/2})^T lam~_i + (dN_{i+1}/dh_{i+1/2})^T lam~_{i+1},
//   mu_i = lam~_i + (dH_{i+1/2}/du_i)^T eta_{i+1/2} + (dH_{i-1/2}/du_i)^T eta_{i-1/2},
// where every (.)^T is the transposed 4x4 block of the same folded table
// entries the forward kernel uses, and the theta-neighbour couplings (KP to
// row j+1, KM to row j-1) become KP of row j-1 and KM of row j+1.  The
// waveform sample of an outer step is linear in the state, so its loss
// gradient enters as a source on the adjoint state of that step.
//
// FP32: a warp owns all theta rows of a range of output columns and walks it
// left to right; the left-edge eta is handed over between the warps of a block.
// FP64: a team of warps does, as in the forward step, with the coupling of Pi
// to Phi in integers (tk_split_adjoint.cuh).
#include <math.h>
#include <string.h>

#include <algorithm>
#include <vector>

#include "tk_solver_impl.h"
#include "tk_split_adjoint.cuh"
#include "tk_stencil.cuh"

namespace tk {

int adj_block_bytes() { return kAdjBytes; }
int adj_block_head() { return kAdjHead; }

namespace {

struct InjectArgs {
    int on;                  // add the observation gradient of sample `sample`
    long long sample, count; // sample index; samples per observer in dwave
    const double *dwave;     // [obs][count][2]: dL/dRe W, dL/dIm W
    const double *w_row;
    ObsDev obs;
};

// Load the adjoint state of column i, add the gradient of the waveform sample
// `sample` taken at this column (if `on` and the column holds an observer),
// and zero it on the radial edges.
template <typename T, int K>
__device__ __forceinline__ void load_lam(const T *__restrict__ lam, int i, int Nr, int lane,
                                         const InjectArgs &inj, int on, long long sample, T (&l)[4][K])
{
    constexpr int NP = 32 * K;
    load_col<T, K>(lam + (size_t)i * 4 * NP + lane * K, l);
    if (on) {
        for (int k = 0; k < inj.obs.n; ++k) {
            const int slot = (i == inj.obs.i0[k]) ? 0 : ((i == inj.obs.i0[k] + 1) ? 1 : -1);
            if (slot < 0) continue;
            const int j0 = inj.obs.j0[k];
            const double wr = slot ? inj.obs.wr1[k] : inj.obs.wr0[k];
            const double *g = inj.dwave + ((size_t)k * inj.count + sample) * 2;
            const double gr = g[0], gi = g[1];
#pragma unroll
            for (int t = 0; t < K; ++t) {
                const int r = lane * K + t;
                double wt = 0.0;
                if (r == j0) wt = wr * (1.0 - inj.obs.ft[k]) * inj.w_row[j0];
                else if (r == j0 + 1) wt = wr * inj.obs.ft[k] * inj.w_row[j0 + 1];
                if (wt != 0.0) {
                    l[0][t] += (T)(wt * gr);
                    l[1][t] += (T)(wt * gi);
                }
            }
        }
    }
    if (i == 0 || i == Nr - 1) zero_col<T, K>(l);
}

// Transposed theta coupling: with the forward coupling sending KP_j x_j to
// row j+1 and KM_j x_j to row j-1, row j receives
//   KP_{j-1} x_{j-1} + KM_{j+1} x_{j+1}
// for both components xr, xi.  The coefficients and the values are shuffled
// separately, which costs two FP64 operations per component.  Row 0 has no
// row -1 and the last padded row no row below: the shuffles return the lane's
// own values there, so those coefficients are masked to zero.
template <typename T, int K>
__device__ __forceinline__ void neighbour_in(const T (&kp)[K], const T (&km)[K], const T (&xr)[K],
                                             const T (&xi)[K], T (&outr)[K], T (&outi)[K])
{
    const FmaK<T> k1 = fma_k<T>();
    const int lane = threadIdx.x & 31;
    const T kp_prv = __shfl_up_sync(kFull, kp[K - 1], 1);
    const T km_nxt = __shfl_down_sync(kFull, km[0], 1);
    T xru[K], xrd[K], xiu[K], xid[K];
    theta_neighbours<T, K>(xr, xru, xrd);
    theta_neighbours<T, K>(xi, xiu, xid);
#pragma unroll
    for (int t = 0; t < K; ++t) {
        T kpd = (t > 0) ? kp[t - 1] : kp_prv;
        T kmu = (t + 1 < K) ? km[t + 1] : km_nxt;
        if (t == 0 && lane == 0) kpd = T(0);
        if (t == K - 1 && lane == 31) kmu = T(0);
        outr[t] = fma(kpd, xrd[t], fma(kmu, xru[t], k1.nz));
        outi[t] = fma(kpd, xid[t], fma(kmu, xiu[t], k1.nz));
    }
}

// Node n's theta-neighbour sources Z_n = (KP_n lamPi_n)(j-1) + (KM_n lamPi_n)(j+1).
template <typename T, int K>
__device__ __forceinline__ void node_z(const T *__restrict__ ntab, const T (&l)[4][K],
                                       T (&zr)[K], T (&zi)[K])
{
    constexpr int NP = 32 * K;
    T kp[K], km[K];
    ldk<T, K>(ntab + N_KP * NP, kp);
    ldk<T, K>(ntab + N_KM * NP, km);
    neighbour_in<T, K>(kp, km, l[2], l[3], zr, zi);
}

// eta at the half node between nodes a (left) and c (right).
template <typename T, int K>
__device__ __forceinline__ void eta_half(const T (&la)[4][K], const T (&lc)[4][K],
                                         const T (&zar)[K], const T (&zai)[K], const T (&zcr)[K],
                                         const T (&zci)[K], const T *__restrict__ ta,
                                         const T *__restrict__ tc, const T E, T (&h)[4][K])
{
    const FmaK<T> k1 = fma_k<T>();
    constexpr int NP = 32 * K;
    T B[K], FR[K], FI[K], PR[K], CI[K];
    // left node: the half node is its h+ (coefficients -B, FP, PPR, C2I)
    ldk<T, K>(ta + N_B * NP, B);
    ldk<T, K>(ta + N_FPR * NP, FR);
    ldk<T, K>(ta + N_FPI * NP, FI);
    ldk<T, K>(ta + N_PPR * NP, PR);
    ldk<T, K>(ta + N_C2I * NP, CI);
#pragma unroll
    for (int t = 0; t < K; ++t) {
        h[0][t] = fma(FI[t], la[3][t], fma(FR[t], la[2][t], fma(-B[t], la[0][t], fma(zar[t], k1.one, zcr[t]))));
        h[1][t] = fma(FR[t], la[3][t], fma(-FI[t], la[2][t], fma(-B[t], la[1][t], fma(zai[t], k1.one, zci[t]))));
        h[2][t] = fma(CI[t], la[3][t], fma(PR[t], la[2][t], fma(E, la[0][t], k1.nz)));
        h[3][t] = fma(PR[t], la[3][t], fma(-CI[t], la[2][t], fma(E, la[1][t], k1.nz)));
    }
    // right node: the half node is its h- (coefficients +B, FM, PMR, C2I)
    ldk<T, K>(tc + N_B * NP, B);
    ldk<T, K>(tc + N_FMR * NP, FR);
    ldk<T, K>(tc + N_FMI * NP, FI);
    ldk<T, K>(tc + N_PMR * NP, PR);
    ldk<T, K>(tc + N_C2I * NP, CI);
#pragma unroll
    for (int t = 0; t < K; ++t) {
        h[0][t] = fma(FI[t], lc[3][t], fma(FR[t], lc[2][t], fma(B[t], lc[0][t], h[0][t])));
        h[1][t] = fma(FR[t], lc[3][t], fma(-FI[t], lc[2][t], fma(B[t], lc[1][t], h[1][t])));
        h[2][t] = fma(CI[t], lc[3][t], fma(PR[t], lc[2][t], fma(E, lc[0][t], h[2][t])));
        h[3][t] = fma(PR[t], lc[3][t], fma(-CI[t], lc[2][t], fma(E, lc[1][t], h[3][t])));
    }
}

// Half node's theta-neighbour sources Y_h = (KP_h etaPi)(j-1) + (KM_h etaPi)(j+1).
template <typename T, int K>
__device__ __forceinline__ void half_y(const T *__restrict__ htab, const T (&h)[4][K],
                                       T (&yr)[K], T (&yi)[K])
{
    constexpr int NP = 32 * K;
    T kp[K], km[K];
    ldk<T, K>(htab + H_KP * NP, kp);
    ldk<T, K>(htab + H_KM * NP, km);
    neighbour_in<T, K>(kp, km, h[2], h[3], yr, yi);
}

// mu at node i from lam~_i, eta+ (half node i+1/2: u_i is its "a") and eta-
// (half node i-1/2: u_i is its "c").
template <typename T, int K>
__device__ __forceinline__ void mu_node(const T (&l)[4][K], const T (&ep)[4][K],
                                        const T (&em)[4][K], const T (&ypr)[K], const T (&ypi)[K],
                                        const T (&ymr)[K], const T (&ymi)[K],
                                        const T *__restrict__ hp_tab, const T *__restrict__ hm_tab,
                                        T (&mu)[4][K])
{
    const FmaK<T> k1 = fma_k<T>();
    constexpr int NP = 32 * K;
    T S[K], FR[K], FI[K], PR[K], PI[K];
    // eta+ with the "a" entries of half node i+1/2
    ldk<T, K>(hp_tab + H_HP * NP, S);
    ldk<T, K>(hp_tab + H_FAR * NP, FR);
    ldk<T, K>(hp_tab + H_FAI * NP, FI);
    ldk<T, K>(hp_tab + H_PAR * NP, PR);
    ldk<T, K>(hp_tab + H_PI * NP, PI);
#pragma unroll
    for (int t = 0; t < K; ++t) {
        mu[0][t] = fma(FI[t], ep[3][t], fma(FR[t], ep[2][t], fma(S[t], ep[0][t],
                       fma(l[0][t], k1.one, fma(ypr[t], k1.one, ymr[t])))));
        mu[1][t] = fma(FR[t], ep[3][t], fma(-FI[t], ep[2][t], fma(S[t], ep[1][t],
                       fma(l[1][t], k1.one, fma(ypi[t], k1.one, ymi[t])))));
        mu[2][t] = fma(PI[t], ep[3][t], fma(PR[t], ep[2][t], fma(ep[0][t], k1.one, l[2][t])));
        mu[3][t] = fma(PR[t], ep[3][t], fma(-PI[t], ep[2][t], fma(ep[1][t], k1.one, l[3][t])));
    }
    // eta- with the "c" entries of half node i-1/2
    ldk<T, K>(hm_tab + H_HQ * NP, S);
    ldk<T, K>(hm_tab + H_FCR * NP, FR);
    ldk<T, K>(hm_tab + H_FCI * NP, FI);
    ldk<T, K>(hm_tab + H_PCR * NP, PR);
    ldk<T, K>(hm_tab + H_PI * NP, PI);
#pragma unroll
    for (int t = 0; t < K; ++t) {
        mu[0][t] = fma(FI[t], em[3][t], fma(FR[t], em[2][t], fma(S[t], em[0][t], mu[0][t])));
        mu[1][t] = fma(FR[t], em[3][t], fma(-FI[t], em[2][t], fma(S[t], em[1][t], mu[1][t])));
        mu[2][t] = fma(PI[t], em[3][t], fma(PR[t], em[2][t], fma(em[0][t], k1.one, mu[2][t])));
        mu[3][t] = fma(PR[t], em[3][t], fma(-PI[t], em[2][t], fma(em[1][t], k1.one, mu[3][t])));
    }
}

// Warps per block of the wide launch (one block per SM): the most warps, in
// multiples of four, whose registers fit in the register file at the count
// the kernel compiles to for this element type and K (FP64: 128 whatever K).
template <typename T, int K>
constexpr int adj_wide_warps()
{
    return sizeof(T) == 8 ? 16 : (K == 1 ? 32 : K == 2 ? 24 : 12);
}

// Shared memory per warp, in theta-columns of NP values: [0, 6) eta at the
// warp's last half node with its neighbour sources (read by the right
// neighbour), [6, 16) lam~, eta+ and its sources at the warp's first column
// (its deferred node).
constexpr int kAdjShared = 16;

template <typename T, int K, int W>
__global__ void __launch_bounds__(W * 32, adj_wide_warps<T, K>() / W)
lw_adjoint_kernel(const T *__restrict__ lam, T *__restrict__ mu_out, const T *__restrict__ half,
                  const T *__restrict__ node, int Nr, T eh, T en, const InjectArgs inj)
{
    constexpr int NP = 32 * K;
    constexpr size_t SP = 4 * NP, HP = (size_t)kNCH * NP, NQ = (size_t)kNCN * NP;
    extern __shared__ __align__(16) unsigned char sh_raw[];
    chain_start();   // lam is the previous launch's output
    T(*sh)[kAdjShared][NP] = reinterpret_cast<T(*)[kAdjShared][NP]>(sh_raw);
    const int lane = threadIdx.x & 31;
    const int wib = threadIdx.x >> 5;
    int i0, i1, left;
    warp_range<W>(Nr, wib, &i0, &i1, &left);
    const int row = lane * K;
    const bool lead = (left < 0);

    T la[4][K], zar[K], zai[K];        // node i: lam~ and its neighbour sources
    T em[4][K], ymr[K], ymi[K];        // half node i-1/2: eta and its neighbour sources
    zero_col<T, K>(em);
#pragma unroll
    for (int t = 0; t < K; ++t) ymr[t] = ymi[t] = T(0);
    if (i1 > i0) {
        load_lam<T, K>(lam, i0, Nr, lane, inj, inj.on, inj.sample, la);
        node_z<T, K>(node + (size_t)i0 * NQ + row, la, zar, zai);
        if (lead && i0 > 0) {
            T ll[4][K], zlr[K], zli[K];
            load_lam<T, K>(lam, i0 - 1, Nr, lane, inj, inj.on, inj.sample, ll);
            node_z<T, K>(node + (size_t)(i0 - 1) * NQ + row, ll, zlr, zli);
            eta_half<T, K>(ll, la, zlr, zli, zar, zai, node + (size_t)(i0 - 1) * NQ + row,
                           node + (size_t)i0 * NQ + row, en, em);
            half_y<T, K>(half + (size_t)(i0 - 1) * HP + row, em, ymr, ymi);
        }
        for (int i = i0; i < i1; ++i) {
            T lc[4][K], zcr[K], zci[K], ep[4][K], ypr[K], ypi[K];
            if (i + 1 < Nr) {
                load_lam<T, K>(lam, i + 1, Nr, lane, inj, inj.on, inj.sample, lc);
                node_z<T, K>(node + (size_t)(i + 1) * NQ + row, lc, zcr, zci);
                eta_half<T, K>(la, lc, zar, zai, zcr, zci, node + (size_t)i * NQ + row,
                               node + (size_t)(i + 1) * NQ + row, en, ep);
                half_y<T, K>(half + (size_t)i * HP + row, ep, ypr, ypi);
            } else {
                zero_col<T, K>(lc);
                zero_col<T, K>(ep);
#pragma unroll
                for (int t = 0; t < K; ++t) zcr[t] = zci[t] = ypr[t] = ypi[t] = T(0);
            }
            if (i == i0 && !lead) {
#pragma unroll
                for (int t = 0; t < K; ++t) {
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        sh[wib][6 + c][row + t] = la[c][t];
                        sh[wib][10 + c][row + t] = ep[c][t];
                    }
                    sh[wib][14][row + t] = ypr[t];
                    sh[wib][15][row + t] = ypi[t];
                }
            } else {
                T mu[4][K];
                const T *hm_tab = half + (size_t)(i > 0 ? i - 1 : 0) * HP + row;
                mu_node<T, K>(la, ep, em, ypr, ypi, ymr, ymi, half + (size_t)i * HP + row, hm_tab, mu);
                store_col<T, K>(mu_out + (size_t)i * SP + row, mu);
            }
#pragma unroll
            for (int c = 0; c < 4; ++c)
#pragma unroll
                for (int t = 0; t < K; ++t) {
                    la[c][t] = lc[c][t];
                    em[c][t] = ep[c][t];
                }
#pragma unroll
            for (int t = 0; t < K; ++t) {
                zar[t] = zcr[t];
                zai[t] = zci[t];
                ymr[t] = ypr[t];
                ymi[t] = ypi[t];
            }
        }
    }
    // em, ymr, ymi now belong to the half node i1 - 1/2: the right neighbour's left edge
#pragma unroll
    for (int t = 0; t < K; ++t) {
#pragma unroll
        for (int c = 0; c < 4; ++c) sh[wib][c][row + t] = em[c][t];
        sh[wib][4][row + t] = ymr[t];
        sh[wib][5][row + t] = ymi[t];
    }
    __syncthreads();
    if (!lead && i1 > i0) {
        T l0[4][K], ep[4][K], el[4][K], ypr[K], ypi[K], yml[K], ymli[K], mu[4][K];
#pragma unroll
        for (int t = 0; t < K; ++t) {
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                el[c][t] = sh[left][c][row + t];
                l0[c][t] = sh[wib][6 + c][row + t];
                ep[c][t] = sh[wib][10 + c][row + t];
            }
            yml[t] = sh[left][4][row + t];
            ymli[t] = sh[left][5][row + t];
            ypr[t] = sh[wib][14][row + t];
            ypi[t] = sh[wib][15][row + t];
        }
        mu_node<T, K>(l0, ep, el, ypr, ypi, yml, ymli, half + (size_t)i0 * HP + row,
                      half + (size_t)(i0 - 1) * HP + row, mu);
        store_col<T, K>(mu_out + (size_t)i0 * SP + row, mu);
    }
}

// FP32: every adjoint step of a tk_adjoint call in one cooperative launch, no
// barrier between steps; each warp waits (bounded) only for its two siblings and,
// at a block's edges, the neighbouring block's edge warp.  Step s:
//   - first phase (every half node and node that involves only the block's
//     columns): it reads the right sibling's first column and overwrites its
//     own last half node, which that sibling read in the last step, so it
//     waits until that sibling has finished step s - 1;
//   - the block's last warp waits until the right neighbouring block's first
//     warp has finished step s - 1, then forms its last column;
//   - the deferred first node: the block's first warp waits until the left
//     neighbouring block's last warp has finished step s - 1 and forms its
//     left half node from that warp's column; every other warp takes its left
//     sibling's last half node once that sibling's first phase is done.
// Same arithmetic on the same operands as lw_adjoint_kernel.
template <typename T, int K, int W>
__device__ __forceinline__ void adj_sweep_async(unsigned char *sh_raw, const T *__restrict__ lam,
                                                T *__restrict__ mu_out, const T *__restrict__ half,
                                                const T *__restrict__ node, int Nr, T en, const InjectArgs &inj,
                                                int on, long long sample, unsigned int *flags,
                                                unsigned int *first_done, unsigned int *step_done, unsigned int s,
                                                int *err)
{
    constexpr int NP = 32 * K;
    constexpr size_t SP = 4 * NP, HP = (size_t)kNCH * NP, NQ = (size_t)kNCN * NP;
    T(*sh)[kAdjShared][NP] = reinterpret_cast<T(*)[kAdjShared][NP]>(sh_raw);
    const int lane = threadIdx.x & 31;
    const int wib = threadIdx.x >> 5;
    int i0, i1, left;
    warp_range<W>(Nr, wib, &i0, &i1, &left);
    // at most Nr / W blocks: every warp has a column (as in step_sweep_async)
    if (i1 <= i0) return;
    const int row = lane * K;
    const bool lead = (left < 0);
    const int b1 = (int)(((long long)(blockIdx.x + 1) * Nr) / gridDim.x);
    const bool last = (i1 == b1);
    const int iend = last ? i1 - 1 : i1;
    const unsigned int nb = gridDim.x;
    if (s > 0 && !last) warp_wait_cta(&step_done[wib + 1], s, err);

    T la[4][K], zar[K], zai[K];        // node i: lam~ and its neighbour sources
    T em[4][K], ymr[K], ymi[K];        // half node i-1/2: eta and its neighbour sources
    zero_col<T, K>(em);
#pragma unroll
    for (int t = 0; t < K; ++t) ymr[t] = ymi[t] = T(0);
    load_lam<T, K>(lam, i0, Nr, lane, inj, on, sample, la);
    node_z<T, K>(node + (size_t)i0 * NQ + row, la, zar, zai);
    // the right half node of column i (from column i + 1) and, for i > i0, its node
    auto column = [&](int i) {
        T lc[4][K], zcr[K], zci[K], ep[4][K], ypr[K], ypi[K];
        if (i + 1 < Nr) {
            load_lam<T, K>(lam, i + 1, Nr, lane, inj, on, sample, lc);
            node_z<T, K>(node + (size_t)(i + 1) * NQ + row, lc, zcr, zci);
            eta_half<T, K>(la, lc, zar, zai, zcr, zci, node + (size_t)i * NQ + row,
                           node + (size_t)(i + 1) * NQ + row, en, ep);
            half_y<T, K>(half + (size_t)i * HP + row, ep, ypr, ypi);
        } else {
            zero_col<T, K>(lc);
            zero_col<T, K>(ep);
#pragma unroll
            for (int t = 0; t < K; ++t) zcr[t] = zci[t] = ypr[t] = ypi[t] = T(0);
        }
        if (i == i0) {
#pragma unroll
            for (int t = 0; t < K; ++t) {
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    sh[wib][6 + c][row + t] = la[c][t];
                    sh[wib][10 + c][row + t] = ep[c][t];
                }
                sh[wib][14][row + t] = ypr[t];
                sh[wib][15][row + t] = ypi[t];
            }
        } else {
            T mu[4][K];
            mu_node<T, K>(la, ep, em, ypr, ypi, ymr, ymi, half + (size_t)i * HP + row,
                          half + (size_t)(i - 1) * HP + row, mu);
            store_col<T, K>(mu_out + (size_t)i * SP + row, mu);
        }
#pragma unroll
        for (int c = 0; c < 4; ++c)
#pragma unroll
            for (int t = 0; t < K; ++t) {
                la[c][t] = lc[c][t];
                em[c][t] = ep[c][t];
            }
#pragma unroll
        for (int t = 0; t < K; ++t) {
            zar[t] = zcr[t];
            zai[t] = zci[t];
            ymr[t] = ypr[t];
            ymi[t] = ypi[t];
        }
    };
    for (int i = i0; i < iend; ++i) column(i);
    if (!last)   // eta at i1 - 1/2 with its sources: the right sibling's left edge
#pragma unroll
        for (int t = 0; t < K; ++t) {
#pragma unroll
            for (int c = 0; c < 4; ++c) sh[wib][c][row + t] = em[c][t];
            sh[wib][4][row + t] = ymr[t];
            sh[wib][5][row + t] = ymi[t];
        }
    warp_publish_cta(&first_done[wib], s + 1);
    if (last) {
        if (s > 0 && blockIdx.x + 1 < nb) warp_wait_flag(flags + blockIdx.x + 1, s, err);
        column(i1 - 1);
        __syncwarp();
    }
    {   // the deferred first node
        T l0[4][K], ep[4][K], el[4][K], ypr[K], ypi[K], yml[K], ymli[K], mu[4][K];
#pragma unroll
        for (int t = 0; t < K; ++t) {
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                l0[c][t] = sh[wib][6 + c][row + t];
                ep[c][t] = sh[wib][10 + c][row + t];
            }
            ypr[t] = sh[wib][14][row + t];
            ypi[t] = sh[wib][15][row + t];
        }
        if (lead) {
            if (s > 0 && blockIdx.x > 0) warp_wait_flag(flags + nb + blockIdx.x - 1, s, err);
            if (i0 > 0) {
                T ll[4][K], zlr[K], zli[K], z0r[K], z0i[K];
                load_lam<T, K>(lam, i0 - 1, Nr, lane, inj, on, sample, ll);
                node_z<T, K>(node + (size_t)(i0 - 1) * NQ + row, ll, zlr, zli);
                node_z<T, K>(node + (size_t)i0 * NQ + row, l0, z0r, z0i);
                eta_half<T, K>(ll, l0, zlr, zli, z0r, z0i, node + (size_t)(i0 - 1) * NQ + row,
                               node + (size_t)i0 * NQ + row, en, el);
                half_y<T, K>(half + (size_t)(i0 - 1) * HP + row, el, yml, ymli);
            } else {
                zero_col<T, K>(el);
#pragma unroll
                for (int t = 0; t < K; ++t) yml[t] = ymli[t] = T(0);
            }
        } else {
            warp_wait_cta(&first_done[left], s + 1, err);
#pragma unroll
            for (int t = 0; t < K; ++t) {
#pragma unroll
                for (int c = 0; c < 4; ++c) el[c][t] = sh[left][c][row + t];
                yml[t] = sh[left][4][row + t];
                ymli[t] = sh[left][5][row + t];
            }
        }
        mu_node<T, K>(l0, ep, el, ypr, ypi, yml, ymli, half + (size_t)i0 * HP + row,
                      half + (size_t)(i0 > 0 ? i0 - 1 : 0) * HP + row, mu);
        store_col<T, K>(mu_out + (size_t)i0 * SP + row, mu);
    }
    if (lead) warp_publish_gpu(flags + blockIdx.x, s + 1);
    if (last) warp_publish_gpu(flags + nb + blockIdx.x, s + 1);
    warp_publish_cta(&step_done[wib], s + 1);
}

// (FP32) Launch step s is the transpose of inner step n_inner - 1 - s: the gradient
// of sample count - 1 - s / substeps is injected at its first sub-step.  The
// adjoint state starts in a0; the result is in a0 or a1 by the parity of
// n_inner.
template <typename T, int K, int W>
__global__ void __launch_bounds__(W * 32, adj_wide_warps<T, K>() / W)
lw_adjoint_persistent_kernel(T *a0, T *a1, const T *__restrict__ half, const T *__restrict__ node, int Nr,
                             T en, const InjectArgs inj, int inject, long long n_inner, int substeps,
                             unsigned int *flags, int *err)
{
    extern __shared__ __align__(16) unsigned char sh_raw[];
    __shared__ unsigned int first_done[W], step_done[W];
    if (threadIdx.x < W) {
        first_done[threadIdx.x] = 0;
        step_done[threadIdx.x] = 0;
    }
    __syncthreads();
    for (long long s = 0; s < n_inner; ++s) {
        const T *lam = (s & 1) ? a1 : a0;
        T *mu = (s & 1) ? a0 : a1;
        adj_sweep_async<T, K, W>(sh_raw, lam, mu, half, node, Nr, en, inj, inject && (s % substeps == 0),
                                 inj.count - 1 - s / substeps, flags, first_done, step_done, (unsigned)s, err);
    }
}

// ---- FP64: teams of warps and integer coupling (tk_split_adjoint.cuh) ----

// load_lam for one row per lane: the waveform gradient and the radial edges on a
// loaded column.
__device__ __forceinline__ void inject_row(int i, int Nr, int row, const InjectArgs &inj, int on, long long sample,
                                           double (&l)[4])
{
    if (on) {
        for (int k = 0; k < inj.obs.n; ++k) {
            const int slot = (i == inj.obs.i0[k]) ? 0 : ((i == inj.obs.i0[k] + 1) ? 1 : -1);
            if (slot < 0) continue;
            const int j0 = inj.obs.j0[k];
            const double wr = slot ? inj.obs.wr1[k] : inj.obs.wr0[k];
            const double *g = inj.dwave + ((size_t)k * inj.count + sample) * 2;
            double wt = 0.0;
            if (row == j0) wt = wr * (1.0 - inj.obs.ft[k]) * inj.w_row[j0];
            else if (row == j0 + 1) wt = wr * inj.obs.ft[k] * inj.w_row[j0 + 1];
            if (wt != 0.0) {
                l[0] += wt * g[0];
                l[1] += wt * g[1];
            }
        }
    }
    if (i == 0 || i == Nr - 1)
#pragma unroll
        for (int c = 0; c < 4; ++c) l[c] = 0.0;
}

template <int K>
__device__ __forceinline__ void load_lam_row(const double *__restrict__ lam, int i, int Nr, int row,
                                             const InjectArgs &inj, int on, long long sample, double (&l)[4])
{
    constexpr int NP = 32 * K;
#pragma unroll
    for (int c = 0; c < 4; ++c) l[c] = __ldcg(lam + (size_t)i * (4 * NP) + c * NP + row);
    inject_row(i, Nr, row, inj, on, sample, l);
}

template <int K>
__device__ __forceinline__ void store_row(double *__restrict__ u, int i, int row, const double (&o)[4])
{
    constexpr int NP = 32 * K;
#pragma unroll
    for (int c = 0; c < 4; ++c) u[(size_t)i * (4 * NP) + c * NP + row] = o[c];
}

template <int K, int W>
__global__ void __launch_bounds__(W * 32, adj_wide_warps<double, K>() / W)
lw_adjoint_team_kernel(const double *__restrict__ lam, double *__restrict__ mu_out, const double *__restrict__ half,
                       const double *__restrict__ node, const unsigned char *__restrict__ tab, size_t pitch, int Nr,
                       double en, const InjectArgs inj, int *err)
{
    extern __shared__ __align__(16) unsigned char sh_raw[];
    __shared__ unsigned long long bars[W][2];
    __shared__ AdjRows rows[W];
    chain_start();   // lam is the previous launch's output
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5, t = wib / K, h = wib % K, row = 32 * h + lane;
    split_ring_init(bars[wib], lane);
    AdjTeam<K> team{rows + t * K, h, lane, 1 + t};
    const AdjSweep<K> sw{reinterpret_cast<AdjRing *>(sh_raw) + wib, bars[wib], tab + h * kAdjBytes, half, node, Nr,
                         en, err, pitch};
    int i0, i1;
    team_range<W, K>(Nr, t, &i0, &i1);
    SplitRingState st;
    if (i1 > i0)
        sw.run(
            st, team,
            [&](int i, double (&l)[4]) { load_lam_row<K>(lam, i, Nr, row, inj, inj.on, inj.sample, l); }, i0, i1,
            false, [] {}, [&](int i, const double (&o)[4]) { store_row<K>(mu_out, i, row, o); });
    sw.drain(st);
}

// Every adjoint step of a tk_adjoint call in one cooperative launch, with the
// waits of the forward persistent sweep (lw_persistent_kernel).  Launch step s
// is the transpose of inner step n_inner - 1 - s, as in
// lw_adjoint_persistent_kernel.
template <int K, int W>
__global__ void __launch_bounds__(W * 32, adj_wide_warps<double, K>() / W)
lw_adjoint_team_persistent_kernel(double *a0, double *a1, const double *__restrict__ half,
                                  const double *__restrict__ node, const unsigned char *__restrict__ tab, size_t pitch,
                                  int Nr, double en, const InjectArgs inj, int inject, long long n_inner, int substeps,
                                  unsigned int *flags, int *err)
{
    extern __shared__ __align__(16) unsigned char sh_raw[];
    __shared__ unsigned int step_done[W];
    __shared__ unsigned long long bars[W][2];
    __shared__ AdjRows rows[W];
    constexpr int TEAMS = W / K;
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5, t = wib / K, h = wib % K, row = 32 * h + lane;
    if (threadIdx.x < W) step_done[threadIdx.x] = 0;
    split_ring_init(bars[wib], lane);
    __syncthreads();
    const int nb = (int)gridDim.x, b = (int)blockIdx.x;
    AdjTeam<K> team{rows + t * K, h, lane, 1 + t};
    const AdjSweep<K> sw{reinterpret_cast<AdjRing *>(sh_raw) + wib, bars[wib], tab + h * kAdjBytes, half, node, Nr,
                         en, err, pitch};
    int i0, i1;
    team_range<W, K>(Nr, t, &i0, &i1);   // at most Nr / TEAMS blocks: every team has a column
    SplitRingState st;
    for (long long s = 0; s < n_inner; ++s) {
        const double *lam = (s & 1) ? a1 : a0;
        double *mu = (s & 1) ? a0 : a1;
        const int on = inject && (s % substeps == 0);
        const long long sample = inj.count - 1 - s / substeps;
        const unsigned int e = (unsigned int)s;
        if (s > 0) {
            if (t > 0) warp_wait_cta(&step_done[wib - K], e, err);
            else if (b > 0) warp_wait_flag(flags + (nb + b - 1) * K + h, e, err);
        }
        sw.run(
            st, team, [&](int i, double (&l)[4]) { load_lam_row<K>(lam, i, Nr, row, inj, on, sample, l); }, i0, i1,
            s + 1 < n_inner,
            [&] {
                if (s == 0) return;
                if (t + 1 < TEAMS) warp_wait_cta(&step_done[wib + K], e, err);
                else if (b + 1 < nb) warp_wait_flag(flags + (b + 1) * K + h, e, err);
            },
            [&](int i, const double (&o)[4]) { store_row<K>(mu, i, row, o); });
        if (t == 0) warp_publish_gpu(flags + b * K + h, e + 1);
        if (t == TEAMS - 1) warp_publish_gpu(flags + (nb + b) * K + h, e + 1);
        warp_publish_cta(&step_done[wib], e + 1);
    }
    sw.drain(st);
}

// The same on grids with no more columns than the chip holds teams: lw_column_kernel
// transposed.  A block has T columns and T + 1 teams; team j owns column T b - 1 +
// j (j > 0) and forms eta at the half node to its right.  A column's sums are
// formed once, by its owner (the block's outer neighbours' by the teams at its
// ends), and the one to the left goes to the left team through shared memory with
// lam~; eta and its sum to the right go to the right team for mu.  Two block
// barriers a step; tables and columns stay in the SM.  us per step, this launch
// (lw_adjoint_team_persistent_kernel, one or two columns per team): 1601 x 32 6.2
// (10.0), 1824 x 32 6.2 (9.3 at 1825), 912 x 64 7.0 (9.6), 456 x 128 7.8 (10.9).
// Bound by the chain pair - barrier - eta - pair - barrier - mu and by the FP64
// pipe of the SMs with four blocks.  first: launch step s is the transposed step
// first + s of the call; stride != 0: step s writes the whole level to a1 + s
// stride, a0 stays.
constexpr int kAdjColumns = 3;

template <int K>
struct AdjColumnShared {
    static constexpr int T = kAdjColumns, NP = 32 * K;
    alignas(16) unsigned char tab[T + 2][K][kAdjBytes];   // of columns T b - 2 ..
    double lam[T + 1][4][NP], eta[T + 1][4][NP];
    long long sum[2][T + 1][2][NP];                       // of lam~ to the left, of eta to the right
    int exp[2][T + 1][2][NP];
    int hot[2][T + 1];
    AdjRows rows[(T + 1) * K];
    unsigned long long bars[(T + 1) * K];
};

template <int K>
__global__ void __launch_bounds__((kAdjColumns + 1) * K * 32, 4 / K)
lw_adjoint_column_kernel(double *a0, double *a1, const double *__restrict__ half, const double *__restrict__ node,
                         const unsigned char *__restrict__ tab, size_t pitch, int Nr, double en,
                         const InjectArgs inj, int inject,
                         long long n_inner, int substeps, unsigned int *flags, int *err, long long first,
                         size_t stride)
{
    constexpr int T = kAdjColumns, NP = 32 * K;
    extern __shared__ __align__(16) unsigned char sh_raw[];
    AdjColumnShared<K> &sh = *reinterpret_cast<AdjColumnShared<K> *>(sh_raw);
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5, j = wib / K, h = wib % K, row = 32 * h + lane;
    const int nb = (int)gridDim.x, b = (int)blockIdx.x, col = b * T - 1 + j;
    const bool owner = j > 0 && col < Nr;              // of a column
    const bool halves = col >= 0 && col + 1 < Nr;      // there is a half node right of it
    const bool before = col > 0 && col < Nr;           // and one left of it
    const FmaK<double> k1 = fma_k<double>();
    AdjTeam<K> team{sh.rows + j * K, h, lane, 1 + j};
    const unsigned char *left = sh.tab[j][h], *own = sh.tab[j + 1][h];   // of columns col - 1 and col
    auto put = [&](double (*p)[NP], const double (&x)[4]) {
#pragma unroll
        for (int k = 0; k < 4; ++k) p[k][row] = x[k];
    };
    auto get = [&](const double (*p)[NP], double (&x)[4]) {
#pragma unroll
        for (int k = 0; k < 4; ++k) x[k] = p[k][row];
    };
    auto put_sums = [&](int w, const AdjSums &s, bool hot) {
#pragma unroll
        for (int g = 0; g < 2; ++g) {
            sh.sum[w][j][g][row] = s.T[g];
            sh.exp[w][j][g][row] = s.O[g];
        }
        if (row == 0) sh.hot[w][j] = hot;
    };
    auto get_sums = [&](int w, int t, AdjSums &s) {
#pragma unroll
        for (int g = 0; g < 2; ++g) {
            s.T[g] = sh.sum[w][t][g][row];
            s.O[g] = sh.exp[w][t][g][row];
        }
        return sh.hot[w][t] != 0;
    };
    const bool extra = j == 0 && before;               // the block left of the first
    bool lost = false;                                 // the tables did not come
    if (halves || extra) {
        if (lane == 0) {
            unsigned long long *bar = &sh.bars[wib];
            mbar_init(bar);
            mbar_init_fence();
            mbar_expect(bar, ((halves ? 1 : 0) + (extra ? 1 : 0)) * kAdjBytes);
            if (halves) bulk_fetch(sh.tab[j + 1][h], tab + col * pitch + h * kAdjBytes, kAdjBytes, bar);
            if (extra) bulk_fetch(sh.tab[0][h], tab + (col - 1) * pitch + h * kAdjBytes, kAdjBytes, bar);
        }
        __syncwarp();
        lost = !warp_mbar_wait(&sh.bars[wib], 0, ErrWord{err});
    }
    double a[4];   // the column's adjoint state
#pragma unroll
    for (int k = 0; k < 4; ++k) a[k] = owner ? __ldcg(a0 + (size_t)col * (4 * NP) + k * NP + row) : 0.0;
    __syncthreads();
#pragma unroll 1
    for (long long s = 0; s < n_inner; ++s) {
        const double *in = stride ? (s > 0 ? a1 + (s - 1) * stride : a0) : (s & 1) ? a1 : a0;
        double *out = stride ? a1 + s * stride : (s & 1) ? a0 : a1;
        const int on = inject && ((first + s) % substeps == 0);
        const long long sample = inj.count - 1 - (first + s) / substeps;
        const unsigned int e = (unsigned int)s;
        // lam~ and its sums
        AdjSums sa, sl;
        adj_zero(sa);
        adj_zero(sl);
        bool hot_a = false;
        if (j == 0 && halves) {
            if (s > 0) warp_wait_flag(flags + (nb + b - 1) * K + h, e, err);
            load_lam_row<K>(in, col, Nr, row, inj, on, sample, a);
        } else if (owner) {
            inject_row(col, Nr, row, inj, on, sample, a);
        }
        if (before && (owner || halves)) {
            const AdjTab<false> t{left, lane};
            hot_a = adj_pair<K, false>(a, t, t.head(), team, sa, sl);
        }
        put(sh.lam[j], a);
        put_sums(0, sl, hot_a);
        double c[4];
        AdjSums sr;
        bool hot_c = false;
        const int2 head = halves ? AdjTab<false>{own, lane}.head() : make_int2(0, 0);
        const bool imag = head.y != 0;
        if (j == T && halves) {
            if (s > 0) warp_wait_flag(flags + (b + 1) * K + h, e, err);
            load_lam_row<K>(in, col + 1, Nr, row, inj, on, sample, c);
            AdjSums unused;
            hot_c = adj_pair<K, false>(c, AdjTab<false>{own, lane}, head, team, unused, sr);
        }
        __syncthreads();
        // eta
        double ep[4];
        AdjSums s1, s2;
        bool hot_p = false;
        if (halves) {
            if (j < T) {
                get(sh.lam[j + 1], c);
                hot_c = get_sums(0, j + 1, sr);
            }
            if (hot_a || hot_c)
                eta_row_cold<K>(a, c, node + (size_t)col * (kNCN * NP) + row, en, team, ep);
            else
                eta_row(a, c, sa, sr, imag, own, lane, en, k1, ep);
            hot_p = adj_pair<K, true>(ep, AdjTab<true>{own, lane}, head, team, s1, s2);
            put(sh.eta[j], ep);
            put_sums(1, s2, hot_p);
        }
        __syncthreads();
        // mu
        if (owner) {
            if (col > 0 && halves) {
                double em[4], o[4];
                AdjSums sm;
                get(sh.eta[j - 1], em);
                const bool hot_m = get_sums(1, j - 1, sm);
                if (hot_p || hot_m)
                    mu_row_cold<K>(a, ep, em, half + (size_t)col * (kNCH * NP) + row, team, o);
                else
                    mu_row(a, ep, em, s1, sm, imag, own, lane, k1, o);
#pragma unroll
                for (int k = 0; k < 4; ++k) a[k] = o[k];
            } else {   // a radial edge
#pragma unroll
                for (int k = 0; k < 4; ++k) a[k] = 0.0;
            }
            if (j == 1 || j == T || s + 1 == n_inner || stride) store_row<K>(out, col, row, a);
            if (j == 1) warp_publish_gpu(flags + b * K + h, e + 1);
            if (j == T) warp_publish_gpu(flags + (nb + b) * K + h, e + 1);
        }
    }
    if (lost) mbar_wait(&sh.bars[wib], 0);
}

// Transpose of the initial-data map of tk_set_initial_data: the adjoint state
// lam0 = dL/du^0 (device layout) to dL/d(input planes) in [Ntheta][Nr].
// independent_pi: the momentum planes were given (4 output planes); else
// Pi_m = b_m (Phi_{m+1} - Phi_{m-1}) / (2 dr*) at interior m (2 output planes).
// Tiles of 32 rows by TI columns (tile_columns) go through shared memory so that
// the planes are written in runs, and the spacing's inverse saves the divisions:
// 16001 x 128 328 -> 36 us, 4001 x 64 48 -> 8.2.
template <typename T, int TI>
__global__ void __launch_bounds__(kTileThreads)
initial_transpose_kernel(int Nr, int Nth, int NP, Divisor d, const T *__restrict__ lam0,
                         const double *__restrict__ b_node, int independent_pi, double *__restrict__ out)
{
    __shared__ double f[4][32][TI + 1];
    const int j0 = blockIdx.x * 32, i0 = blockIdx.y * TI, lane = threadIdx.x & 31, jp = j0 + lane;
    const size_t plane = (size_t)Nth * Nr;
    const int nout = independent_pi ? 4 : 2;
    auto L = [&](int ii, int c) { return (double)lam0[((size_t)ii * 4 + c) * NP + jp]; };
    for (int x = threadIdx.x >> 5; x < TI; x += kTileThreads / 32) {
        const int i = i0 + x;
        double g[4] = {0.0, 0.0, 0.0, 0.0};
        if (i > 0 && i < Nr - 1) {
            for (int c = 0; c < 4; ++c) g[c] = L(i, c);
            if (!independent_pi) {
                for (int c = 0; c < 2; ++c) {
                    if (i - 1 >= 1) g[c] += d.under(b_node[(size_t)(i - 1) * NP + jp] * L(i - 1, 2 + c));
                    if (i + 1 <= Nr - 2) g[c] -= d.under(b_node[(size_t)(i + 1) * NP + jp] * L(i + 1, 2 + c));
                }
            }
        }
        for (int c = 0; c < nout; ++c) f[c][lane][x] = g[c];
    }
    __syncthreads();
    for (int q = threadIdx.x; q < 32 * TI; q += kTileThreads) {
        const int r = q / TI, x = q % TI, i = i0 + x;
        if (j0 + r >= Nth || i >= Nr) continue;
        for (int c = 0; c < nout; ++c) out[c * plane + (size_t)(j0 + r) * Nr + i] = f[c][r][x];
    }
}

// ---- gradients with respect to the black-hole parameters (a or M) ----
//
// With the tables T(p) of one inner step u^{j+1} = A(p) u^j, the loss
// gradient is dL/dp = sum_j lam~^{j+1} . (dA/dp) u^j (+ the initial-data
// term below), lam~^{j+1} the adjoint state the adjoint kernel loads (with
// the waveform gradient of the step added and the radial edges zeroed).  By
// the product rule through the half nodes h = H u,
//   (dA/dp) u at node i = N'(h_{i-1/2}, h_{i+1/2}) + N(h'_{i-1/2}, h'_{i+1/2}),
// where N' is the node update with the derivative tables and no constant
// terms, h' = H' u the half nodes with the derivative tables, and N applies
// the ordinary node tables to h'.  One warp per column range, recomputing
// its left edge.
//
// One launch contracts up to kLamSteps successive steps, blockIdx.y = q the
// transpose's steps first + q of a segment (counted from its end, whose last
// sample is t_last): u^j at u_last - q * (one state), lam~ in lams.p[q].  Every
// block writes its partial sum to its own slot, [q][block], and
// tangent_sum_kernel adds them to acc in the order of the steps, so that the
// sum does not depend on how the steps are grouped (nor the split into blocks,
// a function of Nr alone).  Bound by the FP64 pipe: with a launch per step a
// 1601 x 32 grid had one column per warp, which forms two half nodes to use
// one, 20.8 us a step; with several steps a launch a warp can take more
// columns (four from 1536 radii on; fewer below, where the shortest checkpoint
// interval would leave the chip idle), 11.7 us.
constexpr int kLamSteps = 8;
struct LamSet {
    const double *p[kLamSteps];
};

template <int K>
__global__ void __launch_bounds__(128)
param_tangent_kernel(const double *__restrict__ u_last, const __grid_constant__ LamSet lams, long long first, long long t_last,
                     int substeps, const double *__restrict__ half, const double *__restrict__ node,
                     const double *__restrict__ dhalf, const double *__restrict__ dnode, int Nr,
                     double eh, double en, const InjectArgs inj, double *__restrict__ part_sums)
{
    constexpr int NP = 32 * K;
    constexpr size_t SP = 4 * NP, HP = (size_t)kNCH * NP, NQ = (size_t)kNCN * NP;
    __shared__ double part[4];
    const int lane = threadIdx.x & 31;
    const int wib = threadIdx.x >> 5;
    int i0, i1, left;
    warp_range<4>(Nr, wib, &i0, &i1, &left);
    const int row = lane * K;
    const int q = blockIdx.y;
    const double *__restrict__ u = u_last - (size_t)q * Nr * SP, *__restrict__ lam = lams.p[q];
    const int on = (first + q) % substeps == 0;
    const long long sample = t_last - (first + q) / substeps;
    double sum = 0.0;
    if (i1 > i0) {
        double ua[4][K], hm[4][K], dm[4][K], zero[4][K];
        zero_col<double, K>(zero);
        load_col<double, K>(u + (size_t)i0 * SP + row, ua);
        if (i0 > 0) {
            double ul[4][K];
            load_col<double, K>(u + (size_t)(i0 - 1) * SP + row, ul);
            half_node<double, K>(ul, ua, half + (size_t)(i0 - 1) * HP + row, hm);
            half_node<double, K, false>(ul, ua, dhalf + (size_t)(i0 - 1) * HP + row, dm);
        } else {
            zero_col<double, K>(hm);
            zero_col<double, K>(dm);
        }
        for (int i = i0; i < i1; ++i) {
            double uc[4][K], hp[4][K], dp[4][K];
            if (i + 1 < Nr) {
                load_col<double, K>(u + (size_t)(i + 1) * SP + row, uc);
                half_node<double, K>(ua, uc, half + (size_t)i * HP + row, hp);
                half_node<double, K, false>(ua, uc, dhalf + (size_t)i * HP + row, dp);
            } else {
                zero_col<double, K>(uc);
                zero_col<double, K>(hp);
                zero_col<double, K>(dp);
            }
            if (i >= 1 && i <= Nr - 2) {
                double d1[4][K], d2[4][K], l[4][K];
                full_node<double, K>(hm, hp, zero, dnode + (size_t)i * NQ + row, 0.0, d1);
                full_node<double, K>(dm, dp, zero, node + (size_t)i * NQ + row, en, d2);
                load_lam<double, K>(lam, i, Nr, lane, inj, on, sample, l);
#pragma unroll
                for (int c = 0; c < 4; ++c)
#pragma unroll
                    for (int t = 0; t < K; ++t) sum = fma(l[c][t], d1[c][t] + d2[c][t], sum);
            }
#pragma unroll
            for (int c = 0; c < 4; ++c)
#pragma unroll
                for (int t = 0; t < K; ++t) {
                    ua[c][t] = uc[c][t];
                    hm[c][t] = hp[c][t];
                    dm[c][t] = dp[c][t];
                }
        }
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, off);
    if (lane == 0) part[wib] = sum;
    __syncthreads();
    if (threadIdx.x == 0)
        part_sums[(size_t)q * gridDim.x + blockIdx.x] = (part[0] + part[1]) + (part[2] + part[3]);
}

__global__ void tangent_sum_kernel(const double *__restrict__ part_sums, int blocks, int steps,
                                   double *__restrict__ acc)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= blocks) return;
    double s = acc[k];
    for (int q = 0; q < steps; ++q) s += part_sums[(size_t)q * blocks + k];
    acc[k] = s;
}

// Initial-data term for a momentum derived from Phi^0: Pi^0 = b d_* Phi^0
// depends on the parameter through b, d Pi^0 / dp = (db/dp / b) Pi^0.
// lam0 = dL/du^0.  Partial sums per block into part[blockIdx] (fixed order).
__global__ void param_initial_kernel(int Nr, int Nth, int NP, const double *__restrict__ u0,
                                     const double *__restrict__ lam0, const double *__restrict__ b_node,
                                     const double *__restrict__ db_node, double *__restrict__ part)
{
    __shared__ double ws[8];
    double sum = 0.0;
    const long long n = (long long)Nr * NP;
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < n;
         k += (long long)gridDim.x * blockDim.x) {
        const int i = (int)(k / NP), jp = (int)(k - (long long)i * NP);
        if (jp >= Nth || i == 0 || i == Nr - 1) continue;
        const double f = db_node[k] / b_node[k];
        const size_t col = (size_t)i * 4 * NP + jp;
        sum = fma(lam0[col + 2 * NP], f * u0[col + 2 * NP], sum);
        sum = fma(lam0[col + 3 * NP], f * u0[col + 3 * NP], sum);
    }
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, off);
    if (lane == 0) ws[w] = sum;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int k = 0; k < (int)(blockDim.x >> 5); ++k) t += ws[k];
        part[blockIdx.x] = t;
    }
}

cudaError_t launch_param_tangent(int K, int blocks, int steps, const double *u_last, const LamSet &lams, long long first,
                                 long long t_last, int substeps, const double *half, const double *node,
                                 const double *dhalf, const double *dnode, int Nr, double dt_in,
                                 const InjectArgs &inj, double *part_sums, double *acc, cudaStream_t st)
{
    const double eh = 0.25 * dt_in, en = 0.5 * dt_in;
    const dim3 grid(blocks, steps);
    if (K == 1)
        param_tangent_kernel<1><<<grid, 128, 0, st>>>(u_last, lams, first, t_last, substeps, half, node, dhalf, dnode,
                                                      Nr, eh, en, inj, part_sums);
    else if (K == 2)
        param_tangent_kernel<2><<<grid, 128, 0, st>>>(u_last, lams, first, t_last, substeps, half, node, dhalf, dnode,
                                                      Nr, eh, en, inj, part_sums);
    else
        param_tangent_kernel<4><<<grid, 128, 0, st>>>(u_last, lams, first, t_last, substeps, half, node, dhalf, dnode,
                                                      Nr, eh, en, inj, part_sums);
    tangent_sum_kernel<<<(blocks + 127) / 128, 128, 0, st>>>(part_sums, blocks, steps, acc);
    return cudaGetLastError();
}

// The FP64 tables and the bytes from a column's to the next's (0: one cold block).
struct AdjTables {
    const unsigned char *p;
    size_t pitch;
};

template <typename T, int K, int W>
constexpr size_t adj_smem_bytes()
{
    return sizeof(T) == 8 ? (size_t)W * sizeof(AdjRing) : (size_t)W * kAdjShared * 32 * K * sizeof(T);
}

// The kernels of a precision: one launch per step, and every step in one.
template <typename T, int K, int W>
const void *adj_kernel()
{
    if constexpr (sizeof(T) == 8) return (const void *)lw_adjoint_team_kernel<K, W>;
    else return (const void *)lw_adjoint_kernel<T, K, W>;
}

template <typename T, int K, int W>
const void *adj_persistent_kernel()
{
    if constexpr (sizeof(T) == 8) return (const void *)lw_adjoint_team_persistent_kernel<K, W>;
    else return (const void *)lw_adjoint_persistent_kernel<T, K, W>;
}

template <typename T, int K, int W>
cudaError_t adj_smem_setup()
{
    static DeviceOnce once;
    const cudaError_t e = allow_smem(once, adj_kernel<T, K, W>(), adj_smem_bytes<T, K, W>());
    return e;
}

template <typename T, int K, int W>
cudaError_t launch_adj_shape(const void *lam, void *mu, const void *half, const void *node, AdjTables tab,
                             int Nr, int blocks, double dt_in, const InjectArgs &inj, int *err,
                             cudaStream_t st)
{
    cudaError_t e = adj_smem_setup<T, K, W>();
    if (e != cudaSuccess) return e;
    if constexpr (sizeof(T) == 8)
        return launch_chained<lw_adjoint_team_kernel<K, W>>(
            (unsigned)blocks, W * 32, adj_smem_bytes<T, K, W>(), st, (const double *)lam, (double *)mu,
            (const double *)half, (const double *)node, tab.p, tab.pitch, Nr, 0.5 * dt_in, inj, err);
    else
        return launch_chained<lw_adjoint_kernel<T, K, W>>(
            (unsigned)blocks, W * 32, adj_smem_bytes<T, K, W>(), st, (const T *)lam, (T *)mu, (const T *)half,
            (const T *)node, Nr, (T)(0.25 * dt_in), (T)(0.5 * dt_in), inj);
}

template <typename T, int K>
cudaError_t launch_adj(const void *lam, void *mu, const void *half, const void *node, AdjTables tab, int Nr,
                       int blocks, int warps, double dt_in, const InjectArgs &inj, int *err, cudaStream_t st)
{
    constexpr int WW = adj_wide_warps<T, K>();
    if (warps == WW)
        return launch_adj_shape<T, K, WW>(lam, mu, half, node, tab, Nr, blocks, dt_in, inj, err, st);
    if (warps == kNarrowWarps)
        return launch_adj_shape<T, K, kNarrowWarps>(lam, mu, half, node, tab, Nr, blocks, dt_in, inj, err, st);
    return cudaErrorInvalidValue;
}

cudaError_t launch_adjoint_step(int precision, int K, const void *lam, void *mu, const void *half,
                                const void *node, AdjTables tab, int Nr, int blocks, int warps, double dt_in,
                                const InjectArgs &inj, int *err, cudaStream_t st)
{
    if (precision == 0) {
        if (K == 1) return launch_adj<double, 1>(lam, mu, half, node, tab, Nr, blocks, warps, dt_in, inj, err, st);
        if (K == 2) return launch_adj<double, 2>(lam, mu, half, node, tab, Nr, blocks, warps, dt_in, inj, err, st);
        return launch_adj<double, 4>(lam, mu, half, node, tab, Nr, blocks, warps, dt_in, inj, err, st);
    }
    if (K == 1) return launch_adj<float, 1>(lam, mu, half, node, tab, Nr, blocks, warps, dt_in, inj, err, st);
    if (K == 2) return launch_adj<float, 2>(lam, mu, half, node, tab, Nr, blocks, warps, dt_in, inj, err, st);
    return launch_adj<float, 4>(lam, mu, half, node, tab, Nr, blocks, warps, dt_in, inj, err, st);
}

template <typename T, int K, int W>
int adj_persistent_blocks_w(int Nr, int num_sms)
{
    const void *kern = adj_persistent_kernel<T, K, W>();
    static DeviceOnce once;
    const cudaError_t e0 = allow_smem(once, kern, adj_smem_bytes<T, K, W>());
    int n = 0;
    if (e0 != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kern, W * 32, adj_smem_bytes<T, K, W>()) != cudaSuccess ||
        n < 1)
        return 0;
    constexpr int C = W / (sizeof(T) == 8 ? K : 1);   // columns at a time (FP64: teams)
    long long blocks = (long long)num_sms * n;
    if (blocks > Nr / C) blocks = Nr / C;
    return blocks < 1 ? 0 : (int)blocks;
}

template <typename T, int K>
int adj_persistent_blocks_t(int Nr, int num_sms, int warps)
{
    constexpr int WW = adj_wide_warps<T, K>();
    if (warps == WW) return adj_persistent_blocks_w<T, K, WW>(Nr, num_sms);
    if (warps == kNarrowWarps) return adj_persistent_blocks_w<T, K, kNarrowWarps>(Nr, num_sms);
    return 0;
}

template <typename T, int K, int W>
cudaError_t launch_adj_persistent_w(void *a0, void *a1, const void *half, const void *node,
                                    AdjTables tab, int Nr, int blocks,
                                    double dt_in, const InjectArgs &inj, int inject, long long n_inner,
                                    int substeps, unsigned int *flags, int *err, cudaStream_t st)
{
    T *p0 = (T *)a0, *p1 = (T *)a1;
    const T *h = (const T *)half, *nd = (const T *)node;
    T en = (T)(0.5 * dt_in);
    InjectArgs in = inj;
    void *args64[] = {&p0, &p1, &h, &nd, &tab.p, &tab.pitch, &Nr, &en, &in, &inject, &n_inner, &substeps, &flags, &err};
    void *args32[] = {&p0, &p1, &h, &nd, &Nr, &en, &in, &inject, &n_inner, &substeps, &flags, &err};
    return cudaLaunchCooperativeKernel(adj_persistent_kernel<T, K, W>(), dim3(blocks), dim3(W * 32),
                                       sizeof(T) == 8 ? args64 : args32, adj_smem_bytes<T, K, W>(), st);
}

template <typename T, int K>
cudaError_t launch_adj_persistent_t(void *a0, void *a1, const void *half, const void *node,
                                    AdjTables tab, int Nr, int blocks,
                                    int warps, double dt_in, const InjectArgs &inj, int inject,
                                    long long n_inner, int substeps, unsigned int *flags, int *err,
                                    cudaStream_t st)
{
    constexpr int WW = adj_wide_warps<T, K>();
    if (warps == WW)
        return launch_adj_persistent_w<T, K, WW>(a0, a1, half, node, tab, Nr, blocks, dt_in, inj, inject, n_inner,
                                                 substeps, flags, err, st);
    if (warps == kNarrowWarps)
        return launch_adj_persistent_w<T, K, kNarrowWarps>(a0, a1, half, node, tab, Nr, blocks, dt_in, inj, inject,
                                                           n_inner, substeps, flags, err, st);
    return cudaErrorInvalidValue;
}

// Blocks of the one-column-per-team launch (FP64), 0 where the grid has too many
// columns.
template <int K>
int adj_column_blocks(int Nr, int num_sms)
{
    int n = 0;
    static DeviceOnce once;
    const cudaError_t e0 = allow_smem(once, (const void *)lw_adjoint_column_kernel<K>, sizeof(AdjColumnShared<K>));
    if (e0 != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, lw_adjoint_column_kernel<K>, (kAdjColumns + 1) * K * 32,
                                                      sizeof(AdjColumnShared<K>)) != cudaSuccess)
        return 0;
    const int blocks = (Nr + kAdjColumns - 1) / kAdjColumns;
    return blocks <= num_sms * n ? blocks : 0;
}

int adjoint_column_blocks(int precision, int K, int Nr, int num_sms)
{
    if (precision != 0) return 0;
    return K == 1 ? adj_column_blocks<1>(Nr, num_sms)
         : K == 2 ? adj_column_blocks<2>(Nr, num_sms)
                  : adj_column_blocks<4>(Nr, num_sms);
}

template <int K>
cudaError_t launch_adj_columns(double *a0, double *a1, const void *half, const void *node, AdjTables tab,
                               int Nr, int blocks, double dt_in, const InjectArgs &inj, int inject, long long n_inner,
                               int substeps, unsigned int *flags, int *err, long long first, size_t stride,
                               cudaStream_t st)
{
    const double *h = (const double *)half, *nd = (const double *)node;
    double en = 0.5 * dt_in;
    InjectArgs in = inj;
    void *args[] = {&a0,     &a1,      &h,        &nd,    &tab.p, &tab.pitch, &Nr,    &en, &in,
                    &inject, &n_inner, &substeps, &flags, &err,   &first,     &stride};
    return cudaLaunchCooperativeKernel((const void *)lw_adjoint_column_kernel<K>, dim3(blocks),
                                       dim3((kAdjColumns + 1) * K * 32), args, sizeof(AdjColumnShared<K>), st);
}

cudaError_t launch_adjoint_columns(int K, double *a0, double *a1, const void *half, const void *node,
                                   AdjTables tab, int Nr, int blocks, double dt_in, const InjectArgs &inj,
                                   int inject, long long n_inner, int substeps, unsigned int *flags, int *err,
                                   long long first, size_t stride, cudaStream_t st)
{
    auto go = [&](auto launch) {
        return launch(a0, a1, half, node, tab, Nr, blocks, dt_in, inj, inject, n_inner, substeps, flags, err, first,
                      stride, st);
    };
    return K == 1 ? go(launch_adj_columns<1>) : K == 2 ? go(launch_adj_columns<2>) : go(launch_adj_columns<4>);
}

// Blocks of the persistent adjoint launch for this grid (all resident at
// once, at most Nr / warps), or 0 if it cannot run.
int adjoint_persistent_blocks(int precision, int K, int Nr, int num_sms, int warps)
{
    if (precision == 0)
        return K == 1 ? adj_persistent_blocks_t<double, 1>(Nr, num_sms, warps)
             : K == 2 ? adj_persistent_blocks_t<double, 2>(Nr, num_sms, warps)
                      : adj_persistent_blocks_t<double, 4>(Nr, num_sms, warps);
    return K == 1 ? adj_persistent_blocks_t<float, 1>(Nr, num_sms, warps)
         : K == 2 ? adj_persistent_blocks_t<float, 2>(Nr, num_sms, warps)
                  : adj_persistent_blocks_t<float, 4>(Nr, num_sms, warps);
}

cudaError_t launch_adjoint_persistent(int precision, int K, void *a0, void *a1, const void *half,
                                      const void *node, AdjTables tab, int Nr, int blocks, int warps, double dt_in,
                                      const InjectArgs &inj, int inject, long long n_inner, int substeps,
                                      unsigned int *flags, int *err, cudaStream_t st)
{
    if (precision == 0) {
        if (K == 1)
            return launch_adj_persistent_t<double, 1>(a0, a1, half, node, tab, Nr, blocks, warps, dt_in, inj, inject,
                                                      n_inner, substeps, flags, err, st);
        if (K == 2)
            return launch_adj_persistent_t<double, 2>(a0, a1, half, node, tab, Nr, blocks, warps, dt_in, inj, inject,
                                                      n_inner, substeps, flags, err, st);
        return launch_adj_persistent_t<double, 4>(a0, a1, half, node, tab, Nr, blocks, warps, dt_in, inj, inject,
                                                  n_inner, substeps, flags, err, st);
    }
    if (K == 1)
        return launch_adj_persistent_t<float, 1>(a0, a1, half, node, tab, Nr, blocks, warps, dt_in, inj, inject,
                                                 n_inner, substeps, flags, err, st);
    if (K == 2)
        return launch_adj_persistent_t<float, 2>(a0, a1, half, node, tab, Nr, blocks, warps, dt_in, inj, inject,
                                                 n_inner, substeps, flags, err, st);
    return launch_adj_persistent_t<float, 4>(a0, a1, half, node, tab, Nr, blocks, warps, dt_in, inj, inject,
                                             n_inner, substeps, flags, err, st);
}

template <typename T, int K, int W>
int adj_resident()
{
    int n = 0;
    if (adj_smem_setup<T, K, W>() != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, adj_kernel<T, K, W>(), W * 32,
                                                      adj_smem_bytes<T, K, W>()) != cudaSuccess)
        n = 0;
    return n;
}

template <typename T, int K>
int adj_shape(int Nr, int num_sms, int *warps)
{
    constexpr int WW = adj_wide_warps<T, K>();
    constexpr int KT = sizeof(T) == 8 ? K : 1;   // warps that share a column (FP64: a team)
    if ((long long)Nr >= (long long)num_sms * (WW / KT) && adj_resident<T, K, WW>() >= 1) {
        *warps = WW;
        return num_sms;
    }
    *warps = kNarrowWarps;
    int per_sm = adj_resident<T, K, kNarrowWarps>();
    if (per_sm < 1) per_sm = 1;
    int blocks = num_sms * per_sm;
    if (blocks > Nr / (kNarrowWarps / KT)) blocks = Nr / (kNarrowWarps / KT);
    return blocks < 1 ? 1 : blocks;
}

}  // namespace

int adjoint_grid_shape(int precision, int K, int Nr, int num_sms, int *warps)
{
    if (precision == 0)
        return K == 1 ? adj_shape<double, 1>(Nr, num_sms, warps)
             : K == 2 ? adj_shape<double, 2>(Nr, num_sms, warps)
                      : adj_shape<double, 4>(Nr, num_sms, warps);
    return K == 1 ? adj_shape<float, 1>(Nr, num_sms, warps)
         : K == 2 ? adj_shape<float, 2>(Nr, num_sms, warps)
                  : adj_shape<float, 4>(Nr, num_sms, warps);
}

}  // namespace tk

// The FP64 adjoint's tables, formed from the step's when these have changed.
static tk_status adjoint_tables(tk_solver *S)
{
    if (S->precision != TK_PREC_F64 || S->adj_tab_of == S->coeffs_id) return TK_OK;
    if (!S->adj_tab) {
        if (tkh::alloc(S, (void **)&S->adj_tab, (size_t)S->Nr * S->K * tk::kAdjBytes, true) == TK_OK)
            S->adj_pitch = S->K * tk::kAdjBytes;
        else if (tkh::cold_tables(S))
            S->adj_tab = S->cold + (size_t)S->K * tk::kStepBytes;
        else
            return TK_ERR_OOM;
    }
    if (S->adj_pitch == 0) return TK_OK;
    const dim3 block(S->NP, tk::kAdjTableThreads / S->NP), grid((S->Nr + block.y - 1) / block.y);
    tk::adj_tables_kernel<<<grid, block, 0, S->stream>>>(S->Nr, S->NP, (const double *)S->half,
                                                         (const double *)S->node, S->adj_tab);
    TK_CUDA(S, cudaGetLastError());
    S->adj_tab_of = S->coeffs_id;
    return TK_OK;
}

static tk::AdjTables tables_of(const tk_solver *S) { return {S->adj_tab, S->adj_pitch}; }

extern "C" tk_status tk_adjoint(tk_solver *S, const double *dL_dwave, const double *dL_dfinal,
                                int on_device, double *grad, int grad_on_device, int independent_pi)
{
    tk_status st = tkh::enter(S);
    if (st != TK_OK) return st;
    st = tkh::need_state(S, "tk_adjoint");
    if (st != TK_OK) return st;
    if (!grad) return tkh::fail(S, TK_ERR_ARG, "tk_adjoint: grad is NULL");
    if (!dL_dwave && !dL_dfinal)
        return tkh::fail(S, TK_ERR_ARG, "tk_adjoint: give dL_dwave, dL_dfinal or both");
    if (dL_dwave && S->nobs == 0) return tkh::fail(S, TK_ERR_ARG, "tk_adjoint: no observers");
    const size_t se = (size_t)S->Nr * 4 * S->NP;
    const size_t plane = (size_t)S->Nth * S->Nr;
    // adjoint levels and staging (allocated on first use, kept)
    for (int k = 0; k < 2; ++k)
        if (!S->adj[k]) {
            st = tkh::alloc(S, &S->adj[k], se * S->esz);
            if (st != TK_OK) return st;
        }
    st = adjoint_tables(S);
    if (st != TK_OK) return st;
    const long long count = S->count;
    double *dwave = nullptr;
    double *dfin = nullptr;
    double *gdev = nullptr;
    auto cleanup = [&]() {
        if (dwave && !on_device) cudaFree(dwave);
        if (dfin) cudaFree(dfin);
        if (gdev && !grad_on_device) cudaFree(gdev);
    };
    if (dL_dwave) {
        if (on_device) {
            dwave = const_cast<double *>(dL_dwave);
        } else {
            st = tkh::alloc(S, (void **)&dwave, (size_t)S->nobs * count * 2 * sizeof(double));
            if (st != TK_OK) return st;
            cudaError_t e = cudaMemcpyAsync(dwave, dL_dwave, (size_t)S->nobs * count * 2 * sizeof(double),
                                            cudaMemcpyHostToDevice, S->stream);
            if (e != cudaSuccess) {
                cleanup();
                return tkh::fail(S, TK_ERR_CUDA, "tk_adjoint: %s", cudaGetErrorString(e));
            }
        }
    }
    // lam = dL/du(T): the final-state gradient (or 0)
    cudaError_t e = cudaSuccess;
    if (dL_dfinal) {
        const double *src = dL_dfinal;
        if (!on_device) {
            st = tkh::alloc(S, (void **)&dfin, 4 * plane * sizeof(double));
            if (st != TK_OK) {
                cleanup();
                return st;
            }
            e = cudaMemcpyAsync(dfin, dL_dfinal, 4 * plane * sizeof(double), cudaMemcpyHostToDevice, S->stream);
            src = dfin;
        }
        if (e == cudaSuccess)
            e = tk::launch_import_state(S->precision, S->Nr, S->Nth, S->NP, S->drs, src, src + plane,
                                        src + 2 * plane, src + 3 * plane, S->b_node, S->adj[0], S->num_sms,
                                        S->stream);
    } else {
        e = cudaMemsetAsync(S->adj[0], 0, se * S->esz, S->stream);
    }
    tk::InjectArgs inj;
    memset(&inj, 0, sizeof inj);
    inj.count = count;
    inj.dwave = dwave;
    inj.w_row = S->w_row;
    {
        tk::StepLaunch L;
        tkh::fill_launch(S, L);
        inj.obs = L.obs;
    }
    int cur = 0;
    const double dt_in = S->dt / S->substeps;
    const long long n_inner = count * S->substeps;
    // the solver's launch structure: every step in one persistent launch, or
    // one launch per step
    const int pblocks = (S->persist && n_inner > 0)
                            ? tk::adjoint_persistent_blocks(S->precision, S->K, S->Nr, S->num_sms, S->adj_warps)
                            : 0;
    if (pblocks > 0 && e == cudaSuccess) {
        unsigned int *flags = nullptr;
        const int cblocks = tk::adjoint_column_blocks(S->precision, S->K, S->Nr, S->num_sms);
        const int nflags = 2 * std::max(pblocks, cblocks) * (S->precision == TK_PREC_F64 ? S->K : 1);
        const size_t fbytes = (size_t)nflags * sizeof(unsigned int) + sizeof(int);
        st = tkh::alloc(S, (void **)&flags, fbytes);
        if (st != TK_OK) {
            cleanup();
            return st;
        }
        int *derr = (int *)(flags + nflags);
        int herr = 0;
        e = cudaMemsetAsync(flags, 0, fbytes, S->stream);
        if (e == cudaSuccess && cblocks > 0)
            e = tk::launch_adjoint_columns(S->K, (double *)S->adj[0], (double *)S->adj[1], S->half, S->node, tables_of(S),
                                           S->Nr, cblocks, dt_in, inj, dwave != nullptr, n_inner, S->substeps, flags,
                                           derr, 0, 0, S->stream);
        else if (e == cudaSuccess)
            e = tk::launch_adjoint_persistent(S->precision, S->K, S->adj[0], S->adj[1], S->half, S->node, tables_of(S),
                                              S->Nr, pblocks, S->adj_warps, dt_in, inj, dwave != nullptr, n_inner,
                                              S->substeps, flags, derr, S->stream);
        if (e == cudaSuccess) e = cudaMemcpyAsync(&herr, derr, sizeof(int), cudaMemcpyDeviceToHost, S->stream);
        if (e == cudaSuccess) e = cudaStreamSynchronize(S->stream);
        cudaFree(flags);
        if (e == cudaSuccess && herr) {
            cleanup();
            return tkh::fail(S, TK_ERR_INTERNAL, "tk_adjoint: a block of the persistent launch waited too "
                                                 "long for a neighbour; the gradient is invalid");
        }
        cur = (int)(n_inner & 1);
    } else {
        for (long long t = count - 1; t >= 0 && e == cudaSuccess; --t)
            for (int k = 0; k < S->substeps && e == cudaSuccess; ++k) {
                inj.on = (k == 0) && dwave != nullptr;
                inj.sample = t;
                e = tk::launch_adjoint_step(S->precision, S->K, S->adj[cur], S->adj[cur ^ 1], S->half,
                                            S->node, tables_of(S), S->Nr, S->adj_blocks, S->adj_warps, dt_in, inj,
                                            S->lost + 1, S->stream);
                cur ^= 1;
            }
        if (e == cudaSuccess) e = tkh::mark_unchecked(S, S->stream, 1);
    }
    if (e != cudaSuccess) {
        cleanup();
        return tkh::fail(S, TK_ERR_CUDA, "tk_adjoint: %s", cudaGetErrorString(e));
    }
    // the initial-data map
    const int nout = independent_pi ? 4 : 2;
    if (grad_on_device) {
        gdev = grad;
    } else {
        st = tkh::alloc(S, (void **)&gdev, nout * plane * sizeof(double));
        if (st != TK_OK) {
            cleanup();
            return st;
        }
    }
    const int ti = tk::tile_columns(S->Nr, S->NP, S->num_sms);
    const dim3 gridd(S->NP / 32, (S->Nr + ti - 1) / ti);
    const tk::Divisor d = tk::divisor(2.0 * S->drs);
    auto transpose = [&](auto kern, auto *lam) {
        kern<<<gridd, tk::kTileThreads, 0, S->stream>>>(S->Nr, S->Nth, S->NP, d, lam, S->b_node, independent_pi, gdev);
    };
    if (S->precision == 0)
        transpose(ti == 8 ? tk::initial_transpose_kernel<double, 8> : tk::initial_transpose_kernel<double, 32>,
                  (const double *)S->adj[cur]);
    else
        transpose(ti == 8 ? tk::initial_transpose_kernel<float, 8> : tk::initial_transpose_kernel<float, 32>,
                  (const float *)S->adj[cur]);
    e = cudaGetLastError();
    if (e == cudaSuccess && !grad_on_device)
        e = cudaMemcpyAsync(grad, gdev, nout * plane * sizeof(double), cudaMemcpyDeviceToHost, S->stream);
    if (e == cudaSuccess && (!grad_on_device || !on_device)) e = cudaStreamSynchronize(S->stream);
    cleanup();
    if (e != cudaSuccess) return tkh::fail(S, TK_ERR_CUDA, "tk_adjoint: %s", cudaGetErrorString(e));
    return grad_on_device && on_device ? TK_OK : tkh::check_lost(S, "tk_adjoint");
}

// Gradient of a waveform loss with respect to the spin a (param 0) or the mass
// M (param 1), through checkpointed recomputation of the trajectory.
extern "C" tk_status tk_param_gradient(tk_solver *S, int param, const double *dL_dwave, int on_device,
                                       int checkpoint_every, double *grad)
{
    tk_status st = tkh::enter(S);
    if (st != TK_OK) return st;
    if (!grad || !dL_dwave) return tkh::fail(S, TK_ERR_ARG, "tk_param_gradient: NULL argument");
    if (param != 0 && param != 1) return tkh::fail(S, TK_ERR_ARG, "tk_param_gradient: param %d is not 0 (a) or 1 (M)", param);
    if (S->precision != TK_PREC_F64)
        return tkh::fail(S, TK_ERR_ARG, "tk_param_gradient: FP64 solvers only");
    if (!S->have_state || !S->state_valid || !S->init_valid)
        return tkh::fail(S, TK_ERR_STATE, "tk_param_gradient: needs a trajectory from tk_set_initial_data "
                                          "(not restarted with tk_set_state)");
    if (S->nobs == 0) return tkh::fail(S, TK_ERR_ARG, "tk_param_gradient: no observers");
    const long long count = S->count;
    if (count <= 0) return tkh::fail(S, TK_ERR_STATE, "tk_param_gradient: no steps taken");
    const int k = S->substeps;
    long long C = checkpoint_every;
    if (C <= 0) {
        C = (long long)sqrt((double)count / k);
        if (C < 1) C = 1;
    }
    if (C > count) C = count;
    const long long nck = (count + C - 1) / C;
    const size_t se = (size_t)S->Nr * 4 * S->NP, sb = se * sizeof(double);
    const size_t nh = (size_t)S->Nr * tk::kNCH * S->NP, nn = (size_t)S->Nr * tk::kNCN * S->NP;
    const size_t nb = (size_t)S->Nr * S->NP;

    // the steps contracted per launch: their adjoint states are kept, two in the
    // solver's own buffers (small grids: in the scratch, in a row), the others in
    // the scratch (256 MB at most)
    int Q = (int)std::min<long long>(std::min<long long>(C * k, tk::kLamSteps), 1 + (long long)((256ull << 20) / sb));
    const int blocks = std::max(1, S->Nr / (4 * std::min(4, 1 + S->Nr / 512))), pblocks = 1024;

    // small grids: a segment's levels in one launch (lw_column_kernel writing a
    // trajectory), 4.3 us a step at 1601 x 32 where a launch per step takes 8.6
    const bool columns = S->persist && S->persist_columns && C * k <= 0x7fffffff;
    // and the transposed steps that one tangent launch contracts (6.2 us a step
    // there, 10.6 with a launch each; for fewer than four the launch costs more)
    int cblocks = S->persist && Q >= 4 ? tk::adjoint_column_blocks(0, S->K, S->Nr, S->num_sms) : 0;
    const size_t nflags = (size_t)2 * S->K * std::max(columns ? S->persist_blocks : 0, cblocks);

    // scratch in one allocation, freed on every exit
    double *dwave = nullptr, *scratch = nullptr;
    double *tx = nullptr, *tang = nullptr, *ck = nullptr, *seg = nullptr, *acc = nullptr, *parts = nullptr;
    double *lam_more = nullptr, *pflags = nullptr;
    auto cleanup = [&]() {
        if (scratch) cudaFree(scratch);
        if (dwave && !on_device) cudaFree(dwave);
    };
    auto bail = [&](tk_status s2) {
        cleanup();
        return s2;
    };
    if ((st = adjoint_tables(S)) != TK_OK) return st;
    for (int q = 0; q < 2; ++q)
        if (!S->adj[q] && (st = tkh::alloc(S, &S->adj[q], sb)) != TK_OK) return bail(st);
    if (!S->dhalf && (st = tkh::alloc(S, (void **)&S->dhalf, nh * sizeof(double))) != TK_OK) return bail(st);
    if (!S->dnode && (st = tkh::alloc(S, (void **)&S->dnode, nn * sizeof(double))) != TK_OK) return bail(st);
    if (!S->db_node && (st = tkh::alloc(S, (void **)&S->db_node, nb * sizeof(double))) != TK_OK) return bail(st);
    // (one allocation: each costs some 70 us with its release); without the
    // further adjoint states where the memory does not reach
    for (;; Q = 1, cblocks = 0) {
        struct { double **p; size_t n; } piece[] = {
            {&ck, (size_t)nck * se}, {&seg, (size_t)(C * k) * se}, {&lam_more, (size_t)(cblocks ? Q + 1 : Q - 1) * se},
            {&tx, (size_t)tk::kShifts * 2 * S->Nr * tk::kRadial}, {&tang, (size_t)2 * S->NP},
            {&acc, (size_t)(blocks + pblocks)}, {&parts, (size_t)Q * blocks}, {&pflags, 1 + (nflags + 1) / 2}};
        size_t total = 0;
        for (auto &x : piece) total += (x.n + 31) / 32 * 32;
        st = tkh::alloc(S, (void **)&scratch, total * sizeof(double), Q > 1 || cblocks);
        if (st == TK_OK) {
            double *at = scratch;
            for (auto &x : piece) {
                *x.p = at;
                at += (x.n + 31) / 32 * 32;
            }
            break;
        }
        if (Q == 1 && !cblocks) return bail(st);
    }
    double *lam[tk::kLamSteps + 1];   // a ring of Q + 1 adjoint states
    for (int q = 0; q <= Q; ++q)
        lam[q] = cblocks ? lam_more + (size_t)q * se : q < 2 ? (double *)S->adj[q] : lam_more + (size_t)(q - 2) * se;
    if (on_device) {
        dwave = const_cast<double *>(dL_dwave);
    } else {
        if ((st = tkh::alloc(S, (void **)&dwave, (size_t)S->nobs * count * 2 * sizeof(double))) != TK_OK)
            return bail(st);
        cudaError_t e = cudaMemcpyAsync(dwave, dL_dwave, (size_t)S->nobs * count * 2 * sizeof(double),
                                        cudaMemcpyHostToDevice, S->stream);
        if (e != cudaSuccess) return bail(tkh::fail(S, TK_ERR_CUDA, "tk_param_gradient: %s", cudaGetErrorString(e)));
    }
    cudaError_t e = cudaSuccess;
    const double dt_in = S->dt / k;
    // 1. derivative tables, 4-point central differences in the parameter:
    //    dT/dp = [8 (T(p+d) - T(p-d)) - (T(p+2d) - T(p-2d))] / (12 d)
    {
        const double M = S->kerr.M, a = S->kerr.a;
        double d = 1e-3 * M;
        if (d > 0.25 * (M - fabs(a))) d = 0.25 * (M - fabs(a));
        const double off[tk::kShifts] = {d, -d, 2 * d, -2 * d};
        tk::KerrSet kp = {{}, {8.0 / (12 * d), -8.0 / (12 * d), -1.0 / (12 * d), 1.0 / (12 * d)}};
        for (int q = 0; q < tk::kShifts; ++q) {
            kp.k[q] = S->kerr;
            if (param == 0) kp.k[q].a += off[q];
            else kp.k[q].M += off[q];
        }
        e = tk::launch_table_derivative(kp, S->variable, S->rs_min, S->Nr, S->Nth, S->NP, S->drs, dt_in, tx, tang,
                                        S->dhalf, S->dnode, S->db_node, S->num_sms, S->stream);
    }
    if (e != cudaSuccess) return bail(tkh::fail(S, TK_ERR_CUDA, "tk_param_gradient: %s", cudaGetErrorString(e)));
    // 2. checkpoints of the trajectory every C outer steps, from u^0
    tk::StepLaunch L;
    tkh::fill_launch(S, L);
    L.write_wave = 0;
    unsigned int *flags = (unsigned int *)pflags;
    int *perr = (int *)(flags + nflags);
    L.err = perr;
    if (e == cudaSuccess) e = cudaMemsetAsync(perr, 0, sizeof(int), S->stream);
    // n >= 1 levels after src, to dst, dst + se, ..
    auto levels = [&](const double *src, double *dst, long long n) {
        tk::StepLaunch P = L;
        P.u_in = src;
        if (columns && n >= 2) {
            P.blocks = S->persist_blocks;
            P.columns = S->persist_columns;
            P.stride = se;
            cudaError_t r = cudaMemsetAsync(flags, 0, nflags * sizeof(unsigned int), S->stream);
            return r != cudaSuccess ? r : tk::launch_lw_persistent(P, dst, (int)n, k, flags, perr, S->stream);
        }
        cudaError_t r = cudaSuccess;
        for (long long j = 0; j < n && r == cudaSuccess; ++j, dst += se) {
            P.u_out = dst;
            r = tk::launch_lw_step(P, S->stream);
            P.u_in = dst;
        }
        return r;
    };
    if (e == cudaSuccess) e = cudaMemcpyAsync(ck, S->u_init, sb, cudaMemcpyDeviceToDevice, S->stream);
    for (long long c = 0; c + 1 < nck && e == cudaSuccess; ++c) {
        const double *src = ck + (size_t)c * se;
        double *dst = ck + (size_t)(c + 1) * se;
        if (columns && C * k >= 2) {
            e = levels(src, seg, C * k);
            if (e == cudaSuccess)
                e = cudaMemcpyAsync(dst, seg + (size_t)(C * k - 1) * se, sb, cudaMemcpyDeviceToDevice, S->stream);
            continue;
        }
        // C outer steps: ping-pong through the first two segment slots
        const void *in = src;
        for (long long j = 0; j < C * k && e == cudaSuccess; ++j) {
            void *out = (j == C * k - 1) ? (void *)dst : (void *)(seg + (size_t)(j & 1) * se);
            L.u_in = in;
            L.u_out = out;
            e = tk::launch_lw_step(L, S->stream);
            in = out;
        }
    }
    // 3. backward over the segments: recompute the segment's inner states,
    //    then, Q steps at a time, the adjoint steps and their tangent contraction
    if (e == cudaSuccess) e = cudaMemsetAsync(acc, 0, (size_t)(blocks + pblocks) * sizeof(double), S->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(lam[0], 0, sb, S->stream);
    tk::InjectArgs inj;
    memset(&inj, 0, sizeof inj);
    inj.count = count;
    inj.dwave = dwave;
    inj.w_row = S->w_row;
    inj.obs = L.obs;
    int cur = 0;
    for (long long c = nck - 1; c >= 0 && e == cudaSuccess; --c) {
        const long long t0 = c * C, len = (c == nck - 1) ? count - t0 : C;
        // seg[j] = u^{t0 k + j}, j < len k
        e = cudaMemcpyAsync(seg, ck + (size_t)c * se, sb, cudaMemcpyDeviceToDevice, S->stream);
        if (e == cudaSuccess && len * k > 1) e = levels(seg, seg + se, len * k - 1);
        for (long long g = 0; g < len * k && e == cudaSuccess;) {   // transposed steps from the segment's end
            const int n = (int)std::min<long long>(Q, len * k - g);
            tk::LamSet set = {};
            if (cblocks) {   // lam[0] to lam[1], .., lam[n]
                for (int q = 0; q < n; ++q) set.p[q] = lam[q];
                e = cudaMemsetAsync(flags, 0, nflags * sizeof(unsigned int), S->stream);
                if (e == cudaSuccess)
                    e = tk::launch_adjoint_columns(S->K, lam[0], lam[1], S->half, S->node, tables_of(S), S->Nr, cblocks,
                                                   dt_in, inj, 1, n, k, flags, perr,
                                                   (count - t0 - len) * k + g, se, S->stream);
            }
            for (int q = 0; !cblocks && q < n && e == cudaSuccess; ++q) {
                const int nxt = cur == Q ? 0 : cur + 1;
                set.p[q] = lam[cur];
                inj.on = (g + q) % k == 0;
                inj.sample = t0 + len - 1 - (g + q) / k;
                e = tk::launch_adjoint_step(0, S->K, lam[cur], lam[nxt], S->half, S->node, tables_of(S), S->Nr,
                                            S->adj_blocks, S->adj_warps, dt_in, inj, perr, S->stream);
                cur = nxt;
            }
            if (e == cudaSuccess)
                e = tk::launch_param_tangent(S->K, blocks, n, seg + (size_t)(len * k - 1 - g) * se, set, g,
                                             t0 + len - 1, k, (const double *)S->half, (const double *)S->node,
                                             S->dhalf, S->dnode, S->Nr, dt_in, inj, parts, acc, S->stream);
            if (e == cudaSuccess && cblocks)
                e = cudaMemcpyAsync(lam[0], lam[n], sb, cudaMemcpyDeviceToDevice, S->stream);
            g += n;
        }
    }
    // 4. the initial-data term (momentum derived from Phi^0 through b)
    if (e == cudaSuccess && S->init_pi_derived) {
        tk::param_initial_kernel<<<pblocks, 256, 0, S->stream>>>(S->Nr, S->Nth, S->NP,
                                                                  (const double *)S->u_init,
                                                                  lam[cur], S->b_node,
                                                                  S->db_node, acc + blocks);
        e = cudaGetLastError();
    }
    std::vector<double> h((size_t)blocks + pblocks, 0.0);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(h.data(), acc, h.size() * sizeof(double), cudaMemcpyDeviceToHost, S->stream);
    int herr = 0;
    if (e == cudaSuccess) e = cudaMemcpyAsync(&herr, perr, sizeof(int), cudaMemcpyDeviceToHost, S->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(S->stream);
    if (e == cudaSuccess && herr)
        return bail(tkh::fail(S, TK_ERR_INTERNAL, "tk_param_gradient: a block of the persistent launch waited too long "
                                                  "for a neighbour; the gradient is not valid"));
    if (e != cudaSuccess)
        return bail(tkh::fail(S, e == cudaErrorMemoryAllocation ? TK_ERR_OOM : TK_ERR_CUDA,
                              "tk_param_gradient: %s", cudaGetErrorString(e)));
    double g = 0.0;
    for (size_t q = 0; q < h.size(); ++q) g += h[q];
    *grad = g;
    cleanup();
    return TK_OK;
}
