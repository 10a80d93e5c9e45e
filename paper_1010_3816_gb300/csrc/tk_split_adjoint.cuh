// tk_split_adjoint.cuh -- the transposed FP64 step with its Pi -> Phi coupling
// in integers: tk_split.cuh's forms and teams for the adjoint sweep.
//
// The transpose of the step's Phi -> Pi coupling takes 28 of the 62 FP64
// instructions of a transposed update.  A column's Pi values x enter the Phi
// components of two half nodes (a half node's: of two nodes), with one set of
// coefficients for each and the theta neighbours' share in both,
//   to the left:   F1 x + Z    +- G1 x of the other part
//   to the right:  F2 x + Z    +- G2 x of the other part
//   Z = (KP x)(j-1) + (KM x)(j+1),
// so both sums are formed when the column is met and one of them is kept (as an
// integer) for the next half node (node).  34 FP64 instructions per update are
// left (26 where the coefficients are real).
//
// Measured, 16001 x 128, per step of the persistent launch: 225 us with 62 FP64
// instructions, 147 us (x 32: 37 us); the FP64 pipe is 78 % busy, 1310
// instructions per update and row of a warp are issued.
#pragma once

#include "tk_split.cuh"

namespace tk {
namespace {

// ---- tables ----

// One block of kAdjBytes per column i and 32 rows: what the half node i + 1/2
// and the node i use.  FP64 entries [12][32]: of node i B, PPR, C2I, of node
// i + 1 B, PMR, C2I, of half node i + 1/2 HP, PAR, PI, of half node i - 1/2
// HQ, PCR, PI; limb pairs [12][32]: of node i + 1 FPR, FMR, FPI, FMI, KP of the
// row before, KM of the row after, the same of half node i + 1/2 (FAR, FCR,
// FAI, FCI, KP, KM); [2][32] ints with the exponents of (F1, F2, KP, KM) and
// (G1, G2); [32] ints with the lifts of KM (low half, it multiplies the row
// above) and KP (high half), the same for both; two ints, cold and has imaginary
// coefficients, over the column and every table involved; padding.  A cold block's integers are zero, also where
// the sums formed with them go to a column that is not cold: such sums are marked
// as those of values that call for the FP64 instructions (adj_pair).
enum { A_BA = 0, A_PP, A_CA, A_BC, A_PM, A_CC, A_HP, A_PA, A_PI, A_HQ, A_PC, A_PJ };
enum { A_F1 = 0, A_F2, A_G1, A_G2, A_KP, A_KM };
constexpr int kAdjF64 = 12;
constexpr int kAdjExps = (kAdjF64 + 12) * 256;
constexpr int kAdjHead = kAdjExps + 256 + 128;   // offset of the column's two flags
constexpr int kAdjBytes = kAdjHead + 16;

// The rows' records with the two exponents in one word: sixteen warps' rings
// leave no room for more.
struct AdjRows {
    int4 s[2][32];
    unsigned x[2][32];
    __device__ __forceinline__ void put_exps(int b, int l, int2 e) { x[b][l] = (unsigned)e.x | ((unsigned)e.y << 16); }
    __device__ __forceinline__ int2 exps(int b, int l) const
    {
        return make_int2((int)(x[b][l] & 0xffff), (int)(x[b][l] >> 16));
    }
};

template <int K>
using AdjTeam = SplitTeam<K, AdjRows>;

template <bool HALF>
struct AdjTab {
    const unsigned char *p;
    int lane;
    __device__ __forceinline__ int2 entry(int q) const
    {
        return *reinterpret_cast<const int2 *>(p + ((kAdjF64 + (HALF ? 6 : 0) + q) * 32 + lane) * 8);
    }
    __device__ __forceinline__ int row_exp() const
    {
        return *reinterpret_cast<const int *>(p + kAdjExps + (HALF ? 128 : 0) + lane * 4);
    }
    __device__ __forceinline__ int lifts() const
    {
        return *reinterpret_cast<const int *>(p + kAdjExps + 256 + lane * 4);
    }
    __device__ __forceinline__ int2 head() const { return *reinterpret_cast<const int2 *>(p + kAdjHead); }
};

__device__ __forceinline__ double adj_f64(const unsigned char *p, int q, int lane)
{
    return *reinterpret_cast<const double *>(p + (q * 32 + lane) * 8);
}

// From the unsplit tables; blockDim.x = NP, one thread per point.
constexpr int kAdjTableThreads = 256;
__global__ void __launch_bounds__(kAdjTableThreads)
adj_tables_kernel(int Nr, int NP, const double *__restrict__ half, const double *__restrict__ node,
                  unsigned char *__restrict__ out)
{
    __shared__ int flags[kAdjTableThreads / 32][2];
    const int jp = threadIdx.x, k = threadIdx.y * blockDim.x + threadIdx.x;
    int i = blockIdx.x * blockDim.y + threadIdx.y;
    if (k < kAdjTableThreads / 32 * 2) (&flags[0][0])[k] = 0;
    __syncthreads();
    auto H = [&](int c, int q, int j) {
        return (c < 0 || c >= Nr - 1 || j < 0 || j >= NP) ? 0.0 : half[((size_t)c * kNCH + q) * NP + j];
    };
    auto N = [&](int c, int q, int j) {
        return (c < 1 || c >= Nr - 1 || j < 0 || j >= NP) ? 0.0 : node[((size_t)c * kNCN + q) * NP + j];
    };
    // integers of node c (w = 0) or half node c (w = 1)
    auto entries = [&](int c, int w, double (&v)[6]) {
        if (w == 0) {
            v[A_F1] = N(c, N_FPR, jp), v[A_F2] = N(c, N_FMR, jp), v[A_G1] = N(c, N_FPI, jp), v[A_G2] = N(c, N_FMI, jp);
            v[A_KP] = N(c, N_KP, jp - 1), v[A_KM] = N(c, N_KM, jp + 1);
        } else {
            v[A_F1] = H(c, H_FAR, jp), v[A_F2] = H(c, H_FCR, jp), v[A_G1] = H(c, H_FAI, jp), v[A_G2] = H(c, H_FCI, jp);
            v[A_KP] = H(c, H_KP, jp - 1), v[A_KM] = H(c, H_KM, jp + 1);
        }
    };
    auto terms = [](const double (&v)[6]) {
        return RowTerms{fabs(v[A_F1]) + fabs(v[A_F2]), fabs(v[A_KM]), fabs(v[A_KP])};
    };
    auto other = [](const double (&v)[6]) { return fabs(v[A_G1]) + fabs(v[A_G2]); };
    double vn[6], vh[6];
    int cold = 0;
    const bool in = i < Nr - 1;
    if (!in) i = Nr - 2;   // (the block's threads meet below)
    {   // node i and half node i - 1/2: flags only
        double wn[6], wh[6];
        entries(i, 0, wn);
        entries(i - 1, 1, wh);
        const RowTerms tn = terms(wn), th = terms(wh);
        const RowLifts lift(tn, th, &cold);
        const double gn = other(wn), gh = other(wh);
        RowExps(tn, lift, gn, &cold);
        RowExps(th, lift, gh, &cold);
        if (in && (gn != 0.0 || gh != 0.0)) flags[threadIdx.y][1] = 1;
    }
    entries(i + 1, 0, vn);
    entries(i, 1, vh);
    const RowTerms tn = terms(vn), th = terms(vh);
    const RowLifts lift(tn, th, &cold);
    const double gn = other(vn), gh = other(vh);
    const RowExps xn(tn, lift, gn, &cold), xh(th, lift, gh, &cold);
    // plain stores of the same value
    if (in && cold) flags[threadIdx.y][0] = 1;
    if (in && (gn != 0.0 || gh != 0.0 || N(i, N_C2I, jp) != 0.0 || N(i + 1, N_C2I, jp) != 0.0 ||
               H(i, H_PI, jp) != 0.0 || H(i - 1, H_PI, jp) != 0.0))
        flags[threadIdx.y][1] = 1;
    __syncthreads();
    if (!in) return;
    const int lane = jp & 31;
    unsigned char *block = out + ((size_t)i * (NP / 32) + jp / 32) * kAdjBytes;
    double *d = reinterpret_cast<double *>(block) + lane;
    const double f[kAdjF64] = {N(i, N_B, jp), N(i, N_PPR, jp), N(i, N_C2I, jp),
                               N(i + 1, N_B, jp), N(i + 1, N_PMR, jp), N(i + 1, N_C2I, jp),
                               H(i, H_HP, jp), H(i, H_PAR, jp), H(i, H_PI, jp),
                               H(i - 1, H_HQ, jp), H(i - 1, H_PCR, jp), H(i - 1, H_PI, jp)};
    for (int q = 0; q < kAdjF64; ++q, d += 32) *d = f[q];
    const bool none = flags[threadIdx.y][0] != 0;
    auto put = [&](const double (&v)[6], const RowExps &e) {
        for (int q = 0; q < 6; ++q, d += 32) {
            const int C = q == A_G1 || q == A_G2 ? e.g : q == A_KM ? e.f - lift.u : q == A_KP ? e.f - lift.d : e.f;
            *reinterpret_cast<int2 *>(d) = none ? make_int2(0, 0) : split_entry(v[q], C);
        }
    };
    put(vn, xn);
    put(vh, xh);
    int *x = reinterpret_cast<int *>(block + kAdjExps);
    x[lane] = xn.packed();
    x[32 + lane] = xh.packed();
    x[64 + lane] = lift.packed();
    if (lane < 4) x[96 + lane] = lane < 2 ? flags[threadIdx.y][lane] : 0;
}

// ---- sums ----

// Both sums of a column (half node), to the left (1) and to the right (2), for
// Phi_R and Phi_I, as integers T 2^(O - 1080).
struct AdjSums {
    long long T[2];
    int O[2];
};

// a + b, the smaller one's last places cut off (a place is below 2^-57 of the
// sum's bound), of either sign alike.
__device__ __forceinline__ AdjSums adj_add(const AdjSums &a, const AdjSums &b)
{
    AdjSums r;
#pragma unroll
    for (int g = 0; g < 2; ++g) {
        r.O[g] = max(a.O[g], b.O[g]);
        r.T[g] = shr_zero(a.T[g], r.O[g] - a.O[g]) + shr_zero(b.T[g], r.O[g] - b.O[g]);
    }
    return r;
}

__device__ __forceinline__ void adj_zero(AdjSums &a)
{
    a.T[0] = a.T[1] = 0;
    a.O[0] = a.O[1] = kSplitFloor;
}

// Both sums of the Pi values v[2], v[3] with the block of tab, whose head is
// given; whether the FP64 instructions are called for anywhere in the team, by
// the values or by the tables (a barrier of the team): the sums are then not
// valid, for any column that they go to.
template <int K, bool HALF>
__device__ __forceinline__ bool adj_pair(const double (&v)[4], const AdjTab<HALF> &tab, int2 head,
                                         AdjTeam<K> &team, AdjSums &s1, AdjSums &s2)
{
    const bool imag = head.y != 0;
    SplitInts p;
    split_ints<2>(v, p);
    int4 su, sd;
    int2 eu2, ed2;
    const bool hot = team.exchange(
        make_int4((int)(p.x[0] >> 32), (int)p.x[0], (int)(p.x[1] >> 32), (int)p.x[1]), make_int2(p.e[0], p.e[1]),
        head.x != 0 || max(p.e[0], p.e[1]) >= kSplitMaxExp, su, eu2, sd, ed2);
    // exponents of the products over the F class's: the largest of each sum
    const int rx = tab.row_exp(), cf = (short)(rx & 0xffff), cg = (rx >> 16) - cf;
    const int lx = tab.lifts(), lu = (short)(lx & 0xffff), ld = lx >> 16;
    int f[2];
    f[0] = max(max(eu2.x - lu, ed2.x - ld), max(p.e[0], kSplitFloor - cf));
    f[1] = max(max(eu2.y - lu, ed2.y - ld), max(p.e[1], kSplitFloor - cf));
    if (imag) {
        f[0] = max(f[0], p.e[1] + cg);
        f[1] = max(f[1], p.e[0] + cg);
    }
#pragma unroll
    for (int g = 0; g < 2; ++g) {
        const int uh = g ? su.z : su.x, ul = g ? su.w : su.y, eu = g ? eu2.y : eu2.x;
        const int dh = g ? sd.z : sd.x, dl = g ? sd.w : sd.y, ed = g ? ed2.y : ed2.x;
        const int2 l = limbs(cut(p.x[g], f[g] - p.e[g], p.j[g]));
        SplitSum a, b;
        a.add(limbs(cut(((long long)uh << 32) | (unsigned)ul, f[g] + lu - eu, nonzero(uh, ul))), tab.entry(A_KM));
        a.add(limbs(cut(((long long)dh << 32) | (unsigned)dl, f[g] + ld - ed, nonzero(dh, dl))), tab.entry(A_KP));
        b = a;
        a.add(l, tab.entry(A_F1));
        b.add(l, tab.entry(A_F2));
        if (imag) {   // the other part's, subtracted from the imaginary part
            int2 m = limbs(cut(p.x[1 - g], f[g] - cg - p.e[1 - g], p.j[1 - g]));
            if (g == 1) m = make_int2(-m.x, -m.y);
            a.add(m, tab.entry(A_G1));
            b.add(m, tab.entry(A_G2));
        }
        s1.T[g] = a.take();
        s2.T[g] = b.take();
        s1.O[g] = s2.O[g] = cf + f[g];
    }
    return hot;
}

// ---- eta and mu with the FP64 instructions alone (eta_half and mu_node) ----

// (KP x)(j-1) + (KM x)(j+1) of x = v[2], v[3], from the unsplit table's row.
template <int K>
__device__ __forceinline__ void cold_sources(const double (&v)[4], const double *kp, const double *km,
                                             AdjTeam<K> &team, double (&z)[2])
{
    double up[2], dn[2];
    team.neighbours(v[2], v[3], up, dn);
    const int row = 32 * team.h + team.lane;
    const double a = row > 0 ? kp[-1] : 0.0, b = row + 1 < 32 * K ? km[1] : 0.0;
    const FmaK<double> k1 = fma_k<double>();
#pragma unroll
    for (int g = 0; g < 2; ++g) z[g] = fma(a, dn[g], fma(b, up[g], k1.nz));
}

template <int NP>
__device__ __noinline__ Row4 cold_eta(Row4 a, Row4 c, double zaR, double zaI, double zcR, double zcI,
                                      const double *ta, const double *tc, double E)
{
    const FmaK<double> k1 = fma_k<double>();
    Row4 h;
    {
        const double B = ta[N_B * NP], FR = ta[N_FPR * NP], FI = ta[N_FPI * NP], PR = ta[N_PPR * NP],
                     CI = ta[N_C2I * NP];
        h.v[0] = fma(FI, a.v[3], fma(FR, a.v[2], fma(-B, a.v[0], fma(zaR, k1.one, zcR))));
        h.v[1] = fma(FR, a.v[3], fma(-FI, a.v[2], fma(-B, a.v[1], fma(zaI, k1.one, zcI))));
        h.v[2] = fma(CI, a.v[3], fma(PR, a.v[2], fma(E, a.v[0], k1.nz)));
        h.v[3] = fma(PR, a.v[3], fma(-CI, a.v[2], fma(E, a.v[1], k1.nz)));
    }
    const double B = tc[N_B * NP], FR = tc[N_FMR * NP], FI = tc[N_FMI * NP], PR = tc[N_PMR * NP],
                 CI = tc[N_C2I * NP];
    h.v[0] = fma(FI, c.v[3], fma(FR, c.v[2], fma(B, c.v[0], h.v[0])));
    h.v[1] = fma(FR, c.v[3], fma(-FI, c.v[2], fma(B, c.v[1], h.v[1])));
    h.v[2] = fma(CI, c.v[3], fma(PR, c.v[2], fma(E, c.v[0], h.v[2])));
    h.v[3] = fma(PR, c.v[3], fma(-CI, c.v[2], fma(E, c.v[1], h.v[3])));
    return h;
}

template <int NP>
__device__ __noinline__ Row4 cold_mu(Row4 l, Row4 p, Row4 m, double ypR, double ypI, double ymR, double ymI,
                                     const double *tp, const double *tm)
{
    const FmaK<double> k1 = fma_k<double>();
    Row4 o;
    {
        const double S = tp[H_HP * NP], FR = tp[H_FAR * NP], FI = tp[H_FAI * NP], PR = tp[H_PAR * NP],
                     PI = tp[H_PI * NP];
        o.v[0] = fma(FI, p.v[3], fma(FR, p.v[2], fma(S, p.v[0], fma(l.v[0], k1.one, fma(ypR, k1.one, ymR)))));
        o.v[1] = fma(FR, p.v[3], fma(-FI, p.v[2], fma(S, p.v[1], fma(l.v[1], k1.one, fma(ypI, k1.one, ymI)))));
        o.v[2] = fma(PI, p.v[3], fma(PR, p.v[2], fma(p.v[0], k1.one, l.v[2])));
        o.v[3] = fma(PR, p.v[3], fma(-PI, p.v[2], fma(p.v[1], k1.one, l.v[3])));
    }
    const double S = tm[H_HQ * NP], FR = tm[H_FCR * NP], FI = tm[H_FCI * NP], PR = tm[H_PCR * NP],
                 PI = tm[H_PI * NP];
    o.v[0] = fma(FI, m.v[3], fma(FR, m.v[2], fma(S, m.v[0], o.v[0])));
    o.v[1] = fma(FR, m.v[3], fma(-FI, m.v[2], fma(S, m.v[1], o.v[1])));
    o.v[2] = fma(PI, m.v[3], fma(PR, m.v[2], fma(m.v[0], k1.one, o.v[2])));
    o.v[3] = fma(PR, m.v[3], fma(-PI, m.v[2], fma(m.v[1], k1.one, o.v[3])));
    return o;
}

// ---- eta and mu on a lane's row, for lw_adjoint_column_kernel ----
// (the sweep below has the same operations in place: called from there, these
// cost it four bytes of spills and 1 % of its time)

// eta at the half node between columns with lam~ a and c, from their sums sa and
// sr; p: the table block of the left column.
__device__ __forceinline__ void eta_row(const double (&a)[4], const double (&c)[4], const AdjSums &sa, const AdjSums &sr,
                                        bool imag, const unsigned char *p, int lane, double E, const FmaK<double> &k1,
                                        double (&ep)[4])
{
    const AdjSums s = adj_add(sa, sr);
    const double BA = adj_f64(p, A_BA, lane), BC = adj_f64(p, A_BC, lane);
    const double PP = adj_f64(p, A_PP, lane), PM = adj_f64(p, A_PM, lane);
    ep[0] = fma(BC, c[0], fma(-BA, a[0], split_value(s.T[0], s.O[0])));
    ep[1] = fma(BC, c[1], fma(-BA, a[1], split_value(s.T[1], s.O[1])));
    double x = fma(E, c[0], fma(PP, a[2], fma(E, a[0], k1.nz)));
    double y = fma(E, c[1], fma(PP, a[3], fma(E, a[1], k1.nz)));
    if (imag) {
        const double CA = adj_f64(p, A_CA, lane), CC = adj_f64(p, A_CC, lane);
        x = fma(CC, c[3], fma(CA, a[3], x));
        y = fma(-CC, c[2], fma(-CA, a[2], y));
    }
    ep[2] = fma(PM, c[2], x);
    ep[3] = fma(PM, c[3], y);
}

// The same with the FP64 instructions alone; ta: the left column's row of the
// unsplit node table.
template <int K>
__device__ __forceinline__ void eta_row_cold(const double (&a)[4], const double (&c)[4], const double *ta, double E,
                                             AdjTeam<K> &team, double (&ep)[4])
{
    constexpr int NP = 32 * K;
    double za[2], zc[2];
    const double *tc = ta + kNCN * NP;
    cold_sources<K>(a, ta + N_KP * NP, ta + N_KM * NP, team, za);
    cold_sources<K>(c, tc + N_KP * NP, tc + N_KM * NP, team, zc);
    const Row4 r = cold_eta<NP>(row4(a), row4(c), za[0], za[1], zc[0], zc[1], ta, tc, E);
#pragma unroll
    for (int k = 0; k < 4; ++k) ep[k] = r.v[k];
}

// mu at a node from its lam~ a and eta right (ep) and left (em) of it with their
// sums s1 and sm.
__device__ __forceinline__ void mu_row(const double (&a)[4], const double (&ep)[4], const double (&em)[4],
                                       const AdjSums &s1, const AdjSums &sm, bool imag, const unsigned char *p, int lane,
                                       const FmaK<double> &k1, double (&o)[4])
{
    const AdjSums s = adj_add(s1, sm);
    const double HP = adj_f64(p, A_HP, lane), HQ = adj_f64(p, A_HQ, lane);
    const double PA = adj_f64(p, A_PA, lane), PC = adj_f64(p, A_PC, lane);
    o[0] = fma(HQ, em[0], fma(HP, ep[0], fma(a[0], k1.one, split_value(s.T[0], s.O[0]))));
    o[1] = fma(HQ, em[1], fma(HP, ep[1], fma(a[1], k1.one, split_value(s.T[1], s.O[1]))));
    double x = fma(em[0], k1.one, fma(PA, ep[2], fma(ep[0], k1.one, a[2])));
    double y = fma(em[1], k1.one, fma(PA, ep[3], fma(ep[1], k1.one, a[3])));
    if (imag) {
        const double PI = adj_f64(p, A_PI, lane), PJ = adj_f64(p, A_PJ, lane);
        x = fma(PJ, em[3], fma(PI, ep[3], x));
        y = fma(-PJ, em[2], fma(-PI, ep[2], y));
    }
    o[2] = fma(PC, em[2], x);
    o[3] = fma(PC, em[3], y);
}

// tp: the node's row of the unsplit half-node table.
template <int K>
__device__ __forceinline__ void mu_row_cold(const double (&a)[4], const double (&ep)[4], const double (&em)[4],
                                            const double *tp, AdjTeam<K> &team, double (&o)[4])
{
    constexpr int NP = 32 * K;
    double yp[2], ym[2];
    const double *tm = tp - kNCH * NP;
    cold_sources<K>(ep, tp + H_KP * NP, tp + H_KM * NP, team, yp);
    cold_sources<K>(em, tm + H_KP * NP, tm + H_KM * NP, team, ym);
    const Row4 r = cold_mu<NP>(row4(a), row4(ep), row4(em), yp[0], yp[1], ym[0], ym[1], tp, tm);
#pragma unroll
    for (int k = 0; k < 4; ++k) o[k] = r.v[k];
}

// ---- the sweep of one transposed step over a team's columns ----

struct AdjRing {
    alignas(16) unsigned char tab[2][kAdjBytes];
};

template <int K>
struct AdjSweep {
    AdjRing *ring;
    unsigned long long *bar;
    const unsigned char *tab;   // the warp's block of column 0
    const double *half64, *node64;
    int Nr;
    double E;                   // dt/2
    int *err;
    size_t pitch;               // bytes from a column's blocks to the next's, 0: one for all

    __device__ __forceinline__ void fetch(SplitRingState &st, int slot, int i, int lane) const
    {
        __syncwarp();
        if (lane == 0 && !(st.wait & kLost)) {
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            mbar_expect(&bar[slot], kAdjBytes);
            bulk_fetch(ring->tab[slot], tab + (size_t)i * pitch, kAdjBytes, &bar[slot]);
        }
        st.issue ^= 1u << slot;
    }
    __device__ __forceinline__ void await(SplitRingState &st, int slot) const
    {
        const unsigned parity = (st.wait >> slot) & 1u;
        if (!mbar_test(&bar[slot], parity)) {
            if (!(st.wait & kLost) && !mbar_wait(&bar[slot], parity, err)) {
                st.wait |= kLost;
                atomicExch(err, 1);
            }
            if (st.wait & kLost) return;
        }
        st.wait ^= 1u << slot;
    }
    __device__ __forceinline__ void drain(SplitRingState &st) const
    {
        for (int s = 0; s < 2; ++s)
            if (((st.wait ^ st.issue) >> s) & 1u) mbar_wait(&bar[s], (st.wait >> s) & 1u);
    }

    // Columns [i0, i1): as SplitSweep::run, load(i, l) giving lam~ of column i
    // (with the waveform gradient added, zero on the radial edges).  The edges'
    // own mu, which nothing uses, is stored as zero.
    template <typename Load, typename Right, typename Store>
    __device__ __forceinline__ void run(SplitRingState &st, AdjTeam<K> &team, Load load, int i0, int i1,
                                        bool again, Right before_right, Store store) const
    {
        constexpr int NP = 32 * K;
        const int row = 32 * team.h + team.lane, lane = team.lane;
        const FmaK<double> k1 = fma_k<double>();
        const int ib = i0 > 0 ? i0 - 1 : 0;
        const int ie = i1 < Nr - 1 ? i1 : Nr - 1;   // half nodes (blocks): [ib, ie)
        if (!(((st.wait ^ st.issue) >> st.cur) & 1u) && ib < ie) fetch(st, st.cur, ib, lane);
        double a[4], em[4], un[4];
        AdjSums sa, sm;        // sums to the left: of column i; to the right: of half node i - 1/2
        bool hot_a = false, hot_m = false;
        load(ib, a);
        if (ib + 1 == i1) before_right();
        if (ib + 1 < Nr) load(ib + 1, un);
#pragma unroll
        for (int k = 0; k < 4; ++k) em[k] = 0.0;
        adj_zero(sa);
        adj_zero(sm);
        if (ib > 0) {
            const unsigned char *block = tab + (size_t)(ib - 1) * pitch;
            const AdjTab<false> t{block, lane};
            AdjSums s2;
            hot_a = adj_pair<K, false>(a, t, t.head(), team, sa, s2);
        }
#pragma unroll 1
        for (int i = ib; i < i1; ++i) {
            double o[4];
            if (i + 1 < Nr) {
                double c[4], ep[4];
                AdjSums sc, sr, s1, s2;
                const int nx = i + 1 < ie ? i + 1 : again ? ib : -1;
                if (nx >= 0) fetch(st, st.cur ^ 1, nx, lane);
#pragma unroll
                for (int k = 0; k < 4; ++k) c[k] = un[k];
                if (i + 1 < i1) {
                    if (i + 2 == i1) before_right();
                    if (i + 2 < Nr) load(i + 2, un);
                }
                await(st, st.cur);
                const unsigned char *p = ring->tab[st.cur];
                st.cur ^= 1;
                const int2 head = AdjTab<false>{p, lane}.head();
                const bool imag = head.y != 0;
                // eta at half node i + 1/2
                const bool hot_c = adj_pair<K, false>(c, AdjTab<false>{p, lane}, head, team, sc, sr);
                if (hot_a || hot_c) {
                    double za[2], zc[2];
                    const double *ta = node64 + (size_t)i * (kNCN * NP) + row, *tc = ta + kNCN * NP;
                    cold_sources<K>(a, ta + N_KP * NP, ta + N_KM * NP, team, za);
                    cold_sources<K>(c, tc + N_KP * NP, tc + N_KM * NP, team, zc);
                    const Row4 r = cold_eta<NP>(row4(a), row4(c), za[0], za[1], zc[0], zc[1], ta, tc, E);
#pragma unroll
                    for (int k = 0; k < 4; ++k) ep[k] = r.v[k];
                } else {
                    const AdjSums s = adj_add(sa, sr);
                    const double BA = adj_f64(p, A_BA, lane), BC = adj_f64(p, A_BC, lane);
                    const double PP = adj_f64(p, A_PP, lane), PM = adj_f64(p, A_PM, lane);
                    ep[0] = fma(BC, c[0], fma(-BA, a[0], split_value(s.T[0], s.O[0])));
                    ep[1] = fma(BC, c[1], fma(-BA, a[1], split_value(s.T[1], s.O[1])));
                    double x = fma(E, c[0], fma(PP, a[2], fma(E, a[0], k1.nz)));
                    double y = fma(E, c[1], fma(PP, a[3], fma(E, a[1], k1.nz)));
                    if (imag) {
                        const double CA = adj_f64(p, A_CA, lane), CC = adj_f64(p, A_CC, lane);
                        x = fma(CC, c[3], fma(CA, a[3], x));
                        y = fma(-CC, c[2], fma(-CA, a[2], y));
                    }
                    ep[2] = fma(PM, c[2], x);
                    ep[3] = fma(PM, c[3], y);
                }
                // mu at node i
                const bool hot_p = adj_pair<K, true>(ep, AdjTab<true>{p, lane}, head, team, s1, s2);
                if (i >= i0) {
                    if (i == 0) {
#pragma unroll
                        for (int k = 0; k < 4; ++k) o[k] = 0.0;
                    } else if (hot_p || hot_m) {
                        double yp[2], ym[2];
                        const double *tp = half64 + (size_t)i * (kNCH * NP) + row, *tm = tp - kNCH * NP;
                        cold_sources<K>(ep, tp + H_KP * NP, tp + H_KM * NP, team, yp);
                        cold_sources<K>(em, tm + H_KP * NP, tm + H_KM * NP, team, ym);
                        const Row4 r = cold_mu<NP>(row4(a), row4(ep), row4(em), yp[0], yp[1], ym[0], ym[1], tp, tm);
#pragma unroll
                        for (int k = 0; k < 4; ++k) o[k] = r.v[k];
                    } else {
                        const AdjSums s = adj_add(s1, sm);
                        const double HP = adj_f64(p, A_HP, lane), HQ = adj_f64(p, A_HQ, lane);
                        const double PA = adj_f64(p, A_PA, lane), PC = adj_f64(p, A_PC, lane);
                        o[0] = fma(HQ, em[0], fma(HP, ep[0], fma(a[0], k1.one, split_value(s.T[0], s.O[0]))));
                        o[1] = fma(HQ, em[1], fma(HP, ep[1], fma(a[1], k1.one, split_value(s.T[1], s.O[1]))));
                        double x = fma(em[0], k1.one, fma(PA, ep[2], fma(ep[0], k1.one, a[2])));
                        double y = fma(em[1], k1.one, fma(PA, ep[3], fma(ep[1], k1.one, a[3])));
                        if (imag) {
                            const double PI = adj_f64(p, A_PI, lane), PJ = adj_f64(p, A_PJ, lane);
                            x = fma(PJ, em[3], fma(PI, ep[3], x));
                            y = fma(-PJ, em[2], fma(-PI, ep[2], y));
                        }
                        o[2] = fma(PC, em[2], x);
                        o[3] = fma(PC, em[3], y);
                    }
                    store(i, o);
                }
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    a[k] = c[k];
                    em[k] = ep[k];
                }
                sa = sc;
                sm = s2;
                hot_a = hot_c;
                hot_m = hot_p;
            } else {
#pragma unroll
                for (int k = 0; k < 4; ++k) o[k] = 0.0;
                store(i, o);
            }
        }
    }
};

}  // namespace
}  // namespace tk
