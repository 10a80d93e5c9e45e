// tk_coeffs.cu -- FP64 Kerr coefficient precompute on the device.
//
// 1. The tortoise coordinate (not printed in the paper) is inverted at every
//    radial node r*_i and half node r*_{i+1/2}: x = r - r+ is found by a
//    bracketed Newton iteration in y = ln x, so that Delta = x (r - r-) never
//    suffers the cancellation of r^2 - 2Mr + a^2 near the horizon.
// 2. The coefficients of the first-order system derived from Eq. 1 with the
//    m-mode ansatz of Eq. 2 (Sec. 3.2: "matrices D and S") are evaluated at
//    every (node, theta row) and (half node, theta row), multiplied out with
//    dt, dr*, dtheta into the step kernel's tables, and the angular boundary
//    conditions of Sec. 3.2 are folded into the first and last theta rows.
#include <math.h>
#include <algorithm>

#include "tk_internal.h"
#include "tk_split_tables.cuh"

namespace tk {
namespace {

// Horizons r+- = M +- sqrt(M^2 - a^2) and the tortoise log coefficients.
struct Geo {
    double M, a, rp, rm, Ap, Am;
    int s, m;
};

__device__ Geo geometry(const Kerr &K)
{
    Geo g;
    g.M = K.M;
    g.a = K.a;
    g.s = K.s;
    g.m = K.m;
    const double d = sqrt(K.M * K.M - K.a * K.a);
    g.rp = K.M + d;
    g.rm = K.M - d;
    g.Ap = 2.0 * K.M * g.rp / (g.rp - g.rm);
    g.Am = 2.0 * K.M * g.rm / (g.rp - g.rm);
    return g;
}

__device__ double rstar_of_x(const Geo &P, double x)
{
    // r* = r + Ap ln((r - r+)/2M) - Am ln((r - r-)/2M),  Ap = 2M r+/(r+ - r-),
    // Am = 2M r-/(r+ - r-); d r*/dr = (r^2 + a^2)/Delta.
    const double r = P.rp + x;
    return r + P.Ap * log(x / (2.0 * P.M)) - P.Am * log((r - P.rm) / (2.0 * P.M));
}

__device__ double x_of_rstar(const Geo &P, double target)
{
    // r*(e^y) is increasing in y with slope (r^2 + a^2)/(r - r-): Newton steps
    // inside a bracket [ylo, yhi] of the root, bisection when a step leaves it.
    // x >= max(r*, 2M) has r*(x) >= r* (the logarithms then add at least -M and
    // r+ >= M), which bounds the root from above.  Far out Newton starts from
    // there (r*(e^y) is convex, so it comes down monotonically), further in from
    // the horizon's asymptotics.  It ends when a step no longer changes y, or
    // only goes back to the value before: seven evaluations or fewer, each a
    // serial chain of some 100 FP64 instructions of 64 cycles (with the bracket
    // tested before the end, as once, a converged step fell out of it and up to
    // 52 bisections followed: 307 us for any grid, now 57 at 1601
    // radii and 75 at 4001).
    const double top = log(fmax(target, 2.0 * P.M));
    double ylo = -700.0, yhi = nextafter(top, 1e3);
    double y = (target > P.rp + 4.0 * P.M) ? top : (target - P.rp) / P.Ap + log(2.0 * P.M);
    y = fmin(y, top);
    if (!(y > ylo)) y = 0.5 * (ylo + yhi);
    double before = y;
    for (int it = 0; it < 200; ++it) {
        const double x = exp(y);
        const double r = P.rp + x;
        const double f = rstar_of_x(P, x) - target;
        if (f == 0.0) break;
        if (f < 0.0) ylo = y; else yhi = y;
        double yn = y - f * (r - P.rm) / (r * r + P.a * P.a);
        if (yn == y || yn == before) break;
        if (!(yn > ylo && yn < yhi)) {
            yn = 0.5 * (ylo + yhi);
            if (yn == ylo || yn == yhi) break;
        }
        before = y;
        y = yn;
    }
    return exp(y);
}

// What the coefficients need of a radius (x = r - r+), kRadial doubles.
struct Radial {
    double r, vp, Dl, dDl;       // r, varpi = r^2 + a^2, Delta = x (r - r-), d Delta / dr
    double tor;                  // dr/dr* = Delta / varpi
    double fs, fss;              // (d_* r^3)/r^3, (d_*^2 r^3)/r^3
    double ctr, cti0, cti1;      // Sigma^2 Re C_t, Sigma^2 Im C_t = cti0 + cti1 cos
    double e0, c3i;              // Sigma^2 E0, Sigma^2 Im c3
};
static_assert(sizeof(Radial) == kRadial * sizeof(double), "kRadial");

__device__ Radial radial_part(const Geo &P, double x)
{
    const double M = P.M, a = P.a, s = P.s, m = P.m;
    const double r = P.rp + x, r2 = r * r, a2 = a * a;
    Radial R;
    R.r = r;
    R.vp = r2 + a2;
    R.Dl = x * (r - P.rm);
    R.dDl = 2.0 * (r - M);
    R.tor = R.Dl / R.vp;
    R.fs = 3.0 * R.Dl / (r * R.vp);
    R.fss = R.tor * ((6.0 * r * R.Dl + 3.0 * r2 * R.dDl) / R.vp - 6.0 * r2 * r * R.Dl / (R.vp * R.vp)) / (r2 * r);
    R.ctr = 2.0 * s * (r * R.Dl - M * (r2 - a2));
    R.cti0 = 4.0 * M * a * m * r;
    R.cti1 = 2.0 * s * a * R.Dl;
    R.e0 = 2.0 * r * R.Dl + s * R.dDl * R.vp;
    R.c3i = 2.0 * m * s * a * (r - M);
    return R;
}

// Coefficients of   d_t Phi + b d_* Phi = Pi,
//                   d_t Pi - b d_* Pi - c1 d_* Phi = c2 Pi + c3 Phi + c4 Phi_thth + c5 Phi_th
// obtained from Eq. 1 x (-Delta/(Sigma^2 r^3)) with Psi = e^{i m phi} r^3 Phi and
// Pi = d_t Phi + b d_* Phi.  With the regularised variable Phi = w Phi^ the
// theta-singular potential is replaced by the constant -lambda0 and c5 gains
// the 2 w'/w term.
struct Raw {
    double b, c1r, c1i, c2r, c2i, c3r, c3i, c4, c5;
};

// What they need of a polar angle.
struct Angular {
    double sn, cs, g, V;
};

__device__ Angular angular_part(const Geo &P, int variable, double th)
{
    const double s = P.s, m = P.m;
    Angular A;
    sincos(th, &A.sn, &A.cs);
    if (variable == 0) {
        A.g = A.cs / A.sn;
        A.V = -(m + s * A.cs) * (m + s * A.cs) / (A.sn * A.sn) + s;
    } else {
        const double al = 0.5 * fabs(m + s), be = 0.5 * fabs(m - s);
        const int l0 = max(abs(P.m), abs(P.s));
        const double t2 = tan(0.5 * th);
        A.g = A.cs / A.sn + 2.0 * (al / t2 - be * t2);
        A.V = -(double)(l0 - P.s) * (double)(l0 + P.s + 1);
    }
    return A;
}

__device__ Raw raw_coefficients(const Geo &P, const double *__restrict__ rad, const Angular &A)
{
    const Radial R = *reinterpret_cast<const Radial *>(rad);
    const double a2 = P.a * P.a, m = P.m;
    const double sn2 = A.sn * A.sn;
    const double S2 = R.vp * R.vp - a2 * R.Dl * sn2; // Sigma^2
    const double Sg = sqrt(S2);
    const double b = R.vp / Sg;
    const double db = R.tor * (2.0 * R.r / Sg - R.vp * (4.0 * R.r * R.vp - a2 * R.dDl * sn2) / (2.0 * S2 * Sg));
    const double Ctr = R.ctr / S2;
    const double Cti = (R.cti0 + R.cti1 * A.cs) / S2;
    const double E0 = R.e0 / S2;
    const double c4 = R.Dl / S2;
    Raw o;
    o.b = b;
    o.c1r = b * Ctr + (2.0 * b * b * R.fs + E0) - b * db;
    o.c1i = b * Cti;
    o.c2r = -Ctr;
    o.c2i = -Cti;
    o.c3r = b * b * R.fss + E0 * R.fs + m * m * a2 / S2 + c4 * A.V;
    o.c3i = R.c3i / S2;
    o.c4 = c4;
    o.c5 = c4 * A.g;
    return o;
}

// w(theta) = (1 - cos)^{|m+s|/2} (1 + cos)^{|m-s|/2}, written with half angles
// (1 - cos = 2 sin^2, 1 + cos = 2 cos^2) so that nothing cancels near the poles.
__device__ double weight_w(int s, int m, double th)
{
    const double sh = sin(0.5 * th), ch = cos(0.5 * th);
    return pow(2.0 * sh * sh, 0.5 * fabs((double)(m + s))) * pow(2.0 * ch * ch, 0.5 * fabs((double)(m - s)));
}

__device__ double sl_weight(int s, int m, double th)
{
    const double w = weight_w(s, m, th);
    return sin(th) * w * w;
}

// Self-adjoint stencil of the regularised angular operator on cell j:
//   (1/P)(P F')'  ->  [P_{j+1}(F_{j+1} - F_j) - P_j (F_j - F_{j-1})] / (Q_j dth^2),
// P = sin(theta) w^2 at the faces theta = f dth (zero on both poles), Q_j the
// mean of P over the cell by 4-point Gauss-Legendre on 64 sub-panels.
// ang[j] = P_{j+1}/(Q_j dth^2), ang[NP + j] = P_j/(Q_j dth^2); zero on padding rows.
// One block per row j, one thread per Gauss point (each evaluation is a serial
// chain of two powers, a sine and a cosine: ~10 us, so all of them at once);
// then the first warp adds them, lane l those of sub-panels l and l + 32, and
// the 32 partial sums in a fixed tree order: 32 us, with a warp per row that
// took two panels a lane in turn 88.
constexpr int kStencilPanels = 64;

__device__ void stencil_row(int j, int s, int m, int Nth, int NP, double *__restrict__ ang)
{
    __shared__ double val[kStencilPanels][4], face[2];
    const int tid = threadIdx.x;
    if (j >= Nth) {
        if (tid == 0) {
            ang[j] = 0.0;
            ang[NP + j] = 0.0;
        }
        return;
    }
    const double dth = M_PI / Nth;
    const double xg[2] = {0.3399810435848563, 0.8611363115940526};
    const double wg[2] = {0.6521451548625461, 0.3478548451374538};
    const double h = dth / kStencilPanels;
    {
        const int k = tid >> 2, g = (tid >> 1) & 1;
        const double c = j * dth + (k + 0.5) * h;
        val[k][tid & 3] = sl_weight(s, m, (tid & 1) ? c + 0.5 * h * xg[g] : c - 0.5 * h * xg[g]);
    }
    if (tid < 2) face[tid] = (j + tid == 0 || j + tid == Nth) ? 0.0 : sl_weight(s, m, (j + tid) * dth);
    __syncthreads();
    if (tid >= 32) return;
    double acc = 0.0;
    for (int k = tid; k < kStencilPanels; k += 32)
        for (int g = 0; g < 2; ++g) acc += wg[g] * (val[k][2 * g] + val[k][2 * g + 1]);
    for (int off = 16; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
    if (tid != 0) return;
    const double Q = 0.5 * h * acc / dth;
    ang[j] = face[1] / (Q * dth * dth);
    ang[NP + j] = face[0] / (Q * dth * dth);
}

// The tortoise inversion with the radial parts, and beside it the angular
// stencil: both are serial chains that leave most of the chip idle and share
// nothing, so one launch holds the blocks of both (blockIdx.x < ninv: the
// inversion's).  61 us for both at 1601 x 32 and 79 at 4001 x 64; one after the
// other 57 + 32 and 75 + 32.  The stencil is the same for every black hole of
// the set.
//
// Radii: nodes i in rad[i], half nodes i + 1/2 in rad[Nr + i]; black hole
// blockIdx.y of the set goes to rad + blockIdx.y 2 Nr kRadial.  The first `use`
// threads of a block take a radius each: one warp a block while the warps do
// not exceed the SMs, then more.
constexpr int kPartsThreads = 4 * kStencilPanels;

__global__ void __launch_bounds__(kPartsThreads)
radial_stencil_kernel(const __grid_constant__ KerrSet kp, double rs_min, double drs, int Nr, double *rad, int ninv,
                      int use, int Nth, int NP, double *__restrict__ ang)
{
    if ((int)blockIdx.x >= ninv) {
        if (blockIdx.y == 0) stencil_row((int)blockIdx.x - ninv, kp.k[0].s, kp.k[0].m, Nth, NP, ang);
        return;
    }
    const int k = blockIdx.x * use + threadIdx.x;
    if ((int)threadIdx.x >= use || k >= 2 * Nr - 1) return;
    const Geo P = geometry(kp.k[blockIdx.y]);
    rad += (size_t)blockIdx.y * 2 * Nr * kRadial;
    const double rs = k < Nr ? rs_min + k * drs : rs_min + (k - Nr + 0.5) * drs;
    *reinterpret_cast<Radial *>(rad + (size_t)k * kRadial) = radial_part(P, x_of_rstar(P, rs));
}

// Raw coefficients supplied by the caller: [9][Nth][Nr] in the order of Raw
// (b, c1 re/im, c2 re/im, c3 re/im, c4, c5).
__device__ Raw raw_from(const double *__restrict__ r, int Nth, int Nr, int jp, int i)
{
    const size_t plane = (size_t)Nth * Nr, k = (size_t)jp * Nr + i;
    Raw c;
    c.b = r[k];
    c.c1r = r[plane + k];
    c.c1i = r[2 * plane + k];
    c.c2r = r[3 * plane + k];
    c.c2i = r[4 * plane + k];
    c.c3r = r[5 * plane + k];
    c.c3i = r[6 * plane + k];
    c.c4 = r[7 * plane + k];
    c.c5 = r[8 * plane + k];
    return c;
}

// What the tables hold of one point.
struct Entries {
    double hv[kNCH], nv[kNCN];   // half node i + 1/2, node i
    double bn;                   // b at the node
    double c4n, c4h;             // c4 at the node and at the half node
    double gpv, gmv;             // theta-only stencil factors of the row
};

// Of row jp < NP (polar angle th) and column i; all zero outside the grid.
__device__ __forceinline__ void table_entries(const Geo &P, int variable, int Nr, int Nth, int NP, Divisor ds, Divisor de, double dt,
                                              double dth, double th, int i, int jp, const double *__restrict__ rad,
                                              const double *__restrict__ ang, const Angular &A,
                                              const double *__restrict__ raw_node,
                                              const double *__restrict__ raw_half, Entries &E)
{
    double (&hv)[kNCH] = E.hv, (&nv)[kNCN] = E.nv;
    for (int q = 0; q < kNCH; ++q) hv[q] = 0.0;
    for (int q = 0; q < kNCN; ++q) nv[q] = 0.0;
    E.bn = E.c4n = E.c4h = E.gpv = E.gmv = 0.0;
    const double ith2 = 1.0 / (dth * dth), i2th = 1.0 / (2.0 * dth);
    const double p = (variable == 0 && (abs(P.m) & 1)) ? -1.0 : 1.0;   // ghost parity
    if (jp < Nth && i < Nr) {
        // angular stencil A+ (row j+1), A- (row j-1); the centre gets -(A+ + A-)
        //   literal:     A+- = 1/dth^2 +- cot(theta)/(2 dth) times c4, i.e. c4/dth^2 +- c5/(2 dth)
        //   regularised: A+- = c4 ang[.]  (self-adjoint form, no ghosts)
        const double Ap = (variable != 0) ? ang[jp] : 0.0;
        const double Am = (variable != 0) ? ang[NP + jp] : 0.0;
        if (variable != 0) {
            E.gpv = Ap;
            E.gmv = Am;
        } else {
            double sn, cs;
            sincos(th, &sn, &cs);
            E.gpv = (jp == Nth - 1) ? 0.0 : ith2 + (cs / sn) * i2th;   // ghosts folded on the edge rows
            E.gmv = (jp == 0) ? 0.0 : ith2 - (cs / sn) * i2th;
        }
        {   // node r*_i, Eq. (lw2), step dt
            const Raw c = raw_node ? raw_from(raw_node, Nth, Nr, jp, i)
                                   : raw_coefficients(P, rad + (size_t)i * kRadial, A);
            E.bn = c.b;
            if (i > 0 && i < Nr - 1) {
                E.c4n = c.c4;
                const double h2 = 0.5 * dt;
                const double B = ds.under(dt * c.b);
                const double g1r = ds.under(dt * c.c1r), g1i = ds.under(dt * c.c1i);
                double kp, km;
                if (variable == 0) {
                    kp = h2 * (c.c4 * ith2 + c.c5 * i2th);
                    km = h2 * (c.c4 * ith2 - c.c5 * i2th);
                } else {
                    kp = h2 * c.c4 * Ap;
                    km = h2 * c.c4 * Am;
                }
                const double dg = kp + km;
                double fpr = g1r + h2 * c.c3r - dg, fmr = -g1r + h2 * c.c3r - dg;
                if (variable == 0 && jp == 0) { fpr += p * km; fmr += p * km; km = 0.0; }
                if (variable == 0 && jp == Nth - 1) { fpr += p * kp; fmr += p * kp; kp = 0.0; }
                // entries that multiply half-node Phi values carry the factor eh
                // (the half node returns Phi / eh, see the half-node tables)
                const double eh = 0.25 * dt;
                nv[N_B] = eh * B;
                nv[N_PPR] = B + h2 * c.c2r;
                nv[N_PMR] = -B + h2 * c.c2r;
                nv[N_C2I] = h2 * c.c2i;
                nv[N_FPR] = eh * fpr;
                nv[N_FPI] = eh * (g1i + h2 * c.c3i);
                nv[N_FMR] = eh * fmr;
                nv[N_FMI] = eh * (-g1i + h2 * c.c3i);
                nv[N_KP] = eh * kp;
                nv[N_KM] = eh * km;
            }
        }
        if (i < Nr - 1) {   // half node r*_{i+1/2}, Eq. (lw1), step dt/2
            const Raw c = raw_half ? raw_from(raw_half, Nth, Nr, jp, i)
                                   : raw_coefficients(P, rad + (size_t)(Nr + i) * kRadial, A);
            E.c4h = c.c4;
            const double dtau = 0.5 * dt, e2 = 0.5 * dtau;
            const double B = ds.under(dtau * c.b);
            const double g1r = ds.under(dtau * c.c1r), g1i = ds.under(dtau * c.c1i);
            double kp, km;
            if (variable == 0) {
                kp = e2 * (c.c4 * ith2 + c.c5 * i2th);
                km = e2 * (c.c4 * ith2 - c.c5 * i2th);
            } else {
                kp = e2 * c.c4 * Ap;
                km = e2 * c.c4 * Am;
            }
            const double dg = kp + km;
            double far = -g1r + e2 * c.c3r - dg, fcr = g1r + e2 * c.c3r - dg;
            if (variable == 0 && jp == 0) { far += p * km; fcr += p * km; km = 0.0; }
            if (variable == 0 && jp == Nth - 1) { far += p * kp; fcr += p * kp; kp = 0.0; }
            // the Phi half-node value is returned divided by e2 (= eh): its
            // Pi term e2 (Pi_a + Pi_c) then needs no multiplication
            hv[H_HP] = de.under(0.5 + B);
            hv[H_HQ] = de.under(0.5 - B);
            hv[H_PAR] = 0.5 - B + e2 * c.c2r;
            hv[H_PCR] = 0.5 + B + e2 * c.c2r;
            hv[H_PI] = e2 * c.c2i;
            hv[H_FAR] = far;
            hv[H_FAI] = -g1i + e2 * c.c3i;
            hv[H_FCR] = fcr;
            hv[H_FCI] = g1i + e2 * c.c3i;
            hv[H_KP] = kp;
            hv[H_KM] = km;
        }
    }
}

// One thread per point, a block holding all NP rows of its columns (blockDim.x
// = NP): a column's flags in the step tables are over its rows.  Bound by the
// FP64 pipe: what depends on the radius alone comes from the inversion kernel,
// what depends on the angle alone is formed once per thread, which takes
// columns in turns (with both formed at every point 372 us at 4001 x 64, now
// 217; with the divisions by dr* and e as multiplications where these are powers
// of two 193, 198 with the lifts of the step's tables).
constexpr int kTableThreads = 256;

template <typename T>
__global__ void __launch_bounds__(kTableThreads)
coeff_tables_kernel(Kerr KP, int variable, int Nr, int Nth, int NP, Divisor ds, Divisor de, double dt,
                    const double *__restrict__ rad, const double *__restrict__ ang, T *__restrict__ half,
                    T *__restrict__ node, double *__restrict__ b_node, double *__restrict__ w_row,
                    float *__restrict__ cmp, float *__restrict__ gpm, F32Derive fd,
                    const double *__restrict__ raw_node, const double *__restrict__ raw_half,
                    unsigned char *__restrict__ step)
{
    __shared__ int flags[kTableThreads / 32][2];   // per column: cold, has imaginary coefficients
    const int jp = threadIdx.x;
    const Geo P = geometry(KP);
    const double dth = M_PI / Nth;
    const double th = (jp + 0.5) * dth;
    const Angular A = (jp < Nth && !raw_node) ? angular_part(P, variable, th) : Angular{};
    // the columns of the grid in turns (the row's angular part is formed once)
    for (int c0 = blockIdx.x * blockDim.y; c0 < Nr; c0 += gridDim.x * blockDim.y) {
        const int i = c0 + threadIdx.y;
        if (step) {
            const int k = threadIdx.y * blockDim.x + threadIdx.x;
            __syncthreads();
            if (k < kTableThreads / 32 * 2) (&flags[0][0])[k] = 0;
            __syncthreads();
        }
        T *hcol = half + (size_t)i * kNCH * NP + jp;
        T *ncol = node + (size_t)i * kNCN * NP + jp;
        Entries E;
        table_entries(P, variable, Nr, Nth, NP, ds, de, dt, dth, th, i, jp, rad, ang, A, raw_node, raw_half, E);
        const double (&hv)[kNCH] = E.hv, (&nv)[kNCN] = E.nv;
        if (i == 0 && w_row)
            w_row[jp] = jp >= Nth ? 0.0 : (variable != 0) ? weight_w(P.s, P.m, th) : 1.0;
        if (step) {
            const double hd[kStepHalfF64] = {hv[H_HP], hv[H_HQ], hv[H_PAR], hv[H_PCR], hv[H_PI]};
            const double hs[kSplitEntries] = {hv[H_FAR], hv[H_FCR], hv[H_KP], hv[H_KM], hv[H_FAI], hv[H_FCI]};
            const double nd[kStepNodeF64] = {nv[N_B], nv[N_PPR], nv[N_PMR], nv[N_C2I]};
            const double ns[kSplitEntries] = {nv[N_FMR], nv[N_FPR], nv[N_KP], nv[N_KM], nv[N_FMI], nv[N_FPI]};
            int cold = 0;
            auto terms = [](const double *v) {
                return RowTerms{fabs(v[S_FA]) + fabs(v[S_FC]), 2.0 * fabs(v[S_KP]), 2.0 * fabs(v[S_KM])};
            };
            auto other = [](const double *v) { return fabs(v[S_GA]) + fabs(v[S_GC]); };
            const RowTerms ht = terms(hs), nt = terms(ns);
            const double hg = other(hs), ng = other(ns);
            const RowLifts lift(ht, nt, &cold);
            const RowExps hx(ht, lift, hg, &cold), nx(nt, lift, ng, &cold);
            // plain stores of the same value
            if (cold) flags[threadIdx.y][0] = 1;
            if (hg != 0.0 || ng != 0.0 || hv[H_PI] != 0.0 || nv[N_C2I] != 0.0) flags[threadIdx.y][1] = 1;
            __syncthreads();
            if (i < Nr) {
                const int lane = jp & 31;
                unsigned char *block = step + ((size_t)i * (NP / 32) + jp / 32) * kStepBytes;
                double *d = reinterpret_cast<double *>(block) + lane;
                auto entries = [&](const double *v, const RowExps &e) {
                    for (int q = 0; q < kSplitEntries; ++q, d += 32) {
                        const int C = q >= S_GA ? e.g : q == S_KP ? e.f - lift.u : q == S_KM ? e.f - lift.d : e.f;
                        *reinterpret_cast<int2 *>(d) = flags[threadIdx.y][0] ? make_int2(0, 0) : split_entry(v[q], C);
                    }
                };
                for (int q = 0; q < kStepHalfF64; ++q, d += 32) *d = hd[q];
                entries(hs, hx);
                for (int q = 0; q < kStepNodeF64; ++q, d += 32) *d = nd[q];
                entries(ns, nx);
                int *x = reinterpret_cast<int *>(block + kStepExps);
                x[lane] = hx.packed();
                x[32 + lane] = nx.packed();
                x[64 + lane] = lift.packed();
                if (lane < 4) x[96 + lane] = lane < 2 ? flags[threadIdx.y][lane] : 0;
            }
        }
        if (i >= Nr) continue;
        if constexpr (sizeof(T) == 4) {
            // FP32: sixteen entries rounded from FP64, the other five derived from
            // them in FP32 exactly as the compact-table kernel derives them
            float cv[kNCC];
            cv[C_HP] = (float)hv[H_HP];
            cv[C_PAR] = (float)hv[H_PAR];
            cv[C_PI] = (float)hv[H_PI];
            cv[C_FAR] = (float)hv[H_FAR];
            cv[C_FAI] = (float)hv[H_FAI];
            cv[C_FCR] = (float)hv[H_FCR];
            cv[C_FCI] = (float)hv[H_FCI];
            cv[C_C4H] = (jp < Nth && i < Nr - 1) ? (float)(0.25 * dt * E.c4h) : 0.0f;
            cv[C_B] = (float)nv[N_B];
            cv[C_PMR] = (float)nv[N_PMR];
            cv[C_C2I] = (float)nv[N_C2I];
            cv[C_FPR] = (float)nv[N_FPR];
            cv[C_FPI] = (float)nv[N_FPI];
            cv[C_FMR] = (float)nv[N_FMR];
            cv[C_FMI] = (float)nv[N_FMI];
            cv[C_C4N] = (jp < Nth && i > 0 && i < Nr - 1) ? (float)(0.25 * dt * 0.5 * dt * E.c4n) : 0.0f;
            const float gp = (float)E.gpv, gm = (float)E.gmv;
            if (i == 0 && gpm) {
                gpm[jp] = gp;
                gpm[NP + jp] = gm;
            }
            float h32[kNCH], n32[kNCN];
            h32[H_HP] = cv[C_HP];
            h32[H_HQ] = __fadd_rn(fd.ih, -cv[C_HP]);
            h32[H_PAR] = cv[C_PAR];
            h32[H_PCR] = __fadd_rn(cv[C_PAR], __fmaf_rn(fd.t2, cv[C_HP], -1.0f));
            h32[H_PI] = cv[C_PI];
            h32[H_FAR] = cv[C_FAR];
            h32[H_FAI] = cv[C_FAI];
            h32[H_FCR] = cv[C_FCR];
            h32[H_FCI] = cv[C_FCI];
            h32[H_KP] = __fmul_rn(cv[C_C4H], gp);
            h32[H_KM] = __fmul_rn(cv[C_C4H], gm);
            n32[N_B] = cv[C_B];
            n32[N_PPR] = __fmaf_rn(fd.bn2, cv[C_B], cv[C_PMR]);
            n32[N_PMR] = cv[C_PMR];
            n32[N_C2I] = cv[C_C2I];
            n32[N_FPR] = cv[C_FPR];
            n32[N_FPI] = cv[C_FPI];
            n32[N_FMR] = cv[C_FMR];
            n32[N_FMI] = cv[C_FMI];
            n32[N_KP] = __fmul_rn(cv[C_C4N], gp);
            n32[N_KM] = __fmul_rn(cv[C_C4N], gm);
            for (int q = 0; q < kNCH; ++q) hcol[(size_t)q * NP] = h32[q];
            for (int q = 0; q < kNCN; ++q) ncol[(size_t)q * NP] = n32[q];
            if (cmp) {
                float *ccol = cmp + (size_t)i * kNCC * NP + jp;
                for (int q = 0; q < kNCC; ++q) ccol[(size_t)q * NP] = cv[q];
            }
        } else {
            for (int q = 0; q < kNCH; ++q) hcol[(size_t)q * NP] = (T)hv[q];
            for (int q = 0; q < kNCN; ++q) ncol[(size_t)q * NP] = (T)nv[q];
        }
        b_node[(size_t)i * NP + jp] = E.bn;
    }
}

// The tables' derivative in a parameter of the black hole: the sum over q of
// w[q] times the tables of kp.k[q], whose radial parts are rad[q].  One pass:
// the tables of the shifted parameters stay in registers.  Bound by the FP64
// pipe: 187 us at 1601 x 32; with each shifted table written out and added by
// kernels of their own the four took 350 us and twice the table memory.
__global__ void __launch_bounds__(kTableThreads)
table_derivative_kernel(const __grid_constant__ KerrSet kp, int variable, int Nr, int Nth, int NP, Divisor ds,
                        Divisor de, double dt,
                        const double *__restrict__ rad, const double *__restrict__ ang, double *__restrict__ half,
                        double *__restrict__ node, double *__restrict__ b_node)
{
    const int jp = threadIdx.x;
    const double dth = M_PI / Nth;
    const double th = (jp + 0.5) * dth;
    const Angular A = jp < Nth ? angular_part(geometry(kp.k[0]), variable, th) : Angular{};
    for (int i = blockIdx.x * blockDim.y + threadIdx.y; i < Nr; i += gridDim.x * blockDim.y) {
        double v[kNCH + kNCN + 1];
#pragma unroll
        for (int k = 0; k < kNCH + kNCN + 1; ++k) v[k] = 0.0;
#pragma unroll 1
        for (int q = 0; q < kShifts; ++q) {
            Entries E;
            table_entries(geometry(kp.k[q]), variable, Nr, Nth, NP, ds, de, dt, dth, th, i, jp,
                          rad + (size_t)q * 2 * Nr * kRadial, ang, A, nullptr, nullptr, E);
            const double w = kp.w[q];
#pragma unroll
            for (int k = 0; k < kNCH; ++k) v[k] = fma(w, E.hv[k], v[k]);
#pragma unroll
            for (int k = 0; k < kNCN; ++k) v[kNCH + k] = fma(w, E.nv[k], v[kNCH + k]);
            v[kNCH + kNCN] = fma(w, E.bn, v[kNCH + kNCN]);
        }
#pragma unroll
        for (int k = 0; k < kNCH; ++k) half[((size_t)i * kNCH + k) * NP + jp] = v[k];
#pragma unroll
        for (int k = 0; k < kNCN; ++k) node[((size_t)i * kNCN + k) * NP + jp] = v[kNCH + k];
        b_node[(size_t)i * NP + jp] = v[kNCH + kNCN];
    }
}

// The raw coefficients the precompute forms, [9][Nth][Nr] in the order of Raw,
// at the nodes and (column i < Nr - 1) the half nodes r*_{i+1/2}; column
// Nr - 1 of the half table is zero.  Grid-stride over the Nth * Nr points.
__global__ void raw_export_kernel(Kerr KP, int variable, int Nr, int Nth,
                                  const double *__restrict__ rad, double *__restrict__ out_node,
                                  double *__restrict__ out_half)
{
    const Geo P = geometry(KP);
    const size_t plane = (size_t)Nth * Nr;
    for (size_t k = (size_t)blockIdx.x * blockDim.x + threadIdx.x; k < plane;
         k += (size_t)gridDim.x * blockDim.x) {
        const int jp = (int)(k / Nr), i = (int)(k % Nr);
        const double th = (jp + 0.5) * (M_PI / Nth);
        const Angular A = angular_part(P, variable, th);
        const Raw c = raw_coefficients(P, rad + (size_t)i * kRadial, A);
        const double v[9] = {c.b, c.c1r, c.c1i, c.c2r, c.c2i, c.c3r, c.c3i, c.c4, c.c5};
        for (int q = 0; q < 9; ++q) out_node[q * plane + k] = v[q];
        Raw h = {};
        if (i < Nr - 1) h = raw_coefficients(P, rad + (size_t)(Nr + i) * kRadial, A);
        const double w[9] = {h.b, h.c1r, h.c1i, h.c2r, h.c2i, h.c3r, h.c3i, h.c4, h.c5};
        for (int q = 0; q < 9; ++q) out_half[q * plane + k] = w[q];
    }
}

// Stiffness of the source term at every interior node: a Gershgorin bound on
// the spectrum of the Phi -> Pi coupling c3 + c4 (angular stencil), i.e. on
// omega^2 of the fastest angular oscillation, and the radial speed b.  The two
// maxima are written as the bit patterns of non-negative doubles, which order
// like unsigned integers: out[0] = max omega^2, out[1] = max b.
__global__ void stiffness_kernel(Kerr KP, int variable, int Nr, int Nth, int NP,
                                 const double *__restrict__ rad, const double *__restrict__ ang,
                                 unsigned long long *__restrict__ out)
{
    const int jp = blockIdx.x * blockDim.x + threadIdx.x;
    const int i = blockIdx.y * blockDim.y + threadIdx.y;
    double w2 = 0.0, bb = 0.0;
    if (jp < Nth && i > 0 && i < Nr - 1) {
        const Geo P = geometry(KP);
        const double dth = M_PI / Nth;
        const double th = (jp + 0.5) * dth;
        const Raw c = raw_coefficients(P, rad + (size_t)i * kRadial, angular_part(P, variable, th));
        const double asum = (variable != 0) ? ang[jp] + ang[NP + jp] : 2.0 / (dth * dth);
        w2 = sqrt(c.c3r * c.c3r + c.c3i * c.c3i) + 2.0 * c.c4 * asum;
        bb = c.b;
    }
    // warp maximum, then one atomic per warp
    for (int off = 16; off > 0; off >>= 1) {
        w2 = fmax(w2, __shfl_xor_sync(0xffffffffu, w2, off));
        bb = fmax(bb, __shfl_xor_sync(0xffffffffu, bb, off));
    }
    if ((threadIdx.x & 31) == 0) {
        atomicMax(out, (unsigned long long)__double_as_longlong(w2));
        atomicMax(out + 1, (unsigned long long)__double_as_longlong(bb));
    }
}

}  // namespace

cudaError_t launch_stiffness(const Kerr &P, int variable, int Nr, int Ntheta, int NP,
                             const double *rad, const double *ang, unsigned long long *out,
                             cudaStream_t st)
{
    cudaError_t e = cudaMemsetAsync(out, 0, 2 * sizeof(unsigned long long), st);
    if (e != cudaSuccess) return e;
    dim3 block(32, 8), grid((NP + 31) / 32, (Nr + 7) / 8);
    stiffness_kernel<<<grid, block, 0, st>>>(P, variable, Nr, Ntheta, NP, rad, ang, out);
    return cudaGetLastError();
}

cudaError_t launch_raw_export(const Kerr &P, int variable, int Nr, int Ntheta, const double *rad, double *out_node,
                              double *out_half, int num_sms, cudaStream_t st)
{
    const size_t n = (size_t)Ntheta * Nr;
    const int blocks = (int)std::min<size_t>((n + 255) / 256, num_sms * 8);
    raw_export_kernel<<<blocks, 256, 0, st>>>(P, variable, Nr, Ntheta, rad, out_node, out_half);
    return cudaGetLastError();
}

// n black holes of the set; ang NULL: the stencil is not wanted.
static cudaError_t launch_parts(const KerrSet &kp, int n, double rs_min, double drs, int Nr, double *rad, int Ntheta,
                                int NP, double *ang, int num_sms, cudaStream_t st)
{
    const int warps = (2 * Nr + 30) / 32;
    const int use = 32 * std::min(kPartsThreads / 32, std::max(1, warps / num_sms));
    const int ninv = (2 * Nr - 1 + use - 1) / use;
    radial_stencil_kernel<<<dim3(ninv + (ang ? NP : 0), n), kPartsThreads, 0, st>>>(kp, rs_min, drs, Nr, rad, ninv,
                                                                                    use, Ntheta, NP, ang);
    return cudaGetLastError();
}

cudaError_t launch_radial_parts(const Kerr &P, double rs_min, double drs, int Nr, double *rad, int Ntheta, int NP,
                                double *ang, int num_sms, cudaStream_t st)
{
    KerrSet kp = {};
    kp.k[0] = P;
    return launch_parts(kp, 1, rs_min, drs, Nr, rad, Ntheta, NP, ang, num_sms, st);
}

// at most four blocks per SM, whose threads take the columns in turns
static dim3 table_grid(int Nr, const dim3 &block, int num_sms)
{
    return dim3(std::min<unsigned>((Nr + block.y - 1) / block.y, num_sms * 4));
}

cudaError_t launch_table_derivative(const KerrSet &kp, int variable, double rs_min, int Nr, int Ntheta, int NP,
                                    double drs, double dt_inner, double *rad, double *ang, double *half,
                                    double *node, double *b_node, int num_sms, cudaStream_t st)
{
    cudaError_t e = launch_parts(kp, kShifts, rs_min, drs, Nr, rad, Ntheta, NP, variable != 0 ? ang : nullptr, num_sms,
                                 st);
    if (e != cudaSuccess) return e;
    const dim3 block(NP, kTableThreads / NP);
    table_derivative_kernel<<<table_grid(Nr, block, num_sms), block, 0, st>>>(
        kp, variable, Nr, Ntheta, NP, divisor(drs), divisor(0.25 * dt_inner), dt_inner, rad, ang, half, node, b_node);
    return cudaGetLastError();
}

cudaError_t launch_coeff_tables(const Kerr &P, int variable, int Nr, int Ntheta, int NP,
                                double drs, double dt_inner, const double *rad, const double *ang, int precision, void *half,
                                void *node, double *b_node, double *w_row, float *cmp, float *gpm,
                                int num_sms, cudaStream_t st, const double *raw_node, const double *raw_half,
                                unsigned char *step)
{
    const F32Derive fd = f32_derive(dt_inner);
    dim3 block(NP, kTableThreads / NP);
    const dim3 grid = table_grid(Nr, block, num_sms);
    const Divisor ds = divisor(drs), de = divisor(0.25 * dt_inner);   // dr*, the half node's e
    if (precision == 0)
        coeff_tables_kernel<double><<<grid, block, 0, st>>>(P, variable, Nr, Ntheta, NP, ds, de, dt_inner,
                                                             rad, ang, (double *)half,
                                                             (double *)node, b_node, w_row, nullptr,
                                                             nullptr, fd, raw_node, raw_half, step);
    else
        coeff_tables_kernel<float><<<grid, block, 0, st>>>(P, variable, Nr, Ntheta, NP, ds, de, dt_inner,
                                                            rad, ang, (float *)half,
                                                            (float *)node, b_node, w_row, cmp, gpm, fd,
                                                            raw_node, raw_half, nullptr);
    return cudaGetLastError();
}

}  // namespace tk
