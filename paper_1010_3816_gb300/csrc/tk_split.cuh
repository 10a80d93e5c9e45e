// tk_split.cuh -- the FP64 Lax-Wendroff step with its Phi -> Pi coupling in
// integers.
//
// GB300's FP64 pipe takes 64 cycles per warp instruction and sub-partition, its
// 32 x 32 + 64 bit integer multiply-add takes 2, and the two run side by side.
// A step needs 54 FP64 instructions per update; 26 of them form the coupling of
// Phi to Pi,
//   FA Phi_a + FC Phi_c + KP (Phi_a + Phi_c)(j+1) + KM (Phi_a + Phi_c)(j-1)
//   +- [GA Phi_a + GC Phi_c of the other part],
// twice (half node and node) for two components, and its sums.  Here these dot
// products are formed in integers, 3 integer multiply-adds per product, and
// enter the FP64 chain as one addend: 28 FP64 instructions per update are left
// (24 where the coefficients are real).
//
// Measured, 25601 x 64, per step of the persistent launch: 147.0 us with the 54
// instructions, 100.2 with this coupling converted by the FP64 conversion
// instruction (which costs as much as a DFMA), 87.6 with the conversion in
// integers too; the FP64 pipe is then 84 % busy, the rest is latency of the
// integer chains with four warps per sub-partition.  25601 x 32: 73.2 -> 43.7,
// x 128: 287 -> 180 us.  More of the node in integers does not pay: with Pi + T
// rounded once there (26 FP64 instructions) 90.0, with B (m - p) + Phi too (22)
// 92.0 us: 37 integer instructions cost what a DFMA does.  All of the step in integers (8 FP64 instructions left)
// took 147 us: its 1235 integer instructions per update are then the bound.
//
// Numbers.  A value is an integer X, 2^59 <= |X| < 2^60, with its own exponent
// e: X 2^(e - 1082), exact.  A table entry is an integer Q with an exponent C
// shared by a class of entries of its row, Q 2^(C - 62), but for the theta
// neighbours' coefficients, which have their own (lower by their lift,
// tk_split_tables.cuh).  Multiplicands are taken as two 32-bit limbs,
// h 2^32 + l with l in [-2^31, 2^31); a sum keeps two 64-bit accumulators, of
// weight 2^64 (h h) and 2^32 (h l + l h).  These cannot overflow whatever the
// data: the integers of class F (F and the lifted K) add up to 2^62, those of G to
// 2^61, so that the first stays below 2^59 and the second below 3.5 2^61.
//
// Alignment.  Each product has the exponent of its value plus that of its entry;
// the values are shifted right to the largest of these, per row and component:
// what is lost lies 2^-60 below a product of the sum's largest exponent.  The
// sum, T = sum / 2^64, stands for T 2^(E - 1080) and is converted to FP64 once
// (split_value).  The l l products, zero in the mean, are left out.  That, and T's
// rounding to an integer, cost up to 2^-53 each of the largest product that the sum's
// exponents allow, typically 2^-56, and the conversion half a unit: an FMA chain
// rounds to 2^-53 of its partial sum at every product.  The row's own two coefficients
// share an exponent, so one that cancels to far less than the other keeps fewer bits
// (as many as its own rounding left it).
// Every operation treats both signs alike, so that conjugate
// data and a -> -a still give conjugate results to the bit.
//
// A team of K warps (NP = 32 K rows, one per lane) walks the columns together;
// the neighbouring rows' sums go through shared memory, with one barrier of the
// team per half node and per node.  One row per lane keeps the loop at 128
// registers, four warps per sub-partition, for every number of rows; with two
// rows per lane (three warps, 168 registers) the same arithmetic took 124 us.
// 20 warps (96 registers, spills): 120 us.
//
// Subnormal values and couplings are taken and rounded like any other (sums are not
// aligned below kSplitFloor, ten places under the smallest subnormal).  Columns
// with a Phi above 1e263, infinite or NaN, and columns whose
// tables are not finite or too large, take the FP64 instructions alone, so that
// such values propagate as IEEE arithmetic has them; Pi only ever meets FP64
// instructions (testing it too took 1 % more on 25601 x 64).
#pragma once

#include "tk_split_tables.cuh"
#include "tk_stencil.cuh"

namespace tk {
namespace {

// ---- integers ----

// Two components of a lane's row as integers: the magnitude, all its bits
// inverted where the value is negative (so that a right shift cuts both signs
// alike), the exponent field (1 for zeros and subnormals, whose magnitudes have no
// leading one), and 1 unless the value is zero.
struct SplitInts {
    long long x[2];
    int e[2];
    int j[2];
};

__device__ __forceinline__ int nonzero(int hi, int lo) { return (int)min((unsigned)(hi | lo), 1u); }

// Right shift, the sign filled in; n >= 64 gives 0 or -1.
__device__ __forceinline__ long long shr_s64(long long x, int n)
{
    long long r;
    asm("shr.s64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(n));
    return r;
}

// A magnitude with inverted bits where negative, n places to the right.  The
// bits cut off are replaced by a 1 in the last place (j = 1), which makes the
// result an ordinary odd integer, the same for both signs but for its sign,
// and unbiased.
__device__ __forceinline__ long long cut(long long x, int n, int j) { return shr_s64(x, n) | j; }

// That form of an ordinary integer.
__device__ __forceinline__ long long inverted(long long v) { return v + (v >> 63); }

// An ordinary integer shifted right, rounded towards zero.
__device__ __forceinline__ long long shr_zero(long long v, int n)
{
    const long long s = v >> 63;
    return shr_s64(v + s, n) - s;
}

__device__ __forceinline__ int2 limbs(long long x)
{
    return make_int2((int)(x >> 32) + (int)((unsigned)x >> 31), (int)x);
}

// Of components C0 and C0 + 1.
template <int C0>
__device__ __forceinline__ void split_ints(const double (&u)[4], SplitInts &o)
{
#pragma unroll
    for (int k = C0; k < C0 + 2; ++k) {
        const unsigned hi = (unsigned)__double2hiint(u[k]);
        const unsigned lo = (unsigned)__double2loint(u[k]);
        const int f = (int)((hi >> 20) & 0x7ffu), e = max(f, 1), j = nonzero((int)(hi & 0x7fffffffu), (int)lo);
        const unsigned m = (hi & 0xfffffu) + ((unsigned)min(f, 1) << 20);
        const unsigned s = (unsigned)((int)hi >> 31), mask = (unsigned)-j;
        const unsigned xh = (__funnelshift_l(lo, m, 7) ^ s) & mask, xl = ((lo << 7) ^ s) & mask;
        o.x[k - C0] = ((long long)(int)xh << 32) | xl;
        o.e[k - C0] = e;
        o.j[k - C0] = j;
    }
}

// The accumulators of a class's sum.
struct SplitSum {
    long long s2 = 0, s1 = 1ll << 31;
    __device__ __forceinline__ void add(int2 x, int2 q)
    {
        s2 += (long long)x.x * q.x;
        s1 += (long long)x.x * q.y;
        s1 += (long long)x.y * q.x;
    }
    // sum / 2^64, the lower accumulator rounded to the nearest (ties to even)
    __device__ __forceinline__ long long take() const
    {
        int r = (int)(s1 >> 32);
        if ((int)s1 == 0) r &= ~1;
        return s2 + r;
    }
};

// q, whose place 10 stands for 2^-1074, rounded to a subnormal number.
__device__ __forceinline__ double split_subnormal(unsigned long long q, unsigned sign)
{
    q += 0x1ffu + (((unsigned)q >> 10) & 1u);
    return __longlong_as_double((long long)((q >> 10) | ((unsigned long long)sign << 32)));
}

// T 2^(o - 1080) in FP64, rounded to the nearest (ties to even); o >= kSplitFloor.
// In integers: the conversion instruction holds the FP64 pipe as long as a DFMA
// does.  Where a pulse's tails underflow, whole columns take the branch: with a DFMA
// in it (a normal number times 2^-64) 16001 x 128 took 127 us a step instead of 118.
// ANY: the branch takes any o, which the forward step does not need, but whose
// schedule is the faster one there (25601 x 64 88.7 -> 87.6 us, 4999 x 45 20.5 -> 20.1;
// 8001 x 128 59.1 -> 59.5) and the slower one in the transposed step (147.0 -> 147.8).
template <bool ANY = false>
__device__ __forceinline__ double split_value(long long T, int o)
{
    const long long s = T >> 63;
    const unsigned long long m = (unsigned long long)((T ^ s) - s);   // < 2^62
    const unsigned mh = (unsigned)(m >> 32), ml = (unsigned)m;
    int n = __clz((int)mh);
    if (mh == 0) n = 32 + __clz((int)ml);
    unsigned long long q = m << (n - 1);             // the leading bit at place 62 (|T| < 2^62)
    q += 0x1ffu + (((unsigned)q >> 10) & 1u);        // 53 bits stay, a carry goes into the exponent
    const unsigned qh = (unsigned)(q >> 32), ql = (unsigned)q;
    const int e = o - n + 6;   // exponent field
    const unsigned lo = __funnelshift_r(ql, qh, 10);
    const unsigned hi = ((qh >> 10) + ((unsigned)(e - 1) << 20)) | ((unsigned)s & 0x80000000u);
    if (e > 0 || m == 0) return __hiloint2double(m != 0 ? (int)hi : 0, (int)lo);
    const int up = o - kSplitFloor;
    return split_subnormal(!ANY || up >= 0 ? m << up : (m >> min(-up, 63)) | 1u, (unsigned)s & 0x80000000u);
}

// ---- teams ----

// What a row's neighbours need of it, one record per row, in two buffers used
// in turn (a warp writes a buffer again only after a barrier that every reader
// of its last contents has passed).  Through shared memory also within a warp:
// twelve shuffles took longer.
struct SplitRows {
    int4 s[2][32];
    int2 x[2][32];
    __device__ __forceinline__ void put_exps(int b, int l, int2 e) { x[b][l] = e; }
    __device__ __forceinline__ int2 exps(int b, int l) const { return x[b][l]; }
};

// A warp's place in its team.
template <int K, class Rows = SplitRows>
struct SplitTeam {
    Rows *rows;        // the team's K
    int h;             // this warp's rows are 32 h ..
    int lane;
    int bar;           // the team's named barrier
    int buf = 0;

    // Whether p is true in any lane of the team; a barrier of the team.
    __device__ __forceinline__ bool any(bool p) const
    {
        if constexpr (K == 1) {
            __syncwarp();
            return __any_sync(kFull, p) != 0;
        } else {
            unsigned r;
            asm volatile(
                "{\n .reg .pred a, b;\n setp.ne.u32 a, %1, 0;\n barrier.cta.red.or.pred b, %2, %3, a;\n"
                " selp.u32 %0, 1, 0, b;\n}"
                : "=r"(r)
                : "r"((unsigned)p), "r"(bar), "n"(32 * K)
                : "memory");
            return r != 0;
        }
    }
    // Exchange the rows' records with a barrier of the team; whether p is true
    // in any of its lanes.  The rows beyond the first and the last are these
    // themselves (their coefficients are zero).
    __device__ __forceinline__ bool exchange(int4 s, int2 e, bool p, int4 &su, int2 &eu, int4 &sd, int2 &ed)
    {
        rows[h].s[buf][lane] = s;
        rows[h].put_exps(buf, lane, e);
        const bool r = any(p);
        const int row = 32 * h + lane;
        const int u = min(row + 1, 32 * K - 1), d = max(row - 1, 0);
        su = rows[u >> 5].s[buf][u & 31];
        eu = rows[u >> 5].exps(buf, u & 31);
        sd = rows[d >> 5].s[buf][d & 31];
        ed = rows[d >> 5].exps(buf, d & 31);
        buf ^= 1;
        return r;
    }
    // The neighbouring rows' values of two FP64 numbers (cold columns, samples).
    __device__ __forceinline__ void neighbours(double r, double i, double (&up)[2], double (&dn)[2])
    {
        int4 su, sd;
        int2 eu, ed;
        exchange(make_int4(__double2hiint(r), __double2loint(r), __double2hiint(i), __double2loint(i)),
                 make_int2(0, 0), false, su, eu, sd, ed);
        up[0] = __hiloint2double(su.x, su.y);
        up[1] = __hiloint2double(su.z, su.w);
        dn[0] = __hiloint2double(sd.x, sd.y);
        dn[1] = __hiloint2double(sd.z, sd.w);
    }
};

// One table (NODE: the node's, else the half node's) of a column's block, as
// one warp of the team holds it (kStepBytes).
template <bool NODE>
struct StepTab {
    static constexpr int kF64 = NODE ? kStepHalfF64 + kSplitEntries : 0;
    static constexpr int kInt = kF64 + (NODE ? kStepNodeF64 : kStepHalfF64);
    const unsigned char *p;
    int lane;
    __device__ __forceinline__ double f64(int q) const
    {
        return *reinterpret_cast<const double *>(p + ((kF64 + q) * 32 + lane) * 8);
    }
    __device__ __forceinline__ int2 entry(int q) const
    {
        return *reinterpret_cast<const int2 *>(p + ((kInt + q) * 32 + lane) * 8);
    }
    __device__ __forceinline__ int row_exp() const
    {
        return *reinterpret_cast<const int *>(p + kStepExps + (NODE ? 128 : 0) + lane * 4);
    }
    __device__ __forceinline__ int lifts() const
    {
        return *reinterpret_cast<const int *>(p + kStepExps + 256 + lane * 4);
    }
    __device__ __forceinline__ int2 head() const { return *reinterpret_cast<const int2 *>(p + kStepHead); }
};

// The coupling of Phi (values a left and c right of the point) to Pi_R and
// Pi_I, as integers T 2^(O - 1080).  False (the same in the whole team) where
// a value or the table (cold) calls for the FP64 instructions.
template <int K, bool NODE>
__device__ __forceinline__ bool split_coupling(const SplitInts &a, const SplitInts &c, const StepTab<NODE> &tab,
                                               bool cold, bool imag, SplitTeam<K> &team, long long (&T)[2],
                                               int (&O)[2])
{
    int e1[2], sh[2], sl[2];
#pragma unroll
    for (int g = 0; g < 2; ++g) {
        e1[g] = max(a.e[g], c.e[g]);
        const long long s = inverted(cut(a.x[g], e1[g] - a.e[g], a.j[g]) + cut(c.x[g], e1[g] - c.e[g], c.j[g]));
        sh[g] = (int)(s >> 32);
        sl[g] = (int)s;
    }
    int4 su, sd;
    int2 eu2, ed2;
    const bool over =
        team.exchange(make_int4(sh[0], sl[0], sh[1], sl[1]), make_int2(e1[0], e1[1]),
                      cold || max(e1[0], e1[1]) >= kSplitMaxExp, su, eu2, sd, ed2);
    if (over) return false;
    // exponents of the products over the F class's: the largest of each sum
    const int rx = tab.row_exp(), cf = (short)(rx & 0xffff), cg = (rx >> 16) - cf;
    const int lx = tab.lifts(), lu = (short)(lx & 0xffff), ld = lx >> 16;
    int f[2];
    f[0] = max(max(eu2.x - lu, ed2.x - ld), max(e1[0], kSplitFloor - cf));
    f[1] = max(max(eu2.y - lu, ed2.y - ld), max(e1[1], kSplitFloor - cf));
    if (imag) {
        f[0] = max(f[0], e1[1] + cg);
        f[1] = max(f[1], e1[0] + cg);
    }
#pragma unroll
    for (int g = 0; g < 2; ++g) {
        const int uh = g ? su.z : su.x, ul = g ? su.w : su.y, eu = g ? eu2.y : eu2.x;
        const int dh = g ? sd.z : sd.x, dl = g ? sd.w : sd.y, ed = g ? ed2.y : ed2.x;
        SplitSum s;
        s.add(limbs(cut(a.x[g], f[g] - a.e[g], a.j[g])), tab.entry(S_FA));
        s.add(limbs(cut(c.x[g], f[g] - c.e[g], c.j[g])), tab.entry(S_FC));
        s.add(limbs(cut(((long long)uh << 32) | (unsigned)ul, f[g] + lu - eu, nonzero(uh, ul))), tab.entry(S_KP));
        s.add(limbs(cut(((long long)dh << 32) | (unsigned)dl, f[g] + ld - ed, nonzero(dh, dl))), tab.entry(S_KM));
        if (imag) {   // the other part's, subtracted from the real part
            const int o = 1 - g, n = f[g] - cg;
            int2 la = limbs(cut(a.x[o], n - a.e[o], a.j[o])), lc = limbs(cut(c.x[o], n - c.e[o], c.j[o]));
            if (g == 0) {
                la = make_int2(-la.x, -la.y);
                lc = make_int2(-lc.x, -lc.y);
            }
            s.add(la, tab.entry(S_GA));
            s.add(lc, tab.entry(S_GC));
        }
        T[g] = s.take();
        O[g] = cf + f[g];
    }
    return true;
}

// ---- Eqs. (lw1) and (lw2) on a lane's row ----

struct Row4 {
    double v[4];
};

// With the FP64 instructions alone, from the unsplit tables (half_node and
// full_node's operations).
template <int NPR>
__device__ __noinline__ Row4 cold_half(Row4 a, Row4 c, double uR, double uI, double dR, double dI, const double *tab)
{
    const FmaK<double> k1 = fma_k<double>();
    double q[kNCH];
    for (int k = 0; k < kNCH; ++k) q[k] = tab[k * NPR];
    const double sPR = fma(a.v[2], k1.one, c.v[2]), sPI = fma(a.v[3], k1.one, c.v[3]);
    Row4 h;
    h.v[0] = fma(q[H_HQ], c.v[0], fma(q[H_HP], a.v[0], sPR));
    h.v[1] = fma(q[H_HQ], c.v[1], fma(q[H_HP], a.v[1], sPI));
    double x = fma(q[H_PAR], a.v[2], k1.nz);
    x = fma(q[H_PCR], c.v[2], x);
    x = fma(-q[H_PI], sPI, x);
    x = fma(q[H_FAR], a.v[0], x);
    x = fma(-q[H_FAI], a.v[1], x);
    x = fma(q[H_FCR], c.v[0], x);
    x = fma(-q[H_FCI], c.v[1], x);
    x = fma(q[H_KP], uR, x);
    h.v[2] = fma(q[H_KM], dR, x);
    double y = fma(q[H_PAR], a.v[3], k1.nz);
    y = fma(q[H_PCR], c.v[3], y);
    y = fma(q[H_PI], sPR, y);
    y = fma(q[H_FAR], a.v[1], y);
    y = fma(q[H_FAI], a.v[0], y);
    y = fma(q[H_FCR], c.v[1], y);
    y = fma(q[H_FCI], c.v[0], y);
    y = fma(q[H_KP], uI, y);
    h.v[3] = fma(q[H_KM], dI, y);
    return h;
}

template <int NPR>
__device__ __noinline__ Row4 cold_node(Row4 m, Row4 p, Row4 u, double uR, double uI, double dR, double dI,
                                       const double *tab, double e)
{
    const FmaK<double> k1 = fma_k<double>();
    double q[kNCN];
    for (int k = 0; k < kNCN; ++k) q[k] = tab[k * NPR];
    const double sPR = fma(p.v[2], k1.one, m.v[2]), sPI = fma(p.v[3], k1.one, m.v[3]);
    Row4 o;
    o.v[0] = fma(e, sPR, fma(q[N_B], m.v[0], fma(-q[N_B], p.v[0], u.v[0])));
    o.v[1] = fma(e, sPI, fma(q[N_B], m.v[1], fma(-q[N_B], p.v[1], u.v[1])));
    double x = fma(q[N_PPR], p.v[2], u.v[2]);
    x = fma(q[N_PMR], m.v[2], x);
    x = fma(-q[N_C2I], sPI, x);
    x = fma(q[N_FPR], p.v[0], x);
    x = fma(-q[N_FPI], p.v[1], x);
    x = fma(q[N_FMR], m.v[0], x);
    x = fma(-q[N_FMI], m.v[1], x);
    x = fma(q[N_KP], uR, x);
    o.v[2] = fma(q[N_KM], dR, x);
    double y = fma(q[N_PPR], p.v[3], u.v[3]);
    y = fma(q[N_PMR], m.v[3], y);
    y = fma(q[N_C2I], sPR, y);
    y = fma(q[N_FPR], p.v[1], y);
    y = fma(q[N_FPI], p.v[0], y);
    y = fma(q[N_FMR], m.v[1], y);
    y = fma(q[N_FMI], m.v[0], y);
    y = fma(q[N_KP], uI, y);
    o.v[3] = fma(q[N_KM], dI, y);
    return o;
}

__device__ __forceinline__ Row4 row4(const double (&x)[4]) { return {x[0], x[1], x[2], x[3]}; }

// Eq. (lw1) between columns a and c (half_node's result: Phi divided by e);
// half64: the lane's row of the unsplit table.
template <int K>
__device__ __forceinline__ void split_half_node(const double (&a)[4], const SplitInts &pa, const double (&c)[4],
                                                const SplitInts &pc, const unsigned char *block, SplitTeam<K> &team,
                                                const double *half64, const FmaK<double> &k1, double (&h)[4])
{
    const StepTab<false> tab{block, team.lane};
    const int2 head = tab.head();
    const bool imag = head.y != 0;
    const double sPR = fma(a[2], k1.one, c[2]);
    const double sPI = fma(a[3], k1.one, c[3]);
    const double HP = tab.f64(D_HP), HQ = tab.f64(D_HQ);
    h[0] = fma(HQ, c[0], fma(HP, a[0], sPR));
    h[1] = fma(HQ, c[1], fma(HP, a[1], sPI));
    long long T[2];
    int O[2];
    if (!split_coupling<K, false>(pa, pc, tab, head.x != 0, imag, team, T, O)) {
        double up[2], dn[2];
        team.neighbours(fma(a[0], k1.one, c[0]), fma(a[1], k1.one, c[1]), up, dn);
        const Row4 r = cold_half<32 * K>(row4(a), row4(c), up[0], up[1], dn[0], dn[1], half64);
#pragma unroll
        for (int k = 0; k < 4; ++k) h[k] = r.v[k];
        return;
    }
    const double PA = tab.f64(D_PAR), PC = tab.f64(D_PCR);
    double x = fma(PC, c[2], fma(PA, a[2], split_value<true>(T[0], O[0])));
    double y = fma(PC, c[3], fma(PA, a[3], split_value<true>(T[1], O[1])));
    if (imag) {
        const double PI = tab.f64(D_PI);
        x = fma(-PI, sPI, x);
        y = fma(PI, sPR, y);
    }
    h[2] = x;
    h[3] = y;
}

// Eq. (lw2) (full_node's result) from the half nodes left (m) and right (p).
template <int K>
__device__ __forceinline__ void split_full_node(const double (&m)[4], const SplitInts &pm, const double (&p)[4],
                                                const SplitInts &pp, const double (&u)[4], const unsigned char *block,
                                                SplitTeam<K> &team, const double *node64, double en,
                                                const FmaK<double> &k1, double (&out)[4])
{
    const StepTab<true> tab{block, team.lane};
    const int2 head = tab.head();
    const bool imag = head.y != 0;
    const double B = tab.f64(D_B), PP = tab.f64(D_PPR), PM = tab.f64(D_PMR);
    const double sPR = fma(p[2], k1.one, m[2]);
    const double sPI = fma(p[3], k1.one, m[3]);
    out[0] = fma(en, sPR, fma(B, m[0], fma(-B, p[0], u[0])));
    out[1] = fma(en, sPI, fma(B, m[1], fma(-B, p[1], u[1])));
    double x = fma(PM, m[2], fma(PP, p[2], u[2]));
    double y = fma(PM, m[3], fma(PP, p[3], u[3]));
    if (imag) {
        const double CI = tab.f64(D_C2I);
        x = fma(-CI, sPI, x);
        y = fma(CI, sPR, y);
    }
    long long T[2];
    int O[2];
    if (!split_coupling<K, true>(pm, pp, tab, head.x != 0, imag, team, T, O)) {
        double up[2], dn[2];
        team.neighbours(fma(p[0], k1.one, m[0]), fma(p[1], k1.one, m[1]), up, dn);
        const Row4 r = cold_node<32 * K>(row4(m), row4(p), row4(u), up[0], up[1], dn[0], dn[1], node64, en);
#pragma unroll
        for (int k = 0; k < 4; ++k) out[k] = r.v[k];
        return;
    }
    out[2] = fma(split_value<true>(T[0], O[0]), k1.one, x);
    out[3] = fma(split_value<true>(T[1], O[1]), k1.one, y);
}

// ---- the sweep of one step over a team's columns ----

// Work split: block b owns columns [b Nr / B, (b+1) Nr / B).  The K warps of a
// team run on K sub-partitions of the SM; the block's columns are cut evenly
// over the 4 / K groups of sub-partitions, and each group's share over its
// teams.
template <int W, int K>
__device__ __forceinline__ void team_range(int Nr, int team, int *i0, int *i1)
{
    constexpr int P = 4 / K, G = W / 4;
    const long long B = gridDim.x, b = blockIdx.x;
    const int b0 = (int)((b * Nr) / B), C = (int)(((b + 1) * Nr) / B) - b0;
    int start = b0, cnt = 0;
    for (int w = 0; w <= team; ++w) {
        const int p = w % P, q = w / P;
        const int cp = ((p + 1) * C) / P - (p * C) / P;
        start += cnt;
        cnt = ((q + 1) * cp) / G - (q * cp) / G;
    }
    *i0 = start;
    *i1 = start + cnt;
}

// Per warp in shared memory: the tables of the column being formed and of the
// next one, filled by one bulk copy per column, issued a column ahead.
struct SplitRing {
    alignas(16) unsigned char tab[2][kStepBytes];
};

// The copies' progress, across sweeps: the slot of the next copy to wait for,
// per slot the parity of the next wait and of the copies issued, and whether a wait
// of this lane gave up.
struct SplitRingState {
    unsigned cur = 0, wait = 0, issue = 0;
};
constexpr unsigned kLost = 4;   // in wait

__device__ __forceinline__ void split_ring_init(unsigned long long *bar, int lane)
{
    if (lane == 0) {
        mbar_init(&bar[0]);
        mbar_init(&bar[1]);
        mbar_init_fence();
    }
    __syncwarp();
}

// What a sweep rarely needs: the unsplit tables, for the FP64 instructions alone,
// the word that is raised when a wait for a copy gives up, and (one lane, once a
// column) the bytes from a column's blocks to the next's: 0 where one cold block
// stands for all of them.
struct SweepRare {
    const double *h, *n;
    int *e;
    size_t p;
    __device__ __forceinline__ const double *half() const { return h; }
    __device__ __forceinline__ const double *node() const { return n; }
    __device__ __forceinline__ int *err() const { return e; }
    __device__ __forceinline__ size_t pitch() const { return p; }
};

template <int K, class Rare = SweepRare>
struct SplitSweep {
    SplitRing *ring;
    unsigned long long *bar;   // the warp's two mbarriers, in shared memory (split_ring_init)
    const unsigned char *tab;  // the warp's block of column 0
    Rare rare;
    int Nr;
    double en;

    // Copy column i's block into a slot; the warp has used its last contents.
    __device__ __forceinline__ void fetch(SplitRingState &st, int slot, int i, int lane) const
    {
        __syncwarp();
        if (lane == 0 && !(st.wait & kLost)) {
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            mbar_expect(&bar[slot], kStepBytes);
            bulk_fetch(ring->tab[slot], tab + (size_t)i * rare.pitch(), kStepBytes, &bar[slot]);
        }
        st.issue ^= 1u << slot;
    }
    // After a wait that gave up, a lane waits no more, and no copy is started by
    // lane 0 (the results are then not valid; everything else goes on, so that the
    // team's barriers hold).  Each lane for itself: with a vote of the warp the batch
    // of 128-row members takes 84 us a tick instead of 80.
    __device__ __forceinline__ void await(SplitRingState &st, int slot) const
    {
        const unsigned parity = (st.wait >> slot) & 1u;
        if (!mbar_test(&bar[slot], parity)) {
            if (!(st.wait & kLost) && !mbar_wait(&bar[slot], parity, rare.err())) {
                st.wait |= kLost;
                atomicExch(rare.err(), 1);
            }
            if (st.wait & kLost) return;
        }
        st.wait ^= 1u << slot;
    }
    // Wait (with a limit) for the copies still in flight before the block exits.
    __device__ __forceinline__ void drain(SplitRingState &st) const
    {
        for (int s = 0; s < 2; ++s)
            if (((st.wait ^ st.issue) >> s) & 1u) mbar_wait(&bar[s], (st.wait >> s) & 1u);
    }

    // Columns [i0, i1) of one step.  The half node left of i0 is formed here
    // too (handing it over between teams would cost a second wait and a second
    // order of the loop; it is one of 21 on the flagship grid).
    // before_right() is called before the column i1 is first read; again: a
    // sweep over the same columns follows.
    template <typename Right, typename Store>
    __device__ __forceinline__ void run(SplitRingState &st, SplitTeam<K> &team, const double *__restrict__ u_in,
                                        int i0, int i1, bool again, Right before_right, Store store) const
    {
        constexpr int NP = 32 * K;
        const int row = 32 * team.h + team.lane;
        const FmaK<double> k1 = fma_k<double>();
        const int ib = i0 > 0 ? i0 - 1 : 0;
        const int ie = i1 < Nr - 1 ? i1 : Nr - 1;   // columns with tables: [ib, ie)
        if (((st.wait ^ st.issue) >> st.cur) & 1u) {
        } else if (ib < ie) {
            fetch(st, st.cur, ib, team.lane);
        }
        const double *pu = u_in + (size_t)ib * (4 * NP) + row;
        auto load = [&](const double *p, double (&u)[4]) {
#pragma unroll
            for (int k = 0; k < 4; ++k) u[k] = __ldcg(p + k * NP);
        };
        double a[4], hm[4], un[4];
        SplitInts pa, pm;
#pragma unroll
        for (int k = 0; k < 4; ++k) hm[k] = 0.0;
        split_ints<0>(hm, pm);
        load(pu, a);
        if (ib + 1 == i1) before_right();
        pu += 4 * NP;
        if (ib + 1 < Nr) load(pu, un);
        split_ints<0>(a, pa);
#pragma unroll 1
        for (int i = ib; i < i1; ++i) {
            double o[4];
            if (i + 1 < Nr) {
                double c[4], hp[4];
                SplitInts pc, pp;
                const int nx = i + 1 < ie ? i + 1 : again ? ib : -1;
                if (nx >= 0) fetch(st, st.cur ^ 1, nx, team.lane);
#pragma unroll
                for (int k = 0; k < 4; ++k) c[k] = un[k];
                if (i + 1 < i1) {
                    if (i + 2 == i1) before_right();
                    pu += 4 * NP;
                    if (i + 2 < Nr) load(pu, un);
                }
                split_ints<0>(c, pc);
                await(st, st.cur);
                const unsigned char *block = ring->tab[st.cur];
                st.cur ^= 1;
                split_half_node<K>(a, pa, c, pc, block, team, rare.half() + (size_t)i * (kNCH * NP) + row, k1,
                                   hp);
                split_ints<0>(hp, pp);
                if (i >= i0) {
                    if (i > 0) {
                        split_full_node<K>(hm, pm, hp, pp, a, block, team,
                                           rare.node() + (size_t)i * (kNCN * NP) + row, en, k1, o);
                    } else {
#pragma unroll
                        for (int k = 0; k < 4; ++k) o[k] = 0.0;
                    }
                    store(i, o);
                }
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    a[k] = c[k];
                    hm[k] = hp[k];
                }
                pa = pc;
                pm = pp;
            } else {   // the right edge of the grid
#pragma unroll
                for (int k = 0; k < 4; ++k) o[k] = 0.0;
                store(i, o);
            }
        }
    }
};

// Every observer slot at column i: observe()'s samples from one row per lane.
template <int K>
__device__ __forceinline__ void observe_team(int i, const double (&o)[4], SplitTeam<K> &team, const ObsDev &obs,
                                             double *wave, int64_t cap, const long long *sample_ctr,
                                             const double *w_row, int sample_offset)
{
    for (int k = 0; k < obs.n; ++k) {
        const int slot = (i == obs.i0[k]) ? 0 : ((i == obs.i0[k] + 1) ? 1 : -1);
        if (slot < 0) continue;
        const int j0 = obs.j0[k], l0 = j0 - 32 * team.h;
        double up[2], dn[2];   // row j0 + 1 may be another warp's
        team.neighbours(o[0], o[1], up, dn);
        if (l0 == team.lane) {
            const long long sample = *(volatile const long long *)sample_ctr + sample_offset;
            double *dst = wave + ((size_t)k * cap + sample) * 4 + 2 * slot;
            const double w0 = (1.0 - obs.ft[k]) * w_row[j0];
            const double w1 = obs.ft[k] * w_row[j0 + 1];
            const double cr = w0 * o[0] + w1 * up[0];
            const double ci = w0 * o[1] + w1 * up[1];
            const double wr = slot ? obs.wr1[k] : obs.wr0[k];
            dst[0] = wr * cr;
            dst[1] = wr * ci;
        }
    }
}

}  // namespace
}  // namespace tk
