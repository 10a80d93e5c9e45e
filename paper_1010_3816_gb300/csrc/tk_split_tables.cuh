// tk_split_tables.cuh -- table entries as the integers of tk_split.cuh.
//
// A row's entries form two classes, F (the row's own coefficients and its theta
// neighbours' KU, KD) and G (those of the other part), each with an exponent, so
// that the class's entries add up to less than 2^C.  The neighbours' coefficients
// may be far smaller than the row's own and their values larger by as much (the
// transposed step next to a pole, or any step next to the horizon): with one
// exponent for both, the integers would keep few bits of the product that
// decides.  So KU and KD are lifted by powers of two until they are about half as
// large as the largest term of the class, and the values they meet are taken that
// much lower: every product then keeps its bits against the largest one.
#pragma once

#include <math.h>

#include "tk_internal.h"

namespace tk {
namespace {

// v < 2^result for v >= 0, kSplitAbsent for 0; beyond every limit where v is not
// finite.
__device__ int split_exponent(double v)
{
    if (v == 0.0) return kSplitAbsent;
    const int e = (__double2hiint(v) >> 20) & 0x7ff;
    return e != 0 ? e - 1022 : -1010 - __clzll(__double_as_longlong(v));
}

// The magnitudes of a table's class F: the own coefficients' sum, and each
// neighbour's coefficient times the number of values it multiplies.
struct RowTerms {
    double f, ku, kd;
    __device__ int top() const
    {
        return max(split_exponent(f), max(split_exponent(ku), split_exponent(kd)));
    }
    __device__ static int lift(double k, int top)
    {
        return k == 0.0 ? kLiftAbsent : max(0, top - 1 - split_exponent(k));
    }
};

// The lifts that two tables of a row share, the smaller of each table's (they
// differ by little: both go with the same angular factors); cold where they do
// not.
struct RowLifts {
    int u, d;
    __device__ static int common(int a, int b, int *cold)
    {
        if (a != kLiftAbsent && b != kLiftAbsent && abs(a - b) > kLiftSpread) *cold = 1;
        return min(a, b);
    }
    __device__ RowLifts(const RowTerms &a, const RowTerms &b, int *cold)
    {
        const int ta = a.top(), tb = b.top();
        u = common(RowTerms::lift(a.ku, ta), RowTerms::lift(b.ku, tb), cold);
        d = common(RowTerms::lift(a.kd, ta), RowTerms::lift(b.kd, tb), cold);
    }
    __device__ int packed() const { return (u & 0xffff) | (d << 16); }
};

// The class exponents, F in the low half, G (with the sum g; twice the entries'
// sum, for the room that both classes need in one accumulator) in the high half.
// Sets *cold for tables that are not finite or too large for the split form.
struct RowExps {
    int f, g;
    __device__ RowExps(const RowTerms &t, const RowLifts &l, double gsum, int *cold)
    {
        const int top = t.top();
        g = split_exponent(gsum);
        if (top > kSplitMaxClass || g > kSplitMaxClass) {
            *cold = 1;
            f = g = 0;
            return;
        }
        // a lifted term is below 2^(top - 1) (assembled from bits: a product costs
        // the FP64 pipe 64 cycles)
        const double bound = __hiloint2double(max(top + 1022, 1) << 20, 0);
        auto lifted = [&](double k, int n) { return n == 0 || k == 0.0 ? k : bound; };
        f = split_exponent(t.f + (lifted(t.ku, l.u) + lifted(t.kd, l.d)));
        if (g != kSplitAbsent) ++g;
    }
    __device__ int packed() const { return (f & 0xffff) | (g << 16); }
};

// c 2^(62 - C) rounded to the nearest integer, as limbs; |c| < 2^C.
__device__ int2 split_entry(double c, int C)
{
    const long long b = __double_as_longlong(c);
    int e = (int)((b >> 52) & 0x7ff);
    long long v = b & 0xfffffffffffffll;
    if (e != 0) v |= 1ll << 52;
    else e = 1;
    if (v == 0) return make_int2(0, 0);
    const int up = e - 1075 + 62 - C;    // |c| < 2^C: v stays below 2^62
    if (up >= 0) v <<= up;
    else v = up < -54 ? 0 : (v + (1ll << (-up - 1))) >> -up;
    v |= 1;   // odd, so that the limbs of -c are those of c with the other sign
    if (b < 0) v = -v;
    const int l = (int)v;
    return make_int2((int)((v - l) >> 32), l);
}

}  // namespace
}  // namespace tk
