// tk_split_tables.cuh -- table entries as the integers of tk_split.cuh.
#pragma once

#include <math.h>

#include "tk_internal.h"

namespace tk {
namespace {

// The exponent of a class sum s: s < 2^result, kSplitAbsent for 0; sets *cold
// for a sum that is not finite or too large for the split form.
__device__ int class_exponent(double s, int *cold)
{
    if (s == 0.0) return kSplitAbsent;
    const int e = ((__double2hiint(s) >> 20) & 0x7ff) - 1022;
    if (!(e <= kSplitMaxClass)) {
        *cold = 1;
        return kSplitMaxClass;
    }
    return e;
}

// c 2^(62 - C) rounded to the nearest integer, as limbs; |c| < 2^C.
__device__ int2 split_entry(double c, int C)
{
    const long long b = __double_as_longlong(c);
    const int e = (int)((b >> 52) & 0x7ff);
    if (e == 0) return make_int2(0, 0);
    long long v = (b & 0xfffffffffffffll) | (1ll << 52);
    const int up = e - 1075 + 62 - C;    // <= 9
    if (up >= 0) v <<= up;
    else v = up < -54 ? 0 : (v + (1ll << (-up - 1))) >> -up;
    v |= 1;   // odd, so that the limbs of -c are those of c with the other sign
    if (b < 0) v = -v;
    const int l = (int)v;
    return make_int2((int)((v - l) >> 32), l);
}

}  // namespace
}  // namespace tk
