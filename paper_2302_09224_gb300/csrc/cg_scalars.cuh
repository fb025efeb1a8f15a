// cg_scalars.cuh -- the CG recurrence's scalar steps from FP32-pair sums with
// the results of FP64 arithmetic on them.
//
// Every block of a resident launch takes alpha, beta and the decision to stop
// itself, and an FP64 division or conversion there stands in the way of all of
// them (cg_block.cuh).  Pairs carry some 45 bits, and what leaves is an FP32 step or
// a comparison, so they decide wherever their error cannot change it; next to a
// tie, or outside the range where the error bound holds, FP64 does.  Microseconds
// an iteration with the pairs alone and with this (reliable updates included):
// 20-bit 8^4 10.74 and 10.77, 16^4 17.62 and 17.73, 16^3x64 41.1 and 41.3; 16-bit
// 8^4 10.63 and 10.77.  The functions run on the host too, where their bounds are
// checked.
#pragma once

#include "ff.cuh"

namespace hisq {

// The FP64 forms, out of line: written in place they would be evaluated always
// and then selected.
__host__ __device__ __noinline__ inline float quotient_f64(double num, double den) { return (float)(num / den); }
__host__ __device__ __noinline__ inline bool less_f64(double x, double y) { return x < y; }

// (float)(num / den) for num = a - b (b zero: a alone) and den, each a pair; the
// doubles they stand for, of which the pairs are the leading 48 bits or all of
// them, come from exact(), called only where FP64 decides: exact(n, d) sets
// numerator and denominator.
//
// Error of q = num / den relative to itself: 2^-48 from each operand's own
// truncation, 2^-46 (|a| + |b|) from the difference, 2^-44 from the division
// (product, difference and second digit of 2^-46 each), under 2^-41 together
// while the difference keeps a sixteenth of its operands; FP64's own roundings
// add 2^-52.  The window of 2^-40 covers it.  Magnitudes are kept where every
// error term of the pairs is normal in FP32 or below 2^-45 of the quotient.
template <typename F>
__host__ __device__ __forceinline__ float step_quotient(ff a, ff b, ff den, F exact)
{
    const ff num = a - b;
    const ff q = num / den;
    const float an = fabsf(num.hi), ad = fabsf(den.hi), aq = fabsf(q.hi), w = rn_mul(aq, 0x1p-40f);
    const bool sure = an >= 0x1p-80f && an <= 0x1p80f && ad >= 0x1p-80f && ad <= 0x1p80f && aq >= 0x1p-90f &&
                      aq <= 0x1p90f && an >= rn_mul(rn_add(fabsf(a.hi), fabsf(b.hi)), 0.0625f) &&
                      rn_add(q.hi, rn_add(q.lo, w)) == q.hi && rn_add(q.hi, rn_sub(q.lo, w)) == q.hi;
    if (sure) return q.hi;
    double n, d;
    exact(n, d);
    return quotient_f64(n, d);
}

// x < y for two doubles given to within 2^-20 of themselves by x and y (leading
// parts of pairs); exact(u, v) sets the doubles where the difference is too small
// to tell, or either is not a normal number well inside FP32's range.
template <typename F>
__host__ __device__ __forceinline__ bool decide_less(float x, float y, F exact)
{
    const float m = fmaxf(fabsf(x), fabsf(y));
    if (m >= 0x1p-90f && m <= 0x1p100f && fabsf(rn_sub(x, y)) > rn_mul(m, 0x1p-18f)) return x < y;
    double u, v;
    exact(u, v);
    return less_f64(u, v);
}

}  // namespace hisq
