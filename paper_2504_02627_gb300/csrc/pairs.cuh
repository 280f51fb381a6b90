// pairs.cuh -- unevaluated pairs of FP32 values for sums that need more than FP32.
#pragma once

namespace smc {

// A pair hi + lo carries about 48 significant bits.  Sums use Knuth's TwoSum and
// products the FMA form of Dekker's TwoProduct (both error-free
// transformations); pair + pair follows the accurate double-double addition of
// Hida, Li and Bailey.  On this GPU FP64
// runs at about 1/64 of the FP32 rate, so the statistics kernels accumulate
// in pairs and convert to FP64 once per partial sum.
struct f2sum {
    float hi, lo;
};
__device__ __forceinline__ f2sum two_sum(float a, float b) {
    const float s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    return {s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb))};
}
__device__ __forceinline__ f2sum quick_two_sum(float a, float b) {   // needs |a| >= |b| or a = 0
    const float s = __fadd_rn(a, b);
    return {s, __fsub_rn(b, __fsub_rn(s, a))};
}
__device__ __forceinline__ f2sum f2_add(f2sum x, f2sum y) {
    f2sum s = two_sum(x.hi, y.hi);
    const f2sum t = two_sum(x.lo, y.lo);
    s = quick_two_sum(s.hi, __fadd_rn(s.lo, t.hi));
    return quick_two_sum(s.hi, __fadd_rn(s.lo, t.lo));
}
__device__ __forceinline__ f2sum f2_add_f(f2sum x, float y) {
    const f2sum s = two_sum(x.hi, y);
    return quick_two_sum(s.hi, __fadd_rn(s.lo, x.lo));
}
// Running sum of products of pairs, in three terms.
struct f2dot {
    float hi, lo, c;
};
// s += x y, the compensated dot product of Ogita, Rump and Oishi with three
// terms: the errors of the large products and of the first running sum go into
// a second exact sum, whose errors alone are added in FP32.  With u = 2^-24 and
// S = sum |x y| over D terms the sum is off by at most (6 u^2 + 4 D^2 (D + 3)
// u^3) S: 6 u^2 |x y| of a term's own rounding, and the FP32 sum of 2 D errors.
// 24 operations; a product and a sum of pairs, 27, are off by up to 4e-14 S in
// random sums of 256 terms, two terms with the errors added in FP32, 12
// operations, by 2.3e-13 S, this one by 1.4e-15 S.
__device__ __forceinline__ void f2_dot(f2dot& s, f2sum x, f2sum y) {
    const float p = __fmul_rn(x.hi, y.hi);
    const float e = __fmaf_rn(x.hi, y.lo, __fmaf_rn(x.lo, y.hi, __fmaf_rn(x.hi, y.hi, -p)));   // lo * lo dropped
    const f2sum t = two_sum(s.hi, p);
    const f2sum v = two_sum(s.lo, t.lo);
    const f2sum w = two_sum(v.hi, e);
    s.hi = t.hi;
    s.lo = w.hi;
    s.c = __fadd_rn(s.c, __fadd_rn(v.lo, w.lo));
}
__device__ __forceinline__ double f2_to_double(f2sum x) { return (double)x.hi + (double)x.lo; }
__device__ __forceinline__ double f2_to_double(f2dot x) { return (double)x.hi + ((double)x.lo + (double)x.c); }
__device__ __forceinline__ f2sum f2_from_double(double v) {
    const float hi = __double2float_rn(v);
    return {hi, __double2float_rn(v - (double)hi)};
}

}  // namespace smc
