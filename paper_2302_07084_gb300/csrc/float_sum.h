// Sums of FP32 terms to FP64's accuracy in FP32 operations, for sums whose FP64
// additions would bound a kernel (1/64 of the FP32 rate on this GPU). Plain C++ for
// the host as well: compile there without contraction of a product and a sum.
#pragma once

#ifdef __CUDACC__
#define LNE_FSUM_FN __host__ __device__ __forceinline__
#else
#define LNE_FSUM_FN inline
#endif

namespace lne {

// a + b rounded, and err, its exact rounding error (two-sum, six operations).
LNE_FSUM_FN float two_sum(float a, float b, float *err) {
#ifdef __CUDA_ARCH__
    const float s = __fadd_rn(a, b), t = __fsub_rn(s, a);
    *err = __fadd_rn(__fsub_rn(a, __fsub_rn(s, t)), __fsub_rn(b, t));
#else
    const float s = a + b, t = s - a;
    *err = (a - (s - t)) + (b - t);
#endif
    return s;
}

// A running sum in three floats, hi + lo + tail: hi takes the rounded sum, lo the sum
// of hi's rounding errors, tail the sum of lo's. Off by n^3 / 6 2^-72 of the sum of n
// terms' sizes at most (and the value's own rounding), where n FP64 additions may be off
// by n 2^-53 of it: no worse up to 1,773 terms at their worst.
struct FloatSum {
    float hi, lo, tail;
};

LNE_FSUM_FN void float_sum_add(FloatSum &s, float p) {
    float e, e2;
    s.hi = two_sum(s.hi, p, &e);
    s.lo = two_sum(s.lo, e, &e2);
#ifdef __CUDA_ARCH__
    s.tail = __fadd_rn(s.tail, e2);
#else
    s.tail = s.tail + e2;
#endif
}

// The sum in FP64 (hi + lo is exact there unless lo is below 2^-29 of hi's last place).
LNE_FSUM_FN double float_sum_value(const FloatSum &s) { return (double)s.hi + ((double)s.lo + (double)s.tail); }

}  // namespace lne
