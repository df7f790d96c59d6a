// Sums of FP32 values with more than FP64's precision in FP32 operations.
#pragma once

namespace lbcg {

// A sum of FP32 values as three FP32 terms: two error-free levels (Knuth's
// two-sum) and a third that collects what the second rounds off, itself rounded.
// Over n values of absolute sum S the third stays below about 2 n 2^-48 S, so its
// roundings lose at most 2 n^2 2^-72 S: less than the n 2^-53 S of an FP64
// accumulator for up to 2^18 values.  A product enters with its rounding error
// (one FMA gives it), so a term is not rounded at all.  An SM of this GPU does 2
// FP64 and 128 FP32 additions a clock: the 13 additions of add() cost a fifth of
// one FP64 addition.  Values whose terms may leave FP32's range are the
// caller's to sum again in FP64: finite() is false after an overflow, and a term
// below about 2^-100 may have lost its low part (nearly_zero()).
struct Sum3 {
  float h = 0.f, m = 0.f, l = 0.f;
  __device__ __forceinline__ static void two(float& a, float& b) {  // a + b = a' + b' exactly
    const float s = __fadd_rn(a, b), t = __fadd_rn(s, -a);
    b = __fadd_rn(__fadd_rn(a, -__fadd_rn(s, -t)), __fadd_rn(b, -t));
    a = s;
  }
  __device__ __forceinline__ void add(float x) {
    two(h, x);
    add_low(x);
  }
  // a value at most about 2^-24 of the terms given to add()
  __device__ __forceinline__ void add_low(float x) {
    two(m, x);
    l = __fadd_rn(l, x);
  }
  // (a + a_low) b, where a_low is the rounding error of a
  __device__ __forceinline__ void add_product(float a, float a_low, float b) {
    const float p = __fmul_rn(a, b), q = __fmul_rn(a_low, b);
    add(p);
    add_low(__fmaf_rn(a, b, -p));
    add_low(q);
    l = __fadd_rn(l, __fmaf_rn(a_low, b, -q));
  }
  __device__ __forceinline__ bool finite() const { return isfinite(h); }
  // the sum of squares is too small for the low parts of its terms to be in range
  __device__ __forceinline__ bool nearly_zero() const { return fabsf(h) < 1e-6f; }
  __device__ __forceinline__ double value() const { return (double)h + ((double)m + (double)l); }
  // n plus the sum, also where the two cancel
  __device__ __forceinline__ double plus(int n) const { return ((double)n + (double)h) + ((double)m + (double)l); }
};
// Squares are formed from values scaled by 2^40, so that the square of a value
// near the FP32 round-off of a quantity of order one keeps its bits.
constexpr float SQUARE_SCALE = 1099511627776.0f;  // 2^40
constexpr double SQUARE_UNSCALE = 1.0 / ((double)SQUARE_SCALE * (double)SQUARE_SCALE);

}  // namespace lbcg
