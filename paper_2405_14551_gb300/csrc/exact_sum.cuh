// Sums of FP32 values with more than FP64's precision in FP32 operations.
#pragma once

namespace lbcg {

// A sum of FP32 values held exactly to 72 bits as three FP32 terms (error-free
// transformation of a sum: Knuth's two-sum), more than the 53 bits of an FP64
// accumulator.  An SM of this GPU does 2 FP64 and 128 FP32 additions a clock, so
// the 13 additions here cost a fifth of one FP64 addition.  A sum that is not
// finite keeps its leading term's value (value()).
struct Sum3 {
  float h = 0.f, m = 0.f, l = 0.f;
  __device__ __forceinline__ static void two(float& a, float& b) {  // a + b = a' + b' exactly
    const float s = __fadd_rn(a, b), t = __fadd_rn(s, -a);
    b = __fadd_rn(__fadd_rn(a, -__fadd_rn(s, -t)), __fadd_rn(b, -t));
    a = s;
  }
  __device__ __forceinline__ void add(float x) {
    two(h, x);
    two(m, x);
    l = __fadd_rn(l, x);
  }
  __device__ __forceinline__ void add_product(float a, float b) {  // a b = p + e exactly
    const float p = __fmul_rn(a, b);
    add(p);
    add(__fmaf_rn(a, b, -p));
  }
  __device__ __forceinline__ bool finite() const { return isfinite(h); }
  __device__ __forceinline__ double value() const { return (double)h + ((double)m + (double)l); }
};
// Squares are formed from values scaled by 2^40, so that the square of a value
// near the FP32 round-off of a quantity of order one keeps its bits.
constexpr float SQUARE_SCALE = 1099511627776.0f;  // 2^40
constexpr double SQUARE_UNSCALE = 1.0 / ((double)SQUARE_SCALE * (double)SQUARE_SCALE);

}  // namespace lbcg
