// Several quotients by one denominator.
#pragma once

namespace bmg {

// w / den for several w: q = w r with r = 1 / den rounded, corrected by the
// exact remainder, which gives the rounded quotient (Markstein, "Computation
// of elementary functions on the IBM RISC System/6000 processor", 1990),
// inside the range where no product over- or underflows (judged by the high
// words, in integers: an FP64 comparison takes a slot of the pipe that bounds
// the setup kernels).  Outside it the division itself.
static __device__ __noinline__ double rare_divide(double a, double b) { return a / b; }

struct Denominator {
  double den, r;
  int hd;        // high word of den (its sign and exponent)
  bool rare;
};

__device__ __forceinline__ Denominator denominator(double d) {
  const int hd = __double2hiint(d);
  return Denominator{d, __drcp_rn(d), hd, hd < (200 << 20) || hd > (1800 << 20)};
}

__device__ __forceinline__ double divide(double w, const Denominator& d) {
  const int hw = __double2hiint(w) & 0x7FFFFFFF;
  const bool zero = (hw | __double2loint(w)) == 0;
  if (d.rare || (!zero && (hw < d.hd - (100 << 20) || hw > d.hd + (100 << 20)))) return rare_divide(w, d.den);
  const double q = w * d.r;
  return fma(fma(-q, d.den, w), d.r, q);
}

// FP32 quotients are not what bounds a kernel here.
struct DenominatorF {
  float den;
};
__device__ __forceinline__ DenominatorF denominator(float d) { return DenominatorF{d}; }
__device__ __forceinline__ float divide(float w, const DenominatorF& d) { return w / d.den; }

// Sign bit set, and a number below zero (not -0, not NaN), without an FP64
// comparison.
__device__ __forceinline__ bool sign_bit(double v) { return __double2hiint(v) < 0; }
__device__ __forceinline__ bool sign_bit(float v) { return __float_as_int(v) < 0; }
__device__ __forceinline__ bool below_zero(double v) {
  const unsigned u = unsigned(__double2hiint(v));
  return u - 0x80000000u <= 0x7FF00000u && ((u << 1) | unsigned(__double2loint(v))) != 0;
}
__device__ __forceinline__ bool below_zero(float v) { return v < 0.0f; }

}  // namespace bmg
