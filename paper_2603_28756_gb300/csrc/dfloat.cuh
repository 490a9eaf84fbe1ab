// Double-word FP32 arithmetic for the setup transforms of R*g.
//
// A value is hi + lo, two FP32 numbers, |lo| <= ulp(hi) / 2 once settled: a 48-bit significand, so each
// operation is accurate to about 2^-44 of its operands' magnitude (FP64 carries 2^-53).  The
// transforms that use it (the NUFFT adjoint of Eq. 4: the sparse gather onto the spreading grid,
// the 2D grid FFT, the deconvolution) then run on the FP32 pipe, whose rate on GB300 is
// sixty-four times the FP64 pipe's; their result is stored in FP32.  At the image corners the
// deconvolution amplifies by 4e5 (1.25x grid), and 4e5 * 2^-44 is half of FP32's 2^-24, so the bound alone
// leaves no margin there; measured against 64 bits, the corners' largest error is 1.2e-7 of the image's rms
// (64^2 to 2560^2, 30 to 1000 angles), which is the spreading kernel's own error: it was the same with
// every operation renormalised and the deconvolution in FP64.
//
// The building blocks are the error-free transformations of floating-point arithmetic: Knuth's
// TwoSum (the exact rounding error of a sum) and the FMA-based TwoProduct (the exact rounding error
// of a product, fma(a, b, -ab)).  A sum adds the high parts by TwoSum and the low parts and the error
// in FP32; a product keeps hi * hi exactly and adds the two cross products to its error.  Neither
// renormalises the pair (three operations each).  The low part then stays within a few units in the last
// place of the largest operand since settle() last renormalised (once per butterfly, once per row of
// the gather), and its own rounding within 2^-46 of that operand; it is not bounded by the high part,
// which a cancellation can make as small as it likes.  So the errors are bounded relative to the
// operands' magnitudes, not to the result's, which is the bound an FFT or a dot product needs (their
// errors are judged against the input's norm): R*g's error is 2.6e-8 to 2.7e-8 of its norm, of which FP32
// storage alone makes 2.5e-8 to 2.6e-8.  Every step uses the _rn
// intrinsics, which the compiler never contracts into FMAs, so the transformations stay error-free.
#pragma once
#include <cuda_runtime.h>

namespace tmbir {

struct df {
  float hi, lo;
  df() = default;
  __host__ __device__ constexpr df(float h, float l) : hi(h), lo(l) {}
  // the double-word nearest to d: d rounded to FP32, then the remainder rounded to FP32
  __host__ __device__ constexpr df(double d) : hi((float)d), lo((float)(d - (double)(float)d)) {}
  __host__ __device__ constexpr df(float f) : hi(f), lo(0.f) {}
  __host__ __device__ constexpr df(int i) : df((double)i) {}
  __host__ __device__ explicit operator double() const { return (double)hi + (double)lo; }
};

__device__ __forceinline__ df two_sum(float a, float b) {
  const float s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  return df(s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb)));
}
__device__ __forceinline__ df operator+(df x, df y) {
  const df s = two_sum(x.hi, y.hi);
  return df(s.hi, __fadd_rn(s.lo, __fadd_rn(x.lo, y.lo)));
}
__host__ __device__ constexpr df operator-(df x) { return df(-x.hi, -x.lo); }
__device__ __forceinline__ df operator-(df x, df y) { return x + (-y); }
__device__ __forceinline__ df operator*(df x, df y) {
  const float p = __fmul_rn(x.hi, y.hi);
  const float e = __fmaf_rn(x.hi, y.hi, -p);  // the exact rounding error of hi * hi
  const float t = __fmaf_rn(x.lo, y.hi, __fmul_rn(x.hi, y.lo));
  return df(p, __fadd_rn(e, t));
}
// the pair renormalised, and its FP32 value
__device__ __forceinline__ df settle(df x) { return two_sum(x.hi, x.lo); }
__device__ __forceinline__ float to_float(df x) { return __fadd_rn(x.hi, x.lo); }

// a complex double-word, laid out like double2 (16 bytes, 16-byte aligned)
struct __align__(16) dfc {
  df x, y;
};
__device__ __forceinline__ dfc settle(dfc v) { return dfc{settle(v.x), settle(v.y)}; }
__device__ __forceinline__ float2 settle(float2 v) { return v; }
__device__ __forceinline__ double2 settle(double2 v) { return v; }

}  // namespace tmbir
