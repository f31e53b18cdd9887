// Quotients a / d by a divisor whose correctly rounded reciprocal is formed
// ahead (a kernel argument, or one thread's work behind a wait): Markstein's
// correction of the product (IBM J. Res. Dev. 34, 1990),
//   q = a inv,  a / d = q + (a - q d) inv  with both steps fused,
// gives the rounded quotient in three operations, where an FP64 division is
// some ten of a pipe of 0.4 lanes per clock and scheduler.  Checked against
// division on the host, over every FP32 numerator of a binade; it holds while a,
// d, the quotient and the remainder a - q d stay in the normal range (a
// remainder below it can cost the last bit).  An infinite or NaN product is the
// quotient as it stands.
//
// Host and device, so that a plain C++ build can check it.
#pragma once

#if defined(__CUDACC__)
#define DIV_FN __host__ __device__ __forceinline__
#else
#define DIV_FN inline
#endif
#include <cmath>

namespace ebk {

template <class A>
struct DivBy {
  A d, inv;
  // an infinite divisor (a steady problem's time step) gives 0, as 0 a / 1: its
  // own remainder a - 0 d is not a number
  static DivBy of(double d) { return std::isinf((A)d) ? DivBy{1, 0} : DivBy{(A)d, (A)1 / (A)d}; }
};

// on the integer pipe: an FP64 comparison costs what an FP64 addition does
DIV_FN bool div_finite(double q) {
#if defined(__CUDA_ARCH__)
  return (__double2hiint(q) & 0x7ff00000) != 0x7ff00000;
#else
  return std::isfinite(q);
#endif
}
DIV_FN bool div_finite(float q) {
#if defined(__CUDA_ARCH__)
  return (__float_as_int(q) & 0x7f800000) != 0x7f800000;
#else
  return std::isfinite(q);
#endif
}

template <class A>
DIV_FN A div_by(A a, const DivBy<A>& c) {
  using std::fma;
  const A q = a * c.inv;
  const A r = fma(fma(-q, c.d, a), c.inv, q);
  return div_finite(q) ? r : q;
}

}  // namespace ebk
