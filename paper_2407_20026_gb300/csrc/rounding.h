// Whether the float nearest a computed quotient is certain (CUDA and host code).
#ifndef SSO_ROUNDING_H
#define SSO_ROUNDING_H

#ifdef __CUDACC__
#define SSO_HD __host__ __device__ __forceinline__
#else
#include <math.h>
#define SSO_HD static inline
#endif

namespace sso {
// The bound on everything that separates the computed quotient from the FP64 one
// is relative, 0.93 2^-34 of it.  f is the float nearest the computed quotient,
// in (1/2, 2) and no power of two, rest what it leaves.  Ziv's test in absolute
// terms: rest is farther from half of f's last place than 2^-34 below one and
// 2^-33 from there on, 2^-9 of that half.
SSO_HD bool quotient_certain(float f, float rest) {
  return fabsf(rest) < (f < 1.f ? 0x1.ffp-26f : 0x1.ffp-25f);
}
}  // namespace sso

#endif
