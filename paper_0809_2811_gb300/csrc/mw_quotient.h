// mw_quotient.h -- FP64 quotient without the library division, for host and
// device.
//
// GB300 issues an FP64 instruction every ~25 cycles even for one lane, and the
// library division takes several times the five of this one: with five
// divisions the isobaric end of a step took 5.5 us.  The reciprocal comes from
// FP32 (relative error 1.2e-7, both roundings) and one Newton step (1.5e-14);
// the quotient's remainder, in one fused operation, then corrects it
// (Markstein's form), which leaves the rounding of the last operation: the
// division's own result, but for quotients within 1e-27 of a rounding
// boundary.  (A second Newton step instead of the remainder takes as many
// operations and differs from the division in the last bits of a quarter of
// the quotients.)
#pragma once

#include <cmath>
#include <cstdint>
#include <cstring>

#ifdef __CUDACC__
#define MW_HOST_DEVICE __host__ __device__ __forceinline__
#else
#define MW_HOST_DEVICE inline
#endif

namespace mw {

// Operands below 2^-100 or above 2^100 (zero and what is not finite among
// them) divide.
MW_HOST_DEVICE double quotient(double a, double b) {
  uint64_t ua, ub;
  memcpy(&ua, &a, 8);
  memcpy(&ub, &b, 8);
  const unsigned ea = (unsigned)(ua >> 52) & 0x7ffu, eb = (unsigned)(ub >> 52) & 0x7ffu;
  if (ea - 923u > 200u || eb - 923u > 200u) return a / b;  // (2^-100 to 2^100)
  const float bf = (float)b;
#ifdef __CUDA_ARCH__
  double r = (double)__frcp_rn(bf);
#else
  double r = (double)(1.0f / bf);
#endif
  r = fma(r, fma(-b, r, 1.0), r);
  const double q = a * r;
  return fma(fma(-b, q, a), r, q);
}

}  // namespace mw
