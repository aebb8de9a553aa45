// recip.h -- float64 reciprocals in three float64 instructions (device, and the same on the host).
#ifndef PIFA_RECIP_H_
#define PIFA_RECIP_H_

#include <cmath>
#include <cstdint>
#include <cstring>

#ifdef __CUDACC__
#define PIFA_HD __host__ __device__ __forceinline__
#else
#define PIFA_HD inline
#endif

namespace pifa {

template <typename To, typename From>
PIFA_HD To bits_as(From v) {
  To t;
  memcpy(&t, &v, sizeof t);
  return t;
}

// 1 / d for d > 0: the float32 reciprocal of d's significand, good to 2^-22 (its truncation to 23 bits and one
// rounding), and one step of Halley's third-order iteration r (1 + e + e^2), e = 1 - d r: three float64
// instructions, of 64 cycles each for a warp alone on its scheduler, where the division takes about ten.
// The iteration's e^3 is below 2^-65, the rounding of e + e^2 below 2^-75, so that the result is off by 0.5
// units in the last place for the last multiply-add and less than 0.001 for the rest (0.50002 at most over
// all float32 significands and 64 M other values); the division by 0.5. Outside 2^-959 to 2^959 it is the
// division itself.
PIFA_HD double recip(double d) {
  const uint64_t b = bits_as<uint64_t>(d);
  const int ex = (int)(b >> 52);
  if (ex < 64 || ex > 1982) return 1.0 / d;  // the scale below would leave the normal range
  const float m = bits_as<float>(0x3f800000u | (uint32_t)((b >> 29) & 0x7fffffu));  // [1, 2)
#ifdef __CUDA_ARCH__
  const float q0 = __frcp_rn(m);
#else
  const float q0 = 1.0f / m;
#endif
  const uint32_t q = bits_as<uint32_t>(q0);  // (0.5, 1]
  const uint64_t rb =
      ((uint64_t)((int)(q >> 23) - 127 + 1023 - (ex - 1023)) << 52) | ((uint64_t)(q & 0x7fffffu) << 29);
  const double r = bits_as<double>(rb);
  const double e = fma(-d, r, 1.0);
  return fma(r, fma(e, e, e), r);
}

}  // namespace pifa

#endif  // PIFA_RECIP_H_
