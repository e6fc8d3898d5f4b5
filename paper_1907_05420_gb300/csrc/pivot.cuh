// Reciprocal of a pivot (device code shared by the factor kernels).
#pragma once

namespace kkt {

// FP64, in integer arithmetic.  An FP64 operation keeps a warp 64 cycles on
// this GPU (a conversion to or from FP32 the same pipe), an integer one 4 to 5,
// and the reciprocal heads the dependency chain of every pivot.  With the
// significand m = M 2^-52 in [1, 2) and a seed r = R 2^-24 of 1 / m (R an
// integer of 24 bits, from the FP32 approximation at m's leading 24 bits:
// |1 - m r| < 2^-21), e = 1 - m r is the exact integer E = 2^76 - M R (below
// 2^55, so its low 64 bits hold it), and the three-term series
//     1 / m = r (1 + e + e^2 + ...),  remainder e^3 < 2^-63,
// is summed in fixed point to 62 bits and rounded once: within an ulp of 1/d.
// Pivots of magnitude outside [2^-119, 2^120) use the division (about 650
// cycles).
static __device__ __noinline__ double pivot_recip_div(double d) { return 1.0 / d; }

__device__ __forceinline__ double pivot_recip(double d) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(d);
  const unsigned int hi = (unsigned int)(b >> 32);
  const int ex = (int)((hi >> 20) & 0x7ffu);
  if ((unsigned)(ex - (1023 - 119)) > 238u) return pivot_recip_div(d);
  const unsigned long long M = (b & 0xfffffffffffffULL) | (1ULL << 52);
  float rf;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(rf) : "f"(__uint_as_float(0x3f800000u | (unsigned int)(M >> 29) & 0x7fffffu)));
  const unsigned int rb = __float_as_uint(rf);  // in [0.5, 1]
  const unsigned int R = ((rb & 0x7fffffu) | 0x800000u) << ((rb >> 23) - 126u);
  const long long E = (long long)(0ULL - M * R);
  const long long eh = E >> 25;
  const long long P = E + ((eh * eh) >> 26);                                     // e + e^2 in units of 2^-76
  const long long Q = ((long long)R << 38) + (((long long)R * (P >> 16)) >> 22);  // r (1 + e + e^2) in units of 2^-62
  // Q is about [2^61, 2^62]: 53 bits from 2^52 on, a carry running into the exponent
  const unsigned long long q = (unsigned long long)((Q + 256) >> 9) - (1ULL << 52);
  const unsigned long long r = ((unsigned long long)(2045 - ex) << 52) + q;
  return __longlong_as_double((long long)(r | (b & 0x8000000000000000ULL)));
}
__device__ __forceinline__ float pivot_recip(float d) { return __frcp_rn(d); }

}  // namespace kkt
