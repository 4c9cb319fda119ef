// lb_fixed64.cuh -- sums of doubles in 64-bit integers of one common exponent.
//
// The FP64 pipe issues two lanes per clock and SM, the integer pipe 64: where a group of doubles is only
// added, subtracted and scaled by powers of two (the inverse moment transform), it is cheaper to bring
// them to integers of one scale, combine those exactly, and round once on the way back.  The scale puts
// the largest magnitude's leading bit at bit 57, so a sum of up to 32 of them fits, and values are
// rounded at 2^-58 of the largest: far below the roundings of the same sums in double (2^-53 of each
// partial sum) for every sum that contains the largest value.  Here that is the density, which every link
// contains, unless the flow is far from anything the method describes; a link that lacked the largest value
// could be rounded coarser than in double.  (Cut instead of rounded, and at 2^-55, the error after 100 steps
// was six times that of the double sums: a bias of a fraction of a bit adds up from step to step.)
// Groups with an infinity or a NaN, above 2^1008 or below 2^-950 are left to the caller's double
// arithmetic.
//   Inverse transform of both species: 46 FP64 instructions less per update (177 -> 133; 1472 of them
// hold the pipe as long as about 500 integer ones hold theirs), four steps of 8192 x 2048 and the state
// read back 24.1 -> 20.0 ms.  The densities and momenta formed the same way (133 -> 101) gained 3% there and lost
// 30 to 45% on small lattices, whose halo rows pay the conversions again: they stay in double.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace lbk {

// The exponent field of the scale: the largest exponent field of the group, in place (bits 20..30).
__device__ __forceinline__ uint32_t fixed_field(double x) { return (uint32_t)__double2hiint(x) & 0x7FF00000u; }
__device__ __forceinline__ bool fixed_ok(uint32_t field) { return field - (72u << 20) < (0x7F0u - 72u) << 20; }

// x in units of 2^(e - 57), e the exponent of the field, rounded (halves away from zero).
__device__ __forceinline__ long long to_fixed(double x, uint32_t field) {
  const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
  const uint32_t s = (field - (hi & 0x7FF00000u)) >> 20;  // zero and subnormal values shift out
  const unsigned long long m =
      (((unsigned long long)((hi & 0x000FFFFFu) | 0x00100000u) << 32) | lo) << 6;  // one bit more than kept
  unsigned long long v;
  asm("shr.u64 %0, %1, %2;" : "=l"(v) : "l"(m), "r"(s));  // shifts of 64 and more give 0
  v = (v + 1) >> 1;
  const long long g = (long long)((int)hi >> 31);
  return ((long long)v ^ g) - g;
}

// q 2^EXP in the same units as a double, rounded to nearest, halves to even.
template <int EXP>
__device__ __forceinline__ double from_fixed(long long q, uint32_t field) {
  const uint32_t sign = (uint32_t)(q >> 32) & 0x80000000u;
  const long long g = q >> 63;
  const unsigned long long a = (unsigned long long)((q ^ g) - g);
  const uint32_t ah = (uint32_t)(a >> 32);
  if (ah == 0) {  // small against the group: the conversion instruction, and the scale by the exponent
    if (a == 0) return 0.0;
    const double d = __ull2double_rn(a);
    return __hiloint2double((int)(((uint32_t)__double2hiint(d) + field - ((1023u + 57u - EXP) << 20)) | sign),
                            __double2loint(d));
  }
  const int n = __clz((int)ah);
  const unsigned long long y = a << n;
  const uint32_t yl = (uint32_t)y;
  const unsigned up = (yl & 0x7FFu) + ((yl >> 11) & 1u) > 0x400u ? 1u : 0u;
  const unsigned long long r = (y >> 11) + up;  // 53 bits, the leading one at bit 52 (or 53)
  // exponent of the leading bit: field + (63 - n) - 57 + EXP, less the one that bit 52 itself adds
  const uint32_t top = field + ((uint32_t)(5 + EXP - n) << 20);
  return __hiloint2double((int)(((uint32_t)(r >> 32) + top) | sign), (int)(uint32_t)r);
}

}  // namespace lbk
