// lb_normals64.cuh -- the double-precision Box-Muller pair formed in 64-bit integer arithmetic.
//
// The FP64 pipe issues two lanes per clock and SM (1/64 of the FP32 rate), so on the double path
// everything that need not run there should not: a pair formed with a table-driven logarithm, a
// square root and the addition theorems in double took about 33 FP64 instructions, 231 of the 428 of
// a lattice update.  Here the radius and the angle come from tables in fixed point and only 32- and
// 64-bit integer instructions (which the pipe's idle issue slots have to spare) combine them.
//
//   u = m 2^-24 with m = 2 (k mod 2^23) + 1 odd.
//   radius sqrt(-2 ln u): q = min(m, 2^24 - m) picks a segment by its exponent and 8 leading bits
//   (side m > q: through 1 - u, so that the radii near u = 1 keep their digits); the rest of q, at
//   most 14 bits, is the variable T of a degree-5 polynomial, the Taylor polynomial of the radius at
//   the segment's middle (its next term is below 2^-56 of it).
//   angle 2 pi m 2^-24: the quadrant from the top two bits, a table of (cos, sin) for the next ten
//   and one of (sin d, 1 - cos d) for the twelve below (odd: 2048 entries), by the addition theorems.
//   The products are truncated at 2^-59; the results carry the tables' double rounding.
// Against quadruple precision on 2^18 random pairs and the ends of the range: at most 7.4e-16 off, 6.9e-17
// rms (the table-driven pair in double: 1.2e-15 and 1.2e-16).  That is an absolute error, of numbers that are
// scaled and added to moments: a normal of 1e-10 has fewer relative digits than in double.  FP64 instructions of a lattice update
// 428 -> 208; four steps of 8192 x 2048 and the state read back 56.4 -> 28.4 ms.  327 KB of segments, 48 KB of
// angles, filled once per context: nothing is formed per block any more (the tables in shared memory cost
// each launch of a small lattice about 20 us).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace lbk {

struct NormalTables {
  struct __align__(16) Segment {  // r(T) = 2^-60 sum_k c_k (T/2)^k, T in [0, 1)
    long long c0, c1, c2, c3;
    int c4, c5;
    int pad[2];
  };
  Segment radius[2 * 4096];    // side 0: by u; side 1: by 1 - u
  ulonglong2 turn[1024];       // 2^63 (cos, sin)(2 pi j / 4096)
  ulonglong2 rest[2048];       // 2^73 (sin d, 1 - cos d), d = 2 pi (2 j + 1) 2^-24
};

// High 64 bits of a b, at most three units low (the low half's carries are left out).
__device__ __forceinline__ unsigned long long mulhi64(unsigned long long a, unsigned long long b) {
  const uint32_t a1 = (uint32_t)(a >> 32), a0 = (uint32_t)a, b1 = (uint32_t)(b >> 32), b0 = (uint32_t)b;
  return (unsigned long long)a1 * b1 + __umulhi(a1, b0) + __umulhi(a0, b1);
}

// 2^-59 x as a double with the given sign bit (x > 0), rounded to nearest.
__device__ __forceinline__ double fixed59(unsigned long long x, uint32_t sign) {
  const int s = __clzll((long long)x);
  const unsigned long long y = x << s;
  const unsigned long long bits = (y >> 11) + ((y >> 10) & 1u) + ((unsigned long long)(1026 - s) << 52);
  return __hiloint2double((int)((uint32_t)(bits >> 32) | sign), (int)(uint32_t)bits);
}

__device__ __forceinline__ void normal_pair_fixed(uint32_t a, uint32_t b, double& n0, double& n1,
                                                  const NormalTables* __restrict__ tab) {
  // radius
  const uint32_t m = 2u * (a & 0x7FFFFFu) + 1u, side = m >> 23;
  const uint32_t q = side ? (1u << 24) - m : m;
  const int sh = max(23 - __clz((int)q), 0);  // e - 8 with q in [2^e, 2^(e+1)), zero below 2^9
  const NormalTables::Segment* sg = tab->radius + (side * 4096u + (uint32_t)sh * 256u + (q >> sh));
  const uint32_t T = (q & ((1u << sh) - 1u)) << (31 - sh);  // T/2 in units of 2^-32
  const longlong2 c01 = __ldg(reinterpret_cast<const longlong2*>(sg)), c23 = __ldg(reinterpret_cast<const longlong2*>(sg) + 1);
  const int2 c45 = __ldg(reinterpret_cast<const int2*>(sg) + 4);
  // angle tables
  const uint32_t m2 = 2u * (b & 0x7FFFFFu) + 1u, quad = m2 >> 22;
  const ulonglong2 C = __ldg(tab->turn + ((m2 >> 12) & 1023u)), D = __ldg(tab->rest + ((m2 & 4095u) >> 1));
  long long p = (long long)(c45.x + __mulhi(c45.y, (int)T));
  p = c23.y + (long long)__mulhi((int)p, (int)T);
  p = c23.x + (long long)(int)(p >> 32) * (int)T + __umulhi((uint32_t)p, T);
  p = c01.y + (long long)(int)(p >> 32) * (int)T + __umulhi((uint32_t)p, T);
  p = c01.x + (long long)(int)(p >> 32) * (int)T + __umulhi((uint32_t)p, T);
  const unsigned long long r = (unsigned long long)p;
  // cos(a + d) = C.x - (C.x (1 - cos d) + C.y sin d), sin(a + d) = C.y + (C.x sin d - C.y (1 - cos d))
  const unsigned long long co = C.x - ((mulhi64(C.x, D.y) + mulhi64(C.y, D.x)) >> 9);
  const unsigned long long si =
      C.y + (unsigned long long)((long long)(mulhi64(C.x, D.x) - mulhi64(C.y, D.y)) >> 9);
  const bool swap = quad & 1u;
  const unsigned long long x0 = mulhi64(r, swap ? si : co), x1 = mulhi64(r, swap ? co : si);
  n0 = fixed59(x0, (quad + 1u) << 30 & 0x80000000u);  // negative in quadrants 1 and 2
  n1 = fixed59(x1, quad << 30 & 0x80000000u);         // negative in quadrants 2 and 3
}

// The tables of the current context, filled on its first use of them (lb_step_f64.cu); the address is good
// for the life of that context, so every lb_ctx asks for its own.
cudaError_t normal_tables(const NormalTables** tab);

}  // namespace lbk
