// Float64 products on the integer pipe.
//
// GB300 issues two float64 operations per clock and SM: a warp's float64 FMA
// holds the pipe of its quarter of the SM for 64 cycles, in which the quarter
// issues 64 integer instructions of other kinds.  The float64 stencil passes
// have 8 to 11 float64 operations per point and were bound by that pipe, at
// twice the time of their memory traffic.  Here part of a point's products is
// formed and added in fixed point on the integer pipe instead, while the
// float64 pipe does the rest.
//
// A product u c of two doubles is the floor of the top 62 bits of the 126-bit
// product of their mantissas (left-aligned in 63 bits).  The four terms of a sum
// are rounded to nearest at two guard bits below the largest exponent among
// them and added as 64-bit integers: they are off by at most 2^-57 of the
// largest, where each rounding of a float64 multiply-add chain may be off by
// 2^-53 of it.  The sum is rounded once, to float64.  Rounding, not truncation:
// a truncated term is low at every point of a smooth field alike, and a V-cycle
// amplifies a smooth residual error by orders of magnitude (129^3: 5.8e-16 from
// the exact cycle with truncated terms, against 3.5e-16 of float64 arithmetic).
//
// Operand range: coefficients are positive normal numbers in 2^-230 .. 2^230
// (checked at setup; a hierarchy outside it keeps the float64 kernels).  u may
// be anything: a zero or subnormal u enters as a normal number of at most
// 2^-1022, below the last bit kept as long as the largest term is not tiny
// itself, and soft_sum4() leaves points whose largest term lies outside
// 2^-706 .. 2^774 (all zeros, infinities and NaN among them) and sums that
// cancelled by more than 2^27 to the caller's float64 arithmetic.
#pragma once
#include "mg_device.cuh"

namespace mgdev {

struct S64 {
  unsigned h, l;  // mantissa, leading one at bit 62 of (h, l)
  int e;          // biased exponent
  unsigned s;     // all ones when negative (not set by soft_coef)
};

__host__ __device__ __forceinline__ S64 soft_coef(double c) {
  const unsigned long long b = dbits(c);
  const unsigned long long m = b << 10;
  return {((unsigned)(m >> 32) & 0x3fffffffu) | 0x40000000u, (unsigned)m, (int)((unsigned)(b >> 32) >> 20), 0u};
}
__host__ __device__ __forceinline__ S64 soft_unpack(double u) {
  S64 r = soft_coef(u);
  r.e &= 0x7ff;
  r.s = (unsigned)((int)(unsigned)(dbits(u) >> 32) >> 31);
  return r;
}
// floor of the top half of the mantissas' product plus `half`, the product in [2^60, 2^62)
__host__ __device__ __forceinline__ unsigned long long soft_mul(const S64& u, const S64& c, unsigned long long half) {
#ifdef __CUDA_ARCH__
  unsigned long long t = __umulhi(u.l, c.l);
#else
  unsigned long long t = ((unsigned long long)u.l * c.l) >> 32;
#endif
  t += (unsigned long long)u.h * c.l;  // < 2^63
  t += (unsigned long long)u.l * c.h;  // < 2^64
  return ((unsigned long long)u.h * c.h + half) + (t >> 32);
}
// logical shift right, 0 for s >= 64
__host__ __device__ __forceinline__ unsigned long long soft_shr(unsigned long long v, int s) {
#ifdef __CUDA_ARCH__
  unsigned long long r;
  asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(s));
  return r;
#else
  return s > 63 ? 0 : v >> s;
#endif
}
// half of the bit that a shift right by s >= 1 keeps last; 0 for s > 64
__host__ __device__ __forceinline__ unsigned long long soft_half(int s) {
#ifdef __CUDA_ARCH__
  unsigned long long r;
  asm("shl.b64 %0, %1, %2;" : "=l"(r) : "l"(1ull), "r"(s - 1));
  return r;
#else
  return s > 64 ? 0 : 1ull << (s - 1);
#endif
}
__host__ __device__ __forceinline__ int soft_clz(unsigned v) {
#ifdef __CUDA_ARCH__
  return __clz((int)v);
#else
  return v ? __builtin_clz(v) : 32;
#endif
}

// Sum of the four products u[i] c[i].  Returns false where the caller has to form the sum itself.
__host__ __device__ __forceinline__ bool soft_sum4(const S64 (&u)[4], const S64 (&c)[4], double& out) {
  int E[4], M;
  E[0] = M = u[0].e + c[0].e;
#pragma unroll
  for (int i = 1; i < 4; ++i) {
    E[i] = u[i].e + c[i].e;
    M = E[i] > M ? E[i] : M;
  }
  unsigned long long a = 0;
  unsigned minus = 0;  // minus the number of negative terms (-x = ~x + 1)
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int s = M + 2 - E[i];
    const unsigned long long m = ((unsigned long long)u[i].s << 32) | u[i].s;
    a += soft_shr(soft_mul(u[i], c[i], soft_half(s)), s) ^ m;  // at most 2^60 each
    minus += u[i].s;
  }
  a += 0u - minus;
  const unsigned sg = (unsigned)((int)(unsigned)(a >> 32) >> 31);
  a ^= ((unsigned long long)sg << 32) | sg;
  a += sg & 1u;
  const unsigned top = (unsigned)(a >> 32);
  const int n = soft_clz(top);
  // leading one to bit 62, then to bit 52 with rounding; the value is a 2^(M - 2104)
  const unsigned long long r = ((a << ((n - 1) & 63)) + 0x200ull) >> 10;
  const unsigned hi = (unsigned)(r >> 32) + ((unsigned)(M - 1019 - n) << 20);
  out = bitsd(((unsigned long long)(hi | (sg & 0x80000000u)) << 32) | (unsigned)r);
  return (unsigned)(M - 1340) < 1480u && top != 0;
}

// Whether all four are zeros; their sum in z (-0 where all are -0).
__device__ __forceinline__ bool all_zero(double a, double b, double c, double d, double& z) {
  const unsigned long long some = dbits(a) | dbits(b) | dbits(c) | dbits(d);
  z = bitsd(dbits(a) & dbits(b) & dbits(c) & dbits(d));
  return some << 1 == 0;
}

}  // namespace mgdev
