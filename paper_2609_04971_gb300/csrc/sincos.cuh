// Sine and cosine of an fp64 angle, |a| < 2^64, in integer arithmetic: 0.501 ulp at most on rotary angles (the
// host library's 0.56, CUDA's fp64 functions, which run on this part's slow fp64 pipe, 1.48).
//
// Payne and Hanek's reduction: the angle's 53 bits times 256 bits of 2 / pi give the quadrant and the rest as
// a fraction, which times pi / 4 is the reduced angle r with 64 significant bits.  The Taylor series of 1 -
// sin(r) / r and 1 - cos(r), to r^18, are evaluated in 64-bit fixed point, where a step is one high product.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>
#include <string.h>

namespace bkv {

__host__ __device__ inline uint64_t mul_hi(uint64_t a, uint64_t b) {
#ifdef __CUDA_ARCH__
  return __umul64hi(a, b);
#else
  return static_cast<uint64_t>((static_cast<unsigned __int128>(a) * b) >> 64);
#endif
}

__host__ __device__ inline int leading_zeros(uint64_t v) {  // v != 0
#ifdef __CUDA_ARCH__
  return __clzll(static_cast<long long>(v));
#else
  return __builtin_clzll(v);
#endif
}

// The double nearest to (v / 2^64) 2^ex (ties to even), v != 0, for results in fp64's normal range.
__host__ __device__ inline double fraction_to_double(uint64_t v, int ex, bool negative) {
  const int nz = leading_zeros(v);
  v <<= nz;
  uint64_t m = v >> 11;
  const uint64_t low = v & 0x7ffu;
  m += (low > 0x400u || (low == 0x400u && (m & 1u))) ? 1u : 0u;  // 2^53 after a carry: the exponent's next value
  const uint64_t bits = (static_cast<uint64_t>(1022 - 1 + ex - nz) << 52) + m + (negative ? 1ull << 63 : 0ull);
#ifdef __CUDA_ARCH__
  return __longlong_as_double(static_cast<long long>(bits));
#else
  double d;
  memcpy(&d, &bits, sizeof d);
  return d;
#endif
}

// sn = sin(a), cs = cos(a); from 2^64 on, where a position times a frequency does not come, CUDA's functions.
__host__ __device__ inline void sincos_accurate(double a, double& sn, double& cs) {
  uint64_t bits;
#ifdef __CUDA_ARCH__
  bits = static_cast<uint64_t>(__double_as_longlong(a));
#else
  memcpy(&bits, &a, sizeof bits);
#endif
  const bool minus = bits >> 63;
  const int e = static_cast<int>((bits >> 52) & 0x7ff) - 1023;  // 2^e <= |a| < 2^(e + 1)
  if (e < -32) {  // sin a = a (1 - 2^-66), cos a = 1 - 2^-65
    sn = a;
    cs = 1.0;
    return;
  }
  if (e > 63) {
    ::sincos(a, &sn, &cs);
    return;
  }
  const uint64_t x = ((bits & 0xfffffffffffffull) | 0x10000000000000ull) << 11;  // |a| = x 2^(e - 63)
  // p = x (2 / pi), 320 bits: |a| 2 / pi = p 2^(e - 319)
  constexpr uint64_t t3 = 0xa2f9836e4e441529ull, t2 = 0xfc2757d1f534ddc0ull, t1 = 0xdb6295993c439041ull,
                     t0 = 0xfe5163abdebbc561ull;
  const uint64_t p1l = x * t1, p2l = x * t2, p3l = x * t3;
  uint64_t p1 = p1l + mul_hi(x, t0);
  uint64_t carry = p1 < p1l;
  uint64_t p2 = p2l + mul_hi(x, t1);
  uint64_t c2 = p2 < p2l;
  p2 += carry;
  c2 += p2 < carry;
  uint64_t p3 = p3l + mul_hi(x, t2);
  uint64_t c3 = p3 < p3l;
  p3 += c2;
  c3 += p3 < c2;
  const uint64_t p4 = mul_hi(x, t3) + c3;
  // the quadrant's two bits to the top: 192 bits q2 q1 q0
  uint64_t q2, q1, q0;
  const int s = e - 1;
  if (s > 0) {
    q2 = (p4 << s) | (p3 >> (64 - s));
    q1 = (p3 << s) | (p2 >> (64 - s));
    q0 = (p2 << s) | (p1 >> (64 - s));
  } else if (s == 0) {
    q2 = p4;
    q1 = p3;
    q0 = p2;
  } else {
    q2 = p4 >> -s;
    q1 = (p3 >> -s) | (p4 << (64 + s));
    q0 = (p2 >> -s) | (p3 << (64 + s));
  }
  int n = static_cast<int>(q2 >> 62);
  uint64_t f2 = (q2 << 2) | (q1 >> 62), f1 = (q1 << 2) | (q0 >> 62), f0 = q0 << 2;
  const bool back = f2 >> 63;  // past the middle of the quadrant: counted back from the next one
  if (back) {
    ++n;
    f0 = ~f0 + 1u;
    f1 = ~f1 + (f0 == 0u);
    f2 = ~f2 + (f0 == 0u && f1 == 0u);
  }
  int lz = 0;
  if (f2 == 0u) {
    f2 = f1;
    f1 = f0;
    f0 = 0u;
    lz = 64;
  }
  if (f2 == 0u) f2 = 1u;  // no fp64 angle comes this close to a multiple of pi / 2
  const int z0 = leading_zeros(f2);
  if (z0 > 0) {
    f2 = (f2 << z0) | (f1 >> (64 - z0));
    f1 = (f1 << z0) | (f0 >> (64 - z0));
  }
  lz += z0;
  // r = (f2 f1) (pi / 4) 2^(1 - lz): 64 bits, r1 in [0.39, 0.79) 2^64
  constexpr uint64_t h1 = 0xc90fdaa22168c234ull, h0 = 0xc4c6628b80dc1cd1ull;
  const uint64_t mid = f2 * h1, add1 = mul_hi(f2, h0), add0 = mul_hi(f1, h1);
  uint64_t sum = mid + add1;
  uint64_t up = sum < mid;
  sum += add0;
  up += sum < add0;
  uint64_t r1 = mul_hi(f2, h1) + up;
  int ex = 1 - lz;
  if (!(r1 >> 63)) {
    r1 = (r1 << 1) | (sum >> 63);
    --ex;
  }
  // z = r^2 in units of 2^-64 (r < 1, so ex <= 0)
  const uint64_t r = -ex < 64 ? r1 >> -ex : 0u;
  const uint64_t z = mul_hi(r, r);
  // 1 - sin(r) / r = z (1/3! - z (1/5! - ..)), 1 - cos(r) = z (1/2! - z (1/4! - ..))
  uint64_t u = 0x98ull, v = 0xb41ull;
  u = 0xca96ull - mul_hi(z, u);
  v = 0xd73faull - mul_hi(z, v);
  u = 0xd73f9full - mul_hi(z, u);
  v = 0xc9cba54ull - mul_hi(z, v);
  u = 0xb092309dull - mul_hi(z, u);
  v = 0x8f76c77fcull - mul_hi(z, v);
  u = 0x6b99159fd5ull - mul_hi(z, u);
  v = 0x49f93edde28ull - mul_hi(z, v);
  u = 0x2e3bc74aad8eull - mul_hi(z, u);
  v = 0x1a01a01a01a02ull - mul_hi(z, v);
  u = 0xd00d00d00d00dull - mul_hi(z, u);
  v = 0x5b05b05b05b05bull - mul_hi(z, v);
  u = 0x222222222222222ull - mul_hi(z, u);
  v = 0xaaaaaaaaaaaaaabull - mul_hi(z, v);
  u = 0x2aaaaaaaaaaaaaabull - mul_hi(z, u);
  v = 0x8000000000000000ull - mul_hi(z, v);
  u = mul_hi(z, u);
  v = mul_hi(z, v);
  n &= 3;
  // sin and cos of the reduced angle, and of |a|: 0: s, c  1: c, -s  2: -s, -c  3: -c, s
  const double sr = fraction_to_double(r1 - mul_hi(r1, u), ex, back), cr = v ? fraction_to_double(0u - v, 0, false) : 1.0;
  const double so = (n & 1) ? cr : sr, co = (n & 1) ? sr : cr;
  sn = ((n & 2) != 0) != minus ? -so : so;
  cs = (n == 1 || n == 2) ? -co : co;
}

}  // namespace bkv
