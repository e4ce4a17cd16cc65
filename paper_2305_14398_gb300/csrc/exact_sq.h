// Exact square of an FP32 value as an FP64 bit pattern, with integer
// operations only (GB300's FP64 pipe is ~1/64 of its FP32 rate, so the
// per-amplitude |psi|^2 avoids it except for one correctly rounded add).
//
// x = m * 2^(e - 150) with a 24-bit integer significand m (after normalising
// subnormals); x^2 = m^2 * 2^(2e - 300) where m^2 < 2^48 fits an FP64
// significand exactly.  The result is bit-identical to (double)x * (double)x.
// Host and device code (the host build is the unit test's).
#pragma once

#include <cstdint>

#if defined(__CUDACC__)
#define TQS_HD __host__ __device__ __forceinline__
#else
#define TQS_HD inline
#endif

namespace tqs {

TQS_HD int clz32(uint32_t v) {
#if defined(__CUDA_ARCH__)
  return __clz(static_cast<int>(v));
#else
  return v ? __builtin_clz(v) : 32;
#endif
}

TQS_HD uint64_t sq_f32_as_f64_bits_general(uint32_t xbits);

// Normal x (the common case): m in [2^23, 2^24), m^2 in [2^46, 2^48).  The
// significand field is m^2 shifted so that its leading one lands on bit 52;
// adding the exponent field one below the biased exponent absorbs that
// leading one, so no mask is needed.
TQS_HD uint64_t sq_f32_as_f64_bits(uint32_t xbits) {
  const uint32_t a = xbits & 0x7fffffffu;
  if (a < 0x00800000u) return sq_f32_as_f64_bits_general(xbits);  // zero or subnormal
  const uint32_t m = (a & 0x7fffffu) | 0x800000u;
  const int e = static_cast<int>(a >> 23);
  const uint64_t X = static_cast<uint64_t>(m) * m;
  const bool top47 = (static_cast<uint32_t>(X >> 32) >> 15) != 0;  // bit 47 of X
  const uint64_t Y = X << (top47 ? 5 : 6);
  // biased exponent 2e - 254 + 1023 (top bit 47) or one less (top bit 46), minus 1
  const uint64_t ebits = static_cast<uint64_t>(2 * e + 768 + (top47 ? 1 : 0)) << 52;
  return ebits + Y;
}

// Any finite x, subnormals included.
TQS_HD uint64_t sq_f32_as_f64_bits_general(uint32_t xbits) {
  const uint32_t a = xbits & 0x7fffffffu;
  int e = static_cast<int>(a >> 23);
  uint32_t m = a & 0x7fffffu;
  if (e == 0) {
    if (m == 0) return 0;
    const int s = clz32(m) - 8;  // bring the leading one to bit 23
    m <<= s;
    e = 1 - s;
  } else {
    m |= 0x800000u;
  }
  const uint64_t X = static_cast<uint64_t>(m) * m;  // in [2^46, 2^48)
  const int top = (X >> 47) ? 47 : 46;
  const int E = top + 2 * e - 300;                   // unbiased FP64 exponent
  const uint64_t frac = (X << (52 - top)) & ((uint64_t(1) << 52) - 1);
  return (static_cast<uint64_t>(E + 1023) << 52) | frac;
}

// The FP64 bits of x^2 + y^2 correctly rounded (round to nearest, ties to
// even: the FP64 sum of the exact squares above), integers only.  The larger
// square, m^2 < 2^48 for the 24-bit significand m, is placed with its low bit
// at bit 15 of a 64-bit sum, the other aligned to it (what falls below bit 0
// only matters as "something": it is or-ed into bit 0, which is below the
// rounding position), and the sum, in [2^61, 2^64), is rounded to 53 bits.
TQS_HD uint64_t sq_sum_bits(uint32_t xbits, uint32_t ybits) {
  const uint32_t ax = xbits & 0x7fffffffu, ay = ybits & 0x7fffffffu;
  const uint32_t hi = ax > ay ? ax : ay, lo = ax > ay ? ay : ax;
  if (hi < 0x00800000u) {
    // both zero or subnormal: m < 2^23 at 2^-149 each, the sum is exact
    const uint64_t s = static_cast<uint64_t>(hi) * hi + static_cast<uint64_t>(lo) * lo;
    if (s == 0) return 0;
    const uint32_t sh = static_cast<uint32_t>(s >> 32);
    const int lz = sh ? clz32(sh) : 32 + clz32(static_cast<uint32_t>(s));
    return (static_cast<uint64_t>(1023 - 298 + 62 - lz) << 52) + (s << (lz - 11));
  }
  const int eh = static_cast<int>(hi >> 23);
  const bool sub = lo < 0x00800000u;
  const int el = sub ? 1 : static_cast<int>(lo >> 23);
  const uint32_t mh = (hi & 0x7fffffu) | 0x800000u, ml = (lo & 0x7fffffu) | (sub ? 0u : 0x800000u);
  const uint64_t B = static_cast<uint64_t>(ml) * ml;
  const int r = 2 * (eh - el) - 15;  // bits B moves right
  uint64_t b;
  if (r <= 0) {
    b = B << -r;
  } else {
    b = r < 63 ? B >> r : 0;
    b |= (r < 63 ? (b << r) != B : B != 0) ? 1 : 0;
  }
  const uint64_t s = ((static_cast<uint64_t>(mh) * mh) << 15) + b;
  const uint32_t top = static_cast<uint32_t>(s >> 32);
  const int k = 9 + (top >= 0x40000000u ? 1 : 0) + (top >= 0x80000000u ? 1 : 0);  // bits rounded off
  const uint64_t q = (s + ((uint64_t(1) << (k - 1)) - 1) + ((s >> k) & 1)) >> k;
  return (static_cast<uint64_t>(2 * eh + 759 + k) << 52) + q;
}

#if defined(__CUDACC__)
// |x + iy|^2 correctly rounded to FP64 (bit-identical to (double)x * x +
// (double)y * y): the two squares are exact FP64 values built with integer
// operations, one FP64 add rounds their sum.
__device__ __forceinline__ double sq_sum_f64(float x, float y) {
  const double a = __longlong_as_double(static_cast<long long>(sq_f32_as_f64_bits(__float_as_uint(x))));
  const double b = __longlong_as_double(static_cast<long long>(sq_f32_as_f64_bits(__float_as_uint(y))));
  return __dadd_rn(a, b);
}
#endif

}  // namespace tqs
