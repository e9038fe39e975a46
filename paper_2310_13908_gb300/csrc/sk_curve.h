// sk_curve.h -- place of a point on a Hilbert curve (a CPU test compiles it with
// the host compiler).
#pragma once

#include <cstdint>

#ifdef __CUDACC__
#define SK_CURVE_HD __host__ __device__ __forceinline__
#else
#define SK_CURVE_HD inline
#endif

namespace sk {

constexpr int CURVE_BITS = 10;  // per axis

// Spread the low 10 bits of v so that bit i lands at bit 3i.
SK_CURVE_HD uint32_t spread3(uint32_t v) {
  v &= 0x3ffu;
  v = (v | (v << 16)) & 0x030000ffu;
  v = (v | (v << 8)) & 0x0300f00fu;
  v = (v | (v << 4)) & 0x030c30c3u;
  v = (v | (v << 2)) & 0x09249249u;
  return v;
}

// Place of cell (x, y, z) of a 2^CURVE_BITS grid on the Hilbert curve: Skilling's
// transform (Programming the Hilbert curve, AIP Conf. Proc. 707, 2004): from the
// highest bit down each axis' bit inverts or exchanges the lower bits of the first
// axis, then the Gray code is undone and the axes' bits are interleaved.
SK_CURVE_HD uint32_t hilbert_key(uint32_t x, uint32_t y, uint32_t z) {
  for (uint32_t q = 1u << (CURVE_BITS - 1); q > 1u; q >>= 1) {
    const uint32_t low = q - 1u;
    if (x & q) x ^= low;
    const uint32_t ty = (y & q) ? 0u : (x ^ y) & low;
    x ^= (y & q) ? low : ty;
    y ^= ty;
    const uint32_t tz = (z & q) ? 0u : (x ^ z) & low;
    x ^= (z & q) ? low : tz;
    z ^= tz;
  }
  y ^= x;
  z ^= y;
  uint32_t t = z;  // parity of the bits above each bit
  t ^= t >> 1;
  t ^= t >> 2;
  t ^= t >> 4;
  t ^= t >> 8;
  t >>= 1;
  return spread3(z ^ t) | (spread3(y ^ t) << 1) | (spread3(x ^ t) << 2);
}

}  // namespace sk
