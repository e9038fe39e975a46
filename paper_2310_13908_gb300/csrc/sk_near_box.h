// sk_near_box.h -- the box tests of the FP32 pair kernels: which segments, and
// which of a segment's sources, may have a pair inside rho_c delta with one of a
// warp's targets (a CPU test compiles this with the host compiler, without
// contraction).
//
// The regimes are decided on the FP32 difference of a pair, formed from
// coordinates relative to the segment's frame c: fl(fl(fl(x_hi - c) + x_lo) + r),
// r = -fl(y - c). It deviates from the true x - y by at most three roundings of
// the frame offset, 3 * 2^-24 |y - c| per axis, whatever the pair's distance. The
// box tests hold absolute FP32 positions, a few roundings of the coordinates'
// magnitude off (box_margin), and a source's position rebuilt from its record one
// rounding of |y - c| more. A test that leaves the frame offset out clears a source that
// coincides with a target near the origin, if the segment is wide and delta below
// 1e-8 of its extent: the far formula then divides by zero.
#pragma once

#include <cmath>

#ifdef __CUDACC__
#define SK_BOX_HD __host__ __device__ __forceinline__
#else
#define SK_BOX_HD inline
#endif

namespace sk {
namespace p32 {

// Slack of the box tests per unit of frame offset: 2^-21, twice the four roundings
// above.
constexpr float FRAME_SLACK = 4.76837158203125e-07f;

// Margin added to rho_c delta: absolute FP32 coordinates against frame-relative
// ones, a few roundings of the coordinates' magnitude.
SK_BOX_HD float box_margin(float coord_max, float rc) { return 1.0e-6f * (coord_max + rc); }

// Interval [lo, hi] of one axis, with its slack.
struct Span {
  float lo, hi;
};
// A segment's box on one axis: frame offsets are at most its half extent.
SK_BOX_HD Span segment_span(float lo, float hi) {
  const float e = (0.5f * FRAME_SLACK) * (hi - lo);
  return {lo - e, hi + e};
}
// A source from its segment's frame c and record r = -(y - c).
SK_BOX_HD Span source_span(float c, float r) {
  const float x = c - r, e = FRAME_SLACK * std::fabs(r);
  return {x - e, x + e};
}

// The box of a warp's targets and the squared distance (with box_margin) within
// which a source may have a pair inside rho_c delta with one of them.
struct NearBox {
  float lo[3], hi[3], r2;
  SK_BOX_HD bool reaches(Span x, Span y, Span z) const {
    const float dx = std::fmax(0.f, std::fmax(x.lo - hi[0], lo[0] - x.hi));
    const float dy = std::fmax(0.f, std::fmax(y.lo - hi[1], lo[1] - y.hi));
    const float dz = std::fmax(0.f, std::fmax(z.lo - hi[2], lo[2] - z.hi));
    return dx * dx + dy * dy + dz * dz < r2;
  }
};

}  // namespace p32
}  // namespace sk
