// Which pixels a projected primitive can reach: conservative tests of its
// alpha >= 1/255 ellipse against boxes of pixel centres, used by the compositing
// kernels to leave out work that cannot contribute. A primitive is
//   q(dx, dy) = A dx^2 + 2B dx dy + C dy^2,  alpha = min(0.99, sigma e^{-q/2}),
// so alpha >= 1/255 iff q <= 2 ln(255 sigma). The pixels decide in FP32; the tests
// keep every pixel that could pass there. Plain arithmetic, shared by the kernels and
// a host-side check against the pixels' own FP32 decision.
#pragma once

#include <math.h>
#include <stdint.h>

#if defined(__CUDACC__)
#define NASG_COVER_HD __host__ __device__ __forceinline__
#else
#define NASG_COVER_HD inline
#endif

namespace nasg {

// The largest q that must be kept, for covariance (sa, sb, sc) with determinant 1/idet, mean
// (u, v) and qmax = 2 ln(255 sigma) >= 0; infinity where nothing may be left out.
// q as the pixels compute it is off by a few ulps of its largest term, at most
// 4 (sa sc / det) q: under 1 % of q for sa sc <= 4096 det (axes up to 64 : 1), and a mean
// within 32768 pixels keeps the offsets to 0.002 px. Within these, 3 % and an absolute 4e-3
// leave room; a NaN gives infinity too.
NASG_COVER_HD float cover_limit(float sa, float sc, float idet, float u, float v, float qmax) {
  const bool sure = (sa * idet) * sc <= 4096.f && fabsf(u) <= 32768.f && fabsf(v) <= 32768.f;
  return sure ? fmaf(1.03f, qmax, 4e-3f) : INFINITY;
}

NASG_COVER_HD float cover_div(float a, float b) {
#if defined(__CUDA_ARCH__)
  return __fdividef(a, b);
#else
  return a / b;
#endif
}

// Where on a line at distance t along the other axis the quadratic is smallest: dy = ry dx at a
// given dx, dx = rx dy at a given dy. (An approximate quotient only moves a candidate.)
struct CoverSlopes {
  float rx, ry;
};
NASG_COVER_HD CoverSlopes cover_slopes(float A, float B2, float C) {
  return {cover_div(-0.5f * B2, A), cover_div(-0.5f * B2, C)};
}

// Whether q can be at most `limit` in the box [xl, xh] x [yl, yh] of offsets from the mean. The
// smallest q over the box is 0 with the mean inside, and otherwise lies on one of the two edges
// that face the mean: on each, the minimiser clamped to the edge. Every candidate is a point of
// the box. A NaN keeps the box.
NASG_COVER_HD bool cover_box(float A, float B2, float C, CoverSlopes r, float limit, float xl, float xh, float yl,
                             float yh) {
  const float cx = fminf(fmaxf(0.f, xl), xh), cy = fminf(fmaxf(0.f, yl), yh);
  const float ey = fminf(fmaxf(r.ry * cx, yl), yh), ex = fminf(fmaxf(r.rx * cy, xl), xh);
  const float q1 = A * cx * cx + (B2 * cx + C * ey) * ey;
  const float q2 = C * cy * cy + (B2 * cy + A * ex) * ex;
  return !(q1 > limit && q2 > limit);
}

}  // namespace nasg
