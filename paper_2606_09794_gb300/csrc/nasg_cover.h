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

// The same ellipse by tile rows: for a row of tiles, the tiles whose pixel centres the ellipse
// q <= limit can reach. With dy held, the ellipse spans u + r dy -+ sqrt(h (limit - dy^2 / sc)),
// r = sb / sc, h = det / sc; over a band of dy its right end is furthest at dy = y_right =
// sb sqrt(limit / sa) or, that outside the band, at the band's nearer end (the right boundary is
// concave in dy), its left end at -y_right likewise. The launches that count and that list the
// tiles must agree, so on the device every operation is one that the compiler cannot contract.
struct CoverRows {
  float u, v, r, h;
  float limit, isc, y_right, unused;
};

#if defined(__CUDA_ARCH__)
__device__ __forceinline__ float cover_sqrt(float x) {
  float y;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
#define NASG_COVER_MUL __fmul_rn
#define NASG_COVER_ADD __fadd_rn
#define NASG_COVER_FMA __fmaf_rn
#define NASG_COVER_SQRT cover_sqrt
#else
#define NASG_COVER_MUL(a, b) ((a) * (b))
#define NASG_COVER_ADD(a, b) ((a) + (b))
#define NASG_COVER_FMA(a, b, c) fmaf(a, b, c)
#define NASG_COVER_SQRT sqrtf
#endif

NASG_COVER_HD CoverRows cover_rows(float u, float v, float sa, float sb, float sc, float det, float limit) {
  const float isc = 1.f / sc;
  return {u, v, sb * isc, det * isc, limit, isc, sb * sqrtf(limit / sa), 0.f};
}

// Tiles [*c0, *c1] of tile row `row` (16 x 16 tiles), within [x0, x1]; false for none. The 0.05 px
// cover the rounding of means within 32768 pixels.
NASG_COVER_HD bool cover_row(const CoverRows& c, int row, int x0, int x1, int* c0, int* c1) {
  *c0 = x0;
  *c1 = x1;
  if (!(c.limit < INFINITY)) return true;
  const float yl = NASG_COVER_ADD(float(16 * row) + 0.5f, -c.v), yh = NASG_COVER_ADD(float(16 * row) + 15.5f, -c.v);
  const float yr = fminf(fmaxf(c.y_right, yl), yh), ye = fminf(fmaxf(-c.y_right, yl), yh);
  const float tr = NASG_COVER_FMA(NASG_COVER_MUL(-yr, yr), c.isc, c.limit);
  const float te = NASG_COVER_FMA(NASG_COVER_MUL(-ye, ye), c.isc, c.limit);
  if (tr < 0.f && te < 0.f) return false;
  const float right = NASG_COVER_ADD(NASG_COVER_FMA(c.r, yr, c.u), NASG_COVER_SQRT(NASG_COVER_MUL(c.h, fmaxf(tr, 0.f))));
  const float left = NASG_COVER_ADD(NASG_COVER_FMA(c.r, ye, c.u), -NASG_COVER_SQRT(NASG_COVER_MUL(c.h, fmaxf(te, 0.f))));
  // tile t holds the centres 16 t + 0.5 .. 16 t + 15.5
  const float lo = ceilf(NASG_COVER_MUL(NASG_COVER_ADD(left, -15.55f), 0.0625f));
  const float hi = floorf(NASG_COVER_MUL(NASG_COVER_ADD(right, -0.45f), 0.0625f));
  *c0 = int(fminf(fmaxf(lo, float(x0)), float(x1 + 1)));
  *c1 = int(fmaxf(fminf(hi, float(x1)), float(x0 - 1)));
  return *c0 <= *c1;
}

}  // namespace nasg
