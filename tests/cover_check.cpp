// Host-side check of the compositing kernels' reach tests (csrc/nasg_cover.h) against the pixels'
// own FP32 decision: for random projected primitives (axes of the ellipse from 0.55 to 600
// pixels, up to far beyond the 64 : 1 rule, any orientation, means near and far from the image,
// opacities down to 1/255) every pixel whose FP32 alpha reaches 1/255 lies in a kept box and a kept tile. The
// FP32 operations are the kernels' (no contraction here: the rounding differs by ulps, which is
// what the tests' margins are for). Also counts what the box test leaves out, so that a test that
// keeps everything does not pass. Prints "ok ..." and exits 0, or the first failure and exits 1.
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <random>

#include "nasg_cover.h"

using namespace nasg;

int main() {
  std::mt19937_64 gen(20260101);
  std::uniform_real_distribution<double> U(0.0, 1.0);
  long boxes = 0, out = 0, pixels = 0, tiles = 0, tiles_out = 0;
  for (int it = 0; it < 20000; ++it) {
    // covariance from two axes and an angle; a low-pass of 0.3 as the projection adds
    const double l0 = std::exp(U(gen) * std::log(600.0)), l1 = l0 * std::exp(-U(gen) * (it % 3 ? 3.5 : 8.0));
    const double th = U(gen) * 6.283185307179586, c = std::cos(th), s = std::sin(th);
    const float sa = float(c * c * l0 * l0 + s * s * l1 * l1 + 0.3), sc = float(s * s * l0 * l0 + c * c * l1 * l1 + 0.3);
    const float sb = float(c * s * (l0 * l0 - l1 * l1));
    const float det = sa * sc - sb * sb;
    if (!(det > 0.f)) continue;
    const float idet = 1.f / det;
    const float A = sc * idet, B2 = 2.f * (-sb * idet), C = sa * idet;
    const float sig = float(it % 7 == 0 ? 1.0 / 255.0 + U(gen) * 1e-3 : 0.004 + U(gen) * 0.99);
    if (!(sig * 255.f > 1.f)) continue;
    const float scale = it % 5 == 0 ? 4000.f : 60.f;
    const float u = float((U(gen) - 0.5) * scale + 100.0), v = float((U(gen) - 0.5) * scale + 100.0);
    const float limit = cover_limit(sa, sc, idet, u, v, 2.f * std::log(255.f * sig));
    const CoverSlopes r = cover_slopes(A, B2, C);
    // tile rows: tiles [1, 12] x rows [-1, 12] around the ellipse
    const CoverRows rows = cover_rows(u, v, sa, sb, sc, det, limit);
    for (int row = -1; row <= 12; ++row) {
      int c0, c1;
      const bool some = cover_row(rows, row, 1, 12, &c0, &c1);
      if (some && (c0 < 1 || c1 > 12)) {
        std::printf("FAIL it=%d row %d span %d %d\n", it, row, c0, c1);
        return 1;
      }
      for (int t = 1; t <= 12; ++t) {
        ++tiles;
        if (some && t >= c0 && t <= c1) continue;
        ++tiles_out;
        for (int y = 0; y < 16; ++y)
          for (int x = 0; x < 16; ++x) {
            const float dx = (float(16 * t + x) + 0.5f) - u, dy = (float(16 * row + y) + 0.5f) - v;
            const float q = std::fmaf(A * dx, dx, std::fmaf(B2 * dx, dy, (C * dy) * dy));
            if (q < 12.f && double(sig) * std::exp(-0.5 * double(q)) * (1.0 + 4e-6) >= 1.0 / 255.0) {
              std::printf("FAIL it=%d row %d tile %d pixel %d %d q=%g limit=%g sig=%g\n", it, row, t, x, y, q, limit, sig);
              return 1;
            }
          }
      }
    }
    const int w = 8, h = it & 1 ? 8 : 4;
    for (int by = 0; by < 14; ++by) {
      for (int bx = 0; bx < 14; ++bx) {
        const float fx = 40.f + 8.f * float(bx) + 0.5f, fy = 40.f + float(h * by) + 0.5f;
        const bool keep = !(limit < INFINITY) || cover_box(A, B2, C, r, limit, fx - u, (fx + float(w - 1)) - u, fy - v,
                                                           (fy + float(h - 1)) - v);
        ++boxes;
        if (keep) continue;
        ++out;
        for (int y = 0; y < h; ++y)
          for (int x = 0; x < w; ++x) {
            const float dx = (fx + float(x)) - u, dy = (fy + float(y)) - v;
            const float q = std::fmaf(A * dx, dx, std::fmaf(B2 * dx, dy, (C * dy) * dy));
            ++pixels;
            if (double(sig) * std::exp(-0.5 * double(q)) * (1.0 + 4e-6) >= 1.0 / 255.0) {
              std::printf("FAIL it=%d box %d %d pixel %d %d q=%g limit=%g sig=%g\n", it, bx, by, x, y, q, limit, sig);
              return 1;
            }
          }
      }
    }
  }
  if (out * 4 < boxes || tiles_out * 4 < tiles) {
    std::printf("FAIL only %ld of %ld boxes, %ld of %ld tiles left out\n", out, boxes, tiles_out, tiles);
    return 1;
  }
  std::printf("ok %ld boxes, %ld left out, %ld pixels, %ld tiles, %ld left out\n", boxes, out, pixels, tiles, tiles_out);
  return 0;
}
