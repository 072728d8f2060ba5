// Pixels of a window that can see a box, in plain C++ so that a test can
// compile it alone.
#pragma once

#include <algorithm>
#include <cmath>

namespace ivv {

// Upper bound of the number of pixels of frame f's window whose rays meet the
// box [lo, hi]: the rectangle around the projections of its corners, which
// bounds that of the whole box where every corner lies before the eye (else
// the whole window).  The box is taken a thousandth of its diagonal larger and
// the rectangle two pixels, far more than the tolerances of the hits.
template <typename Frame>
inline double pixels_met(const Frame& f, const double lo[3], const double hi[3]) {
  double d2 = 0;
  for (int a = 0; a < 3; ++a) d2 += (hi[a] - lo[a]) * (hi[a] - lo[a]);
  const double pad = 1e-3 * std::sqrt(d2), whole = (double)f.w * (double)f.h;
  double x0 = 1e300, x1 = -1e300, y0 = 1e300, y1 = -1e300;
  for (int c = 0; c < 8; ++c) {
    double x = 0, y = 0, z = 0;
    for (int a = 0; a < 3; ++a) {
      const double e = ((c >> a) & 1 ? hi[a] + pad : lo[a] - pad) - f.eye[a];
      x += e * f.r[a];
      y += e * f.u[a];
      z += e * f.f[a];
    }
    if (!f.ortho) {
      if (!(z > pad)) return whole;
      x /= z;
      y /= z;
    }
    x = (x / f.sx + 1) * 0.5 * f.W - f.x0;       // in pixels of the window
    y = (1 - y / f.sy) * 0.5 * f.H - f.y0;
    x0 = std::min(x0, x);
    x1 = std::max(x1, x);
    y0 = std::min(y0, y);
    y1 = std::max(y1, y);
  }
  const double w = std::min(std::ceil(x1) + 2, (double)f.w) - std::max(std::floor(x0) - 2, 0.0);
  const double h = std::min(std::ceil(y1) + 2, (double)f.h) - std::max(std::floor(y0) - 2, 0.0);
  if (!(w * h <= whole)) return whole;             // NaN
  return w > 0 && h > 0 ? w * h : 0;
}

}  // namespace ivv
