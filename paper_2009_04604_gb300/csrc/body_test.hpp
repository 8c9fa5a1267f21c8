// body_test.hpp -- the FP32 test that decides most nodes of a moving body's region.
//
// Plain C++ on the host as well, so that its margin can be tested without a GPU.
#pragma once

#ifdef __CUDACC__
#define LBM_BODY_FN __host__ __device__ __forceinline__
#else
#define LBM_BODY_FN inline
#endif

namespace lbm {

// An ellipsoid's reciprocal semi-axes, its rotation about z, and a margin around its
// surface that is wider than the FP32 error.
struct BodySurface {
  float inv[3], ca, sa, tol;
};

// The margin. With u = 2^-24 an offset from the centre carries up to 2 u (|d| + 1) (the
// offset rounded once, a neighbour's step once more), its rotated component 6 u (|d| + 1)
// and the scaled one 9 u (|d| + 1) / r, so that the scaled vector is off by at most
// eps = 9 sqrt(3) u (rmax + 1) / rmin wherever |d| <= rmax, and by eps |d| / rmax beyond.
// A point of the surface or inside it (|d| <= rmax) then never tests above 1 + 2 eps +
// eps^2, and one outside never below 1 - 2 eps: its true length is at least |d| / rmax.
// 2 eps is 1.9e-6 (rmax + 1) / rmin; the margin of 1e-5 rmax / rmin plus 1e-3 (1 + 1 /
// rmin) covers that and eps^2 up to ratios of 10^6. Beyond, no node is decided here.
LBM_BODY_FN BodySurface body_surface(int D, const double r[3], double ca, double sa) {
  BodySurface b;
  float lo = 3e38f, hi = 0.0f;
  for (int a = 0; a < 3; ++a) {
    const float ra = a < D ? (float)(r[a] < 0.0 ? -r[a] : r[a]) : 1.0f;
    b.inv[a] = 1.0f / ra;
    if (a >= D) continue;
    lo = ra < lo ? ra : lo;
    hi = ra > hi ? ra : hi;
  }
  b.ca = (float)ca;
  b.sa = (float)sa;
  const float ratio = hi / lo;
  b.tol = ratio <= 1e6f ? 1e-5f * ratio + 1e-3f * (1.0f + 1.0f / lo) : __builtin_huge_valf();
  return b;
}

// Which side of the surface the offset d from the centre lies on: 1 inside, -1 outside,
// 0 undecided.
LBM_BODY_FN int body_side(const BodySurface &b, float d0, float d1, float d2) {
  const float t0 = (b.ca * d0 + b.sa * d1) * b.inv[0], t1 = (b.ca * d1 - b.sa * d0) * b.inv[1], t2 = d2 * b.inv[2];
  const float t = t0 * t0 + t1 * t1 + t2 * t2;
  if (t < 1.0f - b.tol) return 1;
  if (t > 1.0f + b.tol) return -1;
  return 0;
}

}  // namespace lbm
