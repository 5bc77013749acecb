// Reciprocal of a level's complex pivot (zsweep.cu), with one division.  Plain
// C++, so the same code also builds on its own for host-only tests.
#pragma once

#include <math.h>

#ifdef __CUDACC__
#define ZQ_FN __device__ __forceinline__
#else
#define ZQ_FN static inline
#endif

// q = 1 / (x + i y); returns |x + i y|^2.  The products of the conjugate with the
// reciprocal of the rounded square are corrected by the residual 1 - (x + i y) q,
// which the fused multiply-adds form without the rounding of the square: a real
// pivot's quotient is correctly rounded, and a complex one's error is 0.43 - 0.53
// units of 2^-53 (root mean square) where Smith's scaled division has 0.44 - 0.62
// and quotients corrected against the rounded square 0.60 - 0.74.
ZQ_FN double zquot(double x, double y, double& qx, double& qy) {
  const double n2 = fma(x, x, y * y), inv = 1.0 / n2;
  const double ax = x * inv, ay = -y * inv;
  const double er = fma(y, ay, fma(-x, ax, 1.0)), ei = -fma(x, ay, y * ax);
  qx = fma(ax, er, fma(-ay, ei, ax));
  qy = fma(ax, ei, fma(ay, er, ay));
  return n2;
}
