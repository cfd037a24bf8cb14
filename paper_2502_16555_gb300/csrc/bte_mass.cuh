// g <- M_v^-1 g for one harmonic (g[0 .. nr), unit stride) by the banded Cholesky factor M_v = R R^T:
// chol[p][j] = R[p][p - w + j] ([nr][w + 1]), cinv = 1 / R[p][p]. One thread. For the cubic band (w = 3)
// the last three values stay in registers. Bound by the FP64 units: a step is four operations of a warp.
#pragma once

namespace bte {

__device__ __forceinline__ void mass_solve(double* g, const double* __restrict__ chol, const double* __restrict__ cinv,
                                           int nr, int w) {
  if (w == 3) {
    double y1 = 0.0, y2 = 0.0, y3 = 0.0;  // y[p-1], y[p-2], y[p-3]
    for (int p = 0; p < nr; ++p) {
      const double* r = chol + 4 * p;  // R[p][p-3], R[p][p-2], R[p][p-1], R[p][p]
      const double y = fma(-__ldg(r + 2), y1, fma(-__ldg(r + 1), y2, fma(-__ldg(r), y3, g[p]))) * __ldg(cinv + p);
      g[p] = y;
      y3 = y2, y2 = y1, y1 = y;
    }
    y1 = y2 = y3 = 0.0;  // z[p+1], z[p+2], z[p+3]
    for (int p = nr - 1; p >= 0; --p) {
      double t = g[p];
      if (p + 3 < nr) t = fma(-__ldg(chol + 4 * (p + 3)), y3, t);
      if (p + 2 < nr) t = fma(-__ldg(chol + 4 * (p + 2) + 1), y2, t);
      if (p + 1 < nr) t = fma(-__ldg(chol + 4 * (p + 1) + 2), y1, t);
      t *= __ldg(cinv + p);
      g[p] = t;
      y3 = y2, y2 = y1, y1 = t;
    }
  } else {
    for (int p = 0; p < nr; ++p) {
      const double* r = chol + p * (w + 1);
      double s = g[p];
      for (int j = max(0, w - p); j < w; ++j) s = fma(-__ldg(r + j), g[p - w + j], s);
      g[p] = s * __ldg(cinv + p);
    }
    for (int p = nr - 1; p >= 0; --p) {
      double s = g[p];
      for (int k = p + 1; k <= min(nr - 1, p + w); ++k) s = fma(-__ldg(chol + k * (w + 1) + p - k + w), g[k], s);
      g[p] = s * __ldg(cinv + p);
    }
  }
}

}  // namespace bte
