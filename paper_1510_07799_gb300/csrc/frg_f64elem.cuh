// frg_f64elem.cuh -- operand elements of the FP64 channel products.
#pragma once
#include "frg_common.cuh"

namespace frg {

// Left[r][k] (r local row, k in [0,K)) of channel CH for transfer geometry g.
template <int CH>
__device__ __forceinline__ double2 left_elem(const PointDesc &P, const void *gam, const Geom &g, int r, int k) {
  const int N = P.N;
  if (CH == CH_PP) {
    const int a = g.row_lo + r, p = g.p_lo + k, s = g.x;
    return cmul(vload<false>(gam, N, P.U, a, s - a, p), P.Lpp[(size_t)s * N + p]);
  } else if (CH == CH_DPH) {
    const int t = g.x, k1 = g.row_lo + r;
    const int half = k >= g.D;
    const int p = g.p_lo + (half ? k - g.D : k);
    const double2 L = P.Lph[(size_t)(-t + N - 1) * N + p];
    const double2 A = vload<false>(gam, N, P.U, k1, p, k1 + t);
    if (!half) {
      const double2 C = vload<false>(gam, N, P.U, k1, p, p - t);
      return cmul(make_double2(2.0 * A.x - C.x, 2.0 * A.y - C.y), L);
    }
    return cmul(make_double2(-A.x, -A.y), L);
  } else {
    const int Q = g.x, k3 = g.row_lo + r, p = g.p_lo + k;
    return cmul(vload<false>(gam, N, P.U, p, k3 + Q, k3), P.Lph[(size_t)(Q + N - 1) * N + p]);
  }
}

template <int CH>
__device__ __forceinline__ double2 right_elem(const PointDesc &P, const void *gam, const Geom &g, int k, int c) {
  const int N = P.N;
  if (CH == CH_PP) {
    const int p = g.p_lo + k, s = g.x;
    return vload<false>(gam, N, P.U, p, s - p, c);
  } else if (CH == CH_DPH) {
    const int t = g.x;
    const int half = k >= g.D;
    const int p = g.p_lo + (half ? k - g.D : k);
    return half ? vload<false>(gam, N, P.U, p - t, c, c - t) : vload<false>(gam, N, P.U, p - t, c, p);
  } else {
    const int Q = g.x, p = g.p_lo + k;
    return vload<false>(gam, N, P.U, c, p + Q, p);
  }
}

}  // namespace frg
