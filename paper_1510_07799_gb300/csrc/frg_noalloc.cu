// frg_noalloc.cu -- FP64 right-hand side of one parameter point without any
// device allocation (frg_rhs_noalloc in include/frg.h).
//
// Some callers cannot allocate device memory at the moment they need an rhs:
// a latency-critical loop in which an allocation could stall or synchronise the
// device, or a process whose device memory is owned by another component (a
// framework's caching allocator or a fixed memory budget).  For them the whole
// evaluation is one launch whose parameters travel by value and whose workspace
// is the blocks' shared memory (frg_small.cu).  (Measured at N = 16: 14 us a
// call, against 100 us for a chain of seven launches over a device array.)
#include <cuda_runtime.h>

#include <cmath>

#include "../../include/frg.h"
#include "frg_common.cuh"
#include "frg_small.cuh"

using namespace frg;

static_assert(FRG_NOALLOC_MAX_N == SMALL_MAX_N, "the header's limit is the one-launch rhs's");

extern "C" int frg_rhs_noalloc(const frg_params *p, double Lambda, const void *d_gamma, const void *d_sigma,
                               void *d_dgamma, void *d_dsigma, void *cuda_stream) {
  if (!p || !d_gamma || !d_dgamma || !d_dsigma) return FRG_EINVAL;
  const int N = p->N_f;
  if (N < 2 || N > SMALL_MAX_N || (N & 1)) return FRG_EINVAL;
  if (!(p->T > 0.0) || !(p->Delta > 0.0) || !std::isfinite(p->U) || !std::isfinite(p->eps_d) ||
      !std::isfinite(p->T) || !std::isfinite(p->Delta) || !(Lambda > 0.0) || !std::isfinite(Lambda))
    return FRG_EINVAL;
  const int mask = p->channel_mask == 0 ? FRG_CH_ALL : p->channel_mask;
  if (mask < 0 || mask > 0xF) return FRG_EINVAL;
  if (p->cutoff != FRG_CUTOFF_OMEGA && p->cutoff != FRG_CUTOFF_INTERACTION) return FRG_EINVAL;
  PointDesc pd = {};
  pd.N = N;
  pd.n3 = N * N * N;
  pd.cutoff = p->cutoff;
  pd.U = p->U;
  pd.T = p->T;
  pd.et = p->eps_d + 0.5 * p->U;
  pd.Delta = p->Delta;
  RhsIO io = {};
  io.gam = d_gamma;
  io.sig = static_cast<const double2 *>(d_sigma);
  io.dgam = d_dgamma;
  io.dsig = static_cast<double2 *>(d_dsigma);
  io.active = 1;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  bool in_place;
  if (small_sigma(io, N, st, &in_place) != 0 || launch_rhs_small_value(pd, io, Lambda, mask, in_place, st) != 0)
    return FRG_ECUDA;
  return FRG_OK;
}
