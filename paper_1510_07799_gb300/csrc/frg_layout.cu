// frg_layout.cu -- vertex layouts for the split-precision contraction.
//
// Every operand row of the three channel products is a contiguous run in one
// of four layouts of the FP32 vertex (N = natural [i1][i2][i3],
// W = [i2][i3][i1], X = [i1][i3][i2], and the skewed Z = [i1][i2-i3][i2]),
// each operand read as the entry the channel sum names (no symmetry of the
// vertex is assumed):
//   pp : Left (a, s-a, p)            N   Right (p, s-p, k3)            N
//   dph: A (k1, p, k1+t)             X   B (p-t, k2, p)                X
//        C (k1, p, p-t)              Z   D (p-t, k2, k2-t)             Z
//   xph: Left (p, k3+Q, k3)          W   Right (k1, p+Q, p)            W
// (in Z both direct-channel operands C and D have i2 - i3 = t: C's rows are
// k1, D's rows p - t, both contiguous along i2), and each channel's output
// tile is a run of rows in one layout as well (pp: N, dph: X, xph: W).
// k_relayout writes the natural, W, X and Z copies of a stand-alone evaluation's
// FP64 vertex through layout blocks (frg_lblock.cuh; the split stage kernels
// write the same copies themselves in a flow); k_combine adds the three channel
// outputs into the natural layout through the same blocks.
#include "frg.h"
#include "frg_common.cuh"
#include "frg_layout.cuh"
#include "frg_lblock.cuh"
#include "frg_integrator.cuh"
#include "frg_split.cuh"
#include "frg_combine.cuh"

namespace frg {


// A stand-alone evaluation's vertex (FP64, natural layout) as the FP32 operand
// copies of the contraction: the natural copy (bare U wherever the fourth
// frequency leaves the box) and the W, X and Z copies in `want`, one layout block
// (frg_lblock.cuh) per CTA: whole natural rows in (16-byte loads, all issued
// before the first store), 64-byte row segments of each layout out.  VMAX
// (BF16x3): fold the largest |Re|, |Im| into P.vmax[0].  One pass over the input
// instead of two with an FP32 copy between them: N = 128 20 us against 28 + 13.
template <bool VMAX>
__global__ void __launch_bounds__(LB_THREADS, 5)
    k_relayout(const PointDesc *__restrict__ pt, const double2 *__restrict__ G, int want) {
  extern __shared__ float4 lsm4[];
  chain_wait();
  float2 *sm = reinterpret_cast<float2 *>(lsm4);
  const PointDesc &P = *pt;
  const int N = P.N;
  const LBlock k = lblock(N, N, blockIdx.x);
  if (!k.ok) return;
  const float2 U = make_float2((float)P.U, 0.f);
  // rows (a, b) of n3 elements from g3: pairs of complex values (N is even)
  constexpr int PAIRS = LB * LB * (LC / 2), PER = PAIRS / LB_THREADS;
  double2 v[PER][2];
#pragma unroll
  for (int u = 0; u < PER; ++u) {
    const int e = threadIdx.x + u * LB_THREADS;
    const int c2 = e % (LC / 2), r = e / (LC / 2), b = r % LB, a = r / LB;
    if (a < k.n1 && b < k.n2 && 2 * c2 < k.n3) {
      const double2 *g = G + ((k.g1 + a) * N + (k.g2 + b)) * N + k.g3 + 2 * c2;
      v[u][0] = g[0];
      v[u][1] = g[1];
    }
  }
  float vm = 0.f;
#pragma unroll
  for (int u = 0; u < PER; ++u) {
    const int e = threadIdx.x + u * LB_THREADS;
    const int c2 = e % (LC / 2), r = e / (LC / 2), b = r % LB, a = r / LB;
    if (a < k.n1 && b < k.n2 && 2 * c2 < k.n3) {
      const int i1 = k.g1 + a, i2 = k.g2 + b, i3 = k.g3 + 2 * c2, i4 = i1 + i2 - i3;
      float2 x = round_c64(v[u][0]), y = round_c64(v[u][1]);
      if (VMAX) vm = fmaxf(vm, fmaxf(fmaxf(fabsf(x.x), fabsf(x.y)), fmaxf(fabsf(y.x), fabsf(y.y))));
      if (!inbox(N, i4)) x = U;
      if (!inbox(N, i4 - 1)) y = U;
      const float4 f = make_float4(x.x, x.y, y.x, y.y);
      *reinterpret_cast<float4 *>(P.Y32 + ((i1 * N + i2) * N + i3)) = f;
      *reinterpret_cast<float4 *>(sm + lsidx(a, b, 2 * c2)) = f;
    }
  }
  if (VMAX) {
    vm = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(vm)));
    if ((threadIdx.x & 31) == 0) {
      if (!(vm <= 3.0e38f)) vm = 3.0e38f;
      atomicMax(P.vmax, __float_as_uint(vm));
    }
  }
  __syncthreads();
  lblock_write<false>(P, sm, k, want);
}

// Constant entries of the Z layout: the bare U wherever the third index
// i2 - d + N - 1 or the fourth index i1 + d - (N - 1) of an entry leaves the
// box (the relayout writes every other entry each rhs).  Once per point at
// set-up.
__global__ void k_fill_z(const PointDesc *__restrict__ pts) {
  const PointDesc &P = pts[blockIdx.y];
  if (!P.Y32Z) return;
  const int N = P.N, zrow = 2 * N - 1;
  const size_t total = (size_t)N * zrow * N;
  const float2 u = make_float2((float)P.U, 0.f);
  for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (size_t)gridDim.x * blockDim.x) {
    const int i2 = (int)(e % N);
    const int d = (int)((e / N) % zrow);
    const int i1 = (int)(e / ((size_t)N * zrow));
    const int i3 = i2 - d + N - 1, i4 = i1 + d - (N - 1);
    if (!inbox(N, i3) || !inbox(N, i4)) P.Y32Z[e] = u;
  }
}

template <bool REV, bool ERR, bool OUT64>
__global__ void __launch_bounds__(comb_threads<REV, ERR>(), ERR ? 4 : REV ? LB_MINBLOCKS_WIDE : OUT64 ? LB_MINBLOCKS_OUT : LB_MINBLOCKS)
    k_combine(const PointDesc *__restrict__ pts, const RhsIO *__restrict__ io, int mask, ErrWeights ew) {
  __shared__ __align__(16) float2 sm[LB * LAP];
  chain_wait();
  const RhsIO &o = io[blockIdx.y];
  if (!o.active) return;
  combine_block<REV, ERR, comb_threads<REV, ERR>(), true, OUT64>(pts[blockIdx.y], o, mask, ew, sm);
}

int layout_init() {
  return cudaFuncSetAttribute(k_relayout<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)LB_SMEM) ==
                     cudaSuccess &&
                 cudaFuncSetAttribute(k_relayout<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)LB_SMEM) ==
                     cudaSuccess
             ? 0
             : -3;
}

int launch_relayout(const PointDesc *d_pt, const double2 *gam, int N, int want, bool vmax, cudaStream_t st,
                    bool chain) {
  FRG_COUNT(1);
  return launch_chained(vmax ? k_relayout<true> : k_relayout<false>, lblocks(N, N), LB_THREADS, LB_SMEM, st, chain,
                        d_pt, gam, want) == cudaSuccess
             ? 0
             : -3;
}

int launch_fill_z(const PointDesc *d_pts, int n_points, cudaStream_t st) {
  k_fill_z<<<dim3(512, n_points), 256, 0, st>>>(d_pts);
  FRG_COUNT(1);
  return cudaGetLastError() == cudaSuccess ? 0 : -3;
}

int launch_combine(const PointDesc *d_pts, const RhsIO *d_io, int n_points, int maxN, int mask, cudaStream_t st,
                   bool err, bool canon_half, bool out64, bool chain) {
  const dim3 g(lblocks(maxN, canon_half ? maxN / 2 : maxN), n_points);
  const ErrWeights ew = host_error_weights();
  const bool rev = (mask & FRG_REVERSAL) != 0;
  const int cv = step_carveout(n_points);
  cudaError_t e;
  if (rev && err)
    e = launch_with_carveout(k_combine<true, true, false>, g, comb_threads<true, true>(), 0, st, cv, d_pts, d_io, mask, ew);
  else if (rev && out64)
    e = launch_ex(k_combine<true, false, true>, g, comb_threads<true, false>(), 0, st, cv, chain, d_pts, d_io, mask, ew);
  else if (rev)
    e = launch_with_carveout(k_combine<true, false, false>, g, comb_threads<true, false>(), 0, st, cv, d_pts, d_io, mask, ew);
  else if (err)
    e = launch_with_carveout(k_combine<false, true, false>, g, comb_threads<false, true>(), 0, st, cv, d_pts, d_io, mask, ew);
  else if (out64)
    e = launch_ex(k_combine<false, false, true>, g, comb_threads<false, false>(), 0, st, cv, chain, d_pts, d_io, mask, ew);
  else
    e = launch_with_carveout(k_combine<false, false, false>, g, comb_threads<false, false>(), 0, st, cv, d_pts, d_io,
                             mask, ew);
  FRG_COUNT(1);
  return e == cudaSuccess && cudaGetLastError() == cudaSuccess ? 0 : -3;
}

}  // namespace frg
