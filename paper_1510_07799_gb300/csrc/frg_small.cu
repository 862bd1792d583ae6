// frg_small.cu -- the whole FP64 right-hand side of a small grid in one launch.
//
// On a grid of some 16 frequencies every step of the rhs is latency: propagators,
// bubble tables, three channel products and the self-energy were seven
// dependent launches, and the products ran 32 x 32 tiles of which most was
// padding, on 31 of the 152 SMs (the FP64 units do two multiply-adds per cycle
// and SM, so a padded tile of 16 k takes 16 us).  Here a block takes the entries
// of one k1 and R neighbouring k3, all k2.  It forms the propagators and the
// bubble-weighted operands that its entries share in shared memory,
//   W1[k2][p] = V(k1,k2,p) Lb(p,s-p)                         (pp)
//   Wa[k3][p] = (2 V(k1,p,k3) - V(k1,p,p-t)) Lb(p,p-t), Wb[k3][p] = -V(k1,p,k3) Lb(p,p-t)   (direct)
//   W3[Q][p]  = V(k1,p+Q,p) Lb(p,p+Q)                        (crossed)
// and sums the four products of every entry over the valid p only: no padding,
// no table in memory, one store per entry.  The last blocks form the
// self-energy rhs.  Bound by the FP64 units: 16 multiply-adds per entry and p
// plus the shared weights (their share: rows()).
// Measured (whole call of the allocation-free entry point): N = 16 100 -> 14 us, N =
// 32 183 -> 47, N = 48 353 -> 162, N = 64 572 -> 503 us.
#include <cuda_runtime.h>

#include "frg.h"
#include "frg_common.cuh"
#include "frg_small.cuh"

namespace frg {
namespace small {

constexpr int T = 256;

// k3 per block, and lanes that share an entry's p.  A block's FP64 work is about
// 1.2 + R units (the weights, and R entries per k2), and an SM takes its blocks' work
// one after the other: the smallest R whose blocks still fit the 152 SMs in one go,
// up to N = 36 (more than one block per SM costs N = 18 18.5 against 16.5 us, N = 36 92
// against 77 us), and two or three goes of moderate R above (N = 40 127 us with R = 4,
// 98 with 6, 125 with 14; N = 48 186 with 8, 162 with 16; N = 56 321 with 8, 390 with
// 16).  half: a reversal-symmetric input, the rows k1 < N / 2 and their frequencies.
// (Splitting p further, so that the warps fill the SM's four partitions evenly, gains
// nothing.)
__host__ __device__ inline int rows(int N, bool half) {
  if (half) return N <= 16 ? 1 : N <= 24 ? 2 : 3;
  return N <= 12   ? 1
         : N <= 16 ? 2
         : N <= 20 ? 3
         : N <= 24 ? 4
         : N <= 28 ? 6
         : N <= 32 ? 8
         : N <= 36 ? 9
         : N <= 40 ? 6
         : N <= 48 ? 16
                   : 8;
}
__host__ __device__ inline int lanes(int N, bool half) {
  int l = 16;
  while (l > 1 && N * rows(N, half) * l > T) l >>= 1;
  return l;
}
__host__ __device__ inline int pitch(int N) { return N + 1; }
__host__ __device__ inline int blocks(int N, bool half) {
  const int n = half ? N / 2 : N;
  return n * ((N + rows(N, half) - 1) / rows(N, half)) + (n + T / 32 - 1) / (T / 32);
}
// G, S, B, W1, Wa, Wb, W3
__host__ __device__ inline size_t smem(int N, bool half) {
  const int R = rows(N, half);
  return (size_t)(2 * N + (N + N + 2 * R + N + R - 1) * pitch(N)) * sizeof(double2);
}

// Which part of the rhs a launch covers: everything, or (in-place self-energy) the
// vertex blocks and then the self-energy by one block.
enum Part { ALL, VERTEX, SIGMA };

template <bool HALF>
__device__ __forceinline__ void rhs(const PointDesc &P, const RhsIO &o, double lam, int mask, int part,
                                    int b, double2 *sm) {
  const int N = P.N, R = rows(N, HALF), PL = lanes(N, HALF), W = pitch(N), tid = threadIdx.x;
  const int nb = (N + R - 1) / R, nk = HALF ? N / 2 : N;
  if (b >= (part == VERTEX ? nk * nb : part == SIGMA ? 1 : blocks(N, HALF))) return;
  const double2 *__restrict__ V = static_cast<const double2 *>(o.gam);
  double2 *G = sm, *S = G + N, *B = S + N, *W1 = B + N * W, *Wa = W1 + N * W, *Wb = Wa + R * W, *W3 = Wb + R * W;
  for (int i = tid; i < N; i += T) {
    double2 g, s;
    propagator_at(P, i, lam, o.sig ? o.sig[i] : make_double2(0.0, 0.0), g, s);
    G[i] = g;
    S[i] = s;
  }
  __syncthreads();
  const double sc = P.T * lam;
  if (part == SIGMA || b >= nk * nb) {
    // self-energy: one warp per frequency
    const int lane = tid & 31;
    int w = (part == SIGMA ? 0 : b - nk * nb) * (T / 32) + (tid >> 5);
    for (; w < nk; w += part == SIGMA ? T / 32 : N) {
      double2 acc = make_double2(0.0, 0.0);
      if (mask & FRG_CH_SIGMA)
        for (int p = lane; p < N; p += 32) {
          const double2 a = V[(w * N + p) * N + w], c = V[(w * N + p) * N + p];
          cfma(acc, S[p], make_double2(2.0 * a.x - c.x, 2.0 * a.y - c.y));
        }
      for (int off = 16; off > 0; off >>= 1) {
        acc.x += __shfl_xor_sync(0xffffffffu, acc.x, off);
        acc.y += __shfl_xor_sync(0xffffffffu, acc.y, off);
      }
      if (lane == 0) {
        const double2 v = cscale(acc, sc);
        o.dsig[w] = v;
        if (HALF) o.dsig[N - 1 - w] = make_double2(v.x, -v.y);
      }
    }
    return;
  }
  const int k1 = b / nb, c0 = (b % nb) * R;
  const double2 U = make_double2(P.U, 0.0);
  // every weight below is a bubble Lb(p, q) = Lb(q, p) of two box frequencies
  for (int e = tid; e < N * N; e += T) {
    const int p = e / N, q = e - p * N;
    if (p <= q) B[p * W + q] = B[q * W + p] = cadd(cmul(S[p], G[q]), cmul(G[p], S[q]));
  }
  __syncthreads();
  auto bub = [&](int p, int q) { return B[p * W + q]; };
  if (mask & FRG_CH_PP)
    for (int e = tid; e < N * N; e += T) {
      const int k2 = e / N, p = e - k2 * N, q = k1 + k2 - p;
      if (inbox(N, q)) W1[k2 * W + p] = cmul(V[(k1 * N + k2) * N + p], bub(p, q));
    }
  if (mask & FRG_CH_DPH)
    for (int e = tid; e < R * N; e += T) {
      const int r = e / N, p = e - r * N, k3 = c0 + r, q = p - (k3 - k1);
      if (k3 < N && inbox(N, q)) {
        const double2 L = bub(p, q), A = V[(k1 * N + p) * N + k3], C = V[(k1 * N + p) * N + q];
        Wa[r * W + p] = cmul(make_double2(2.0 * A.x - C.x, 2.0 * A.y - C.y), L);
        Wb[r * W + p] = cmul(make_double2(-A.x, -A.y), L);
      }
    }
  const int Q0 = -(c0 + R - 1);
  if (mask & FRG_CH_XPH)
    for (int e = tid; e < (N + R - 1) * N; e += T) {
      const int d = e / N, p = e - d * N, Q = Q0 + d, q = p + Q;
      if (inbox(N, q))
        W3[d * W + p] = cmul(inbox(N, k1 + Q) ? V[(k1 * N + q) * N + p] : U, bub(p, q));
    }
  __syncthreads();
  const int l = tid & (PL - 1), ne = N * R, step = T / PL;
  double2 *out = static_cast<double2 *>(o.dgam);
  for (int eb = 0; eb < ne; eb += step) {  // (the same trips in every thread: the fold below is warp-wide)
    const int e = eb + tid / PL, k2 = e / R, r = e - k2 * R, k3 = c0 + r;
    const bool on = e < ne && k3 < N;
    const int s = k1 + k2, t = k3 - k1, Q = k2 - k3, k4 = s - k3;
    const bool in4 = inbox(N, k4);
    double2 pp = make_double2(0.0, 0.0), dd = pp, xx = pp;
    if (on && (mask & FRG_CH_PP)) {
      const double2 *w = W1 + k2 * W;
      const int hi = min(N - 1, s);
#pragma unroll 4
      for (int p = max(0, s - (N - 1)) + l; p <= hi; p += PL)
        cfma(pp, w[p], in4 ? V[(p * N + s - p) * N + k3] : U);
    }
    if (on && (mask & FRG_CH_DPH)) {
      const double2 *wa = Wa + r * W, *wb = Wb + r * W;
      const int hi = min(N - 1, N - 1 + t);
#pragma unroll 2
      for (int p = max(0, t) + l; p <= hi; p += PL) {
        const int row = ((p - t) * N + k2) * N;
        cfma(dd, wa[p], in4 ? V[row + p] : U);
        cfma(dd, wb[p], in4 ? V[row + k4] : U);
      }
    }
    if (on && (mask & FRG_CH_XPH)) {
      const double2 *w = W3 + (Q - Q0) * W;
      const int hi = min(N - 1, N - 1 - Q);
#pragma unroll 4
      for (int p = max(0, -Q) + l; p <= hi; p += PL) cfma(xx, w[p], V[(p * N + k2) * N + k3]);
      // a non-finite sum again with the weight on the other factor, as the tiled
      // products have it (which of infinity and NaN an infinite entry gives
      // depends on that)
      if (!isfinite(xx.x) || !isfinite(xx.y)) {
        xx = make_double2(0.0, 0.0);
        for (int p = max(0, -Q) + l; p <= hi; p += PL)
          cfma(xx, cmul(V[(p * N + k2) * N + k3], bub(p, p + Q)), in4 ? V[(k1 * N + p + Q) * N + p] : U);
      }
    }
    double2 v = cadd(cadd(cscale(pp, -sc), cscale(dd, sc)), cscale(xx, -sc));
    for (int off = PL >> 1; off > 0; off >>= 1) {
      v.x += __shfl_xor_sync(0xffffffffu, v.x, off);
      v.y += __shfl_xor_sync(0xffffffffu, v.y, off);
    }
    if (on && l == 0) {
      const int at = (k1 * N + k2) * N + k3;
      out[at] = v;
      if (HALF) out[N * N * N - 1 - at] = make_double2(v.x, -v.y);
    }
  }
}

template <bool HALF>
__global__ void __launch_bounds__(T) k_rhs_small(const PointDesc *__restrict__ pts, const RhsIO *__restrict__ io,
                                                 int n_below, int mask, int part) {
  extern __shared__ double2 sm[];
  chain_wait();
  const PointDesc &P = pts[blockIdx.y];
  const RhsIO &o = io[blockIdx.y];
  if (!o.active || P.N >= n_below) return;
  rhs<HALF>(P, o, *o.lam, mask, part, blockIdx.x, sm);
}

__global__ void __launch_bounds__(T) k_rhs_small_value(const __grid_constant__ PointDesc P,
                                                       const __grid_constant__ RhsIO o, double lam, int mask,
                                                       int part) {
  extern __shared__ double2 sm[];
  rhs<false>(P, o, lam, mask, part, blockIdx.x, sm);
}

// (A host-side setting of the current device's context: set on every call, as the
// context may have changed, and always to the most any size needs, as another thread
// may be between its setting and its launch.)
template <typename K>
bool room(K kernel, size_t bytes) {
  if (bytes <= 48 * 1024) return true;
  size_t most = 0;
  for (int n = 2; n <= SMALL_MAX_N; n += 2) most = smem(n, false) > most ? smem(n, false) : most;
  return bytes <= most &&
         cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most) == cudaSuccess;
}
}  // namespace small

// (in order with an input that overlaps the copy)
__global__ void k_move_sigma(double2 *dst, const double2 *src, int N) {
  const int t = threadIdx.x;
  double2 v;
  if (t < N) v = src[t];
  __syncthreads();
  if (t < N) dst[t] = v;
}

int small_sigma(RhsIO &o, int N, cudaStream_t st, bool *in_place) {
  const auto overlap = [&](const void *p, size_t n) {
    const char *a = reinterpret_cast<const char *>(o.sig), *b = static_cast<const char *>(p);
    return a && a < b + n * sizeof(double2) && b < a + N * sizeof(double2);
  };
  *in_place = overlap(o.dsig, N);
  if (!overlap(o.dgam, (size_t)N * N * N)) return 0;
  k_move_sigma<<<1, SMALL_MAX_N, 0, st>>>(o.dsig, o.sig, N);
  FRG_COUNT(1);
  o.sig = o.dsig;
  *in_place = true;
  return cudaGetLastError() == cudaSuccess ? 0 : -3;
}

int launch_rhs_small(const PointDesc *d_pts, const RhsIO *d_io, int n_points, int maxN, int n_below, int mask,
                     bool sig_in_place, cudaStream_t st, bool chain, bool half) {
  // shared memory and blocks for every size below the bound (both drop where the
  // rows per block step up)
  const int N = maxN < n_below ? maxN : n_below - 1;
  size_t bytes = 0;
  int blocks = 0;
  for (int n = 2; n <= N; n += 2) {
    bytes = small::smem(n, half) > bytes ? small::smem(n, half) : bytes;
    blocks = small::blocks(n, half) > blocks ? small::blocks(n, half) : blocks;
  }
  const auto kernel = half ? small::k_rhs_small<true> : small::k_rhs_small<false>;
  if (!small::room(kernel, bytes)) return -3;
  const int first = sig_in_place ? small::VERTEX : small::ALL;
  if (launch_chained(kernel, dim3(blocks, n_points), small::T, bytes, st, chain, d_pts, d_io, n_below, mask,
                     first) != cudaSuccess)
    return -3;
  FRG_COUNT(1);
  if (sig_in_place) {
    if (launch_chained(kernel, dim3(1, n_points), small::T, bytes, st, chain, d_pts, d_io, n_below, mask,
                       (int)small::SIGMA) != cudaSuccess)
      return -3;
    FRG_COUNT(1);
  }
  return cudaGetLastError() == cudaSuccess ? 0 : -3;
}

int launch_rhs_small_value(const PointDesc &P, const RhsIO &o, double lam, int mask, bool sig_in_place,
                           cudaStream_t st) {
  const size_t bytes = small::smem(P.N, false);
  if (!small::room(small::k_rhs_small_value, bytes)) return -3;
  const int first = sig_in_place ? small::VERTEX : small::ALL;
  small::k_rhs_small_value<<<small::blocks(P.N, false), small::T, bytes, st>>>(P, o, lam, mask, first);
  FRG_COUNT(1);
  if (sig_in_place) {
    small::k_rhs_small_value<<<1, small::T, bytes, st>>>(P, o, lam, mask, small::SIGMA);
    FRG_COUNT(1);
  }
  return cudaGetLastError() == cudaSuccess ? 0 : -3;
}

}  // namespace frg
