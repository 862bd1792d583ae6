// frg_x64.cu -- FP64 channel products on the sm_103a tensor cores by exact
// slicing (the error-free splitting of Ozaki, Ogita, Oishi and Rump, Numer.
// Algorithms 59, 2012, with a fixed-point grid per operand line).
//
// This part's FP64 units run at 1/58 of FP32 (1.2 TFLOP/s measured); the FP16
// tensor cores add integers exactly.  For a channel and transfer the product
//   Out[r][c] = sum_k Left[r][k] Right[k][c]        (index sets: frg_common.cuh)
// is formed as follows.
//  * Every line (a row of the bubble-weighted left operand, a column of the
//    right one) gets one exponent e with |x| < 0.993 2^e over the line, and its
//    values become integers X = rint(x 2^(63 - e)).  A value within 2^10 of its
//    line's bound converts exactly, a smaller one to 2^(e - 64).
//  * X is cut into eight digits of base 256 in [-128, 127] (one 64-bit add of
//    128 in every byte, done when X is stored, makes its bytes the digits + 128),
//    each an exact FP16 value.
//  * Digit products i + j = g <= 7 (i, j counted from the leading digit) of all
//    k go to accumulator g: 36 products, each an integer of at most 2^14.  An FP32
//    accumulator holds every integer up to 2^24, so the accumulators are drained
//    every CHUNK = 4 k-steps: 8 pairs of digits x 128 real terms x 2^14 = 2^24.
//    (With one drain per product, as of 16 or more k-steps, lines whose digits all
//    add up lose units of 2^-32 of the lines' bounds: 4e-9 of the entry at N = 256.)
//    The products left out (i + j >= 8) are below 2^-61 of the bounds per term.
//  * The epilogue adds the accumulators as 64-bit integers and rounds the sum
//    once to FP64.
// So an entry is off by some 2^-60 of the bounds B = 2^(eL + eR) of its two lines,
// where a chain of FP64 multiply-adds is off by 2^-53 of sum |L_k| |R_k| at least.
// The sum of an entry whose terms may all be small against B (a column with values
// more than six binary orders apart and a small result) is formed again term by term in
// FP64, and so is that of a line that has no fixed point (non-finite values, exponents
// beyond 2^+-400): settle.  (Errors against extended precision: tests/test_gpu_x64.py
// over the vertex, tests/test_gpu_x64_bounds.py per entry at the limits.)
//
// Three launches per rhs: k_x64_panels gathers, weights and converts the
// operands into blocks of 16 k x 64 lines; k_x64_products multiplies them
// (persistent CTAs over a longest-first tile schedule); k_x64_combine sums the
// channels into the natural layout.
// Measured, one rhs (all channels): N = 128 6086 -> 398 us, N = 64 674 -> 64 us
// (CUDA cores -> slices).  The eighth digit, the drains and the wider sums are 77 and 4
// us of it, against seven digits drained once per product.
#include <cuda_runtime.h>

#include <algorithm>
#include <vector>

#include "frg.h"
#include "frg_common.cuh"
#include "frg_f64elem.cuh"
#include "frg_ptx.cuh"
#include "frg_sched.cuh"
#include "frg_x64.cuh"

namespace frg {
namespace x64 {
using namespace tc;

constexpr int SL = 8;                       // digits per value
constexpr int NACC = 8;                     // accumulators: digit products i + j = 0 .. 7
constexpr int LINES = 64;                   // lines of an operand block (rows or columns of a tile)
constexpr int KS = 16;                      // complex k per block
constexpr int BLK = LINES * KS;             // elements (re, im) of a block: 16 KB
constexpr int BLK_BYTES = BLK * 16;
constexpr int FIX = 63;                     // fixed-point position: X = x 2^(FIX - e)
constexpr unsigned long long BIAS = 0x8080808080808080ull;  // 128 in each of the eight digit bytes
constexpr int E_LIM = 400;                  // line exponents the path accepts
// k-steps between two drains of the accumulators.  A digit product is at most 2^14,
// a k-step adds 2 KS of them per digit pair, an accumulator has up to NACC pairs: no
// partial sum passes 2^24, up to which FP32 holds every integer.
constexpr int CHUNK = 4;
static_assert((long)NACC * CHUNK * 2 * KS * 128 * 128 <= 1l << 24, "the accumulators' sums are exact integers");
// A line's record: 4096 e + 4 v + UNSLICED (non-finite values, or an exponent beyond
// E_LIM).  |x| < 0.993 2^e over the line.  v of a row: the sum of its |Re| and |Im| is
// below 2^(e + v); of a column: its number of small values, below 2^(e - EVEN - 1).
constexpr int UNSLICED = 1;
constexpr unsigned EVEN = 6;
constexpr int SUM_MAX = 10;  // largest v of a row
__host__ __device__ constexpr int rec_exp(int r) { return r >> 12; }
__host__ __device__ constexpr int rec_val(int r) { return r >> 2 & 1023; }

// -------------------------------------------------------------- panels ----
// One block: eight lines of one operand of one product over its whole
// contraction range.  Eight lanes take the eight lines at one k, so that the
// blocks are written in 128-byte segments; a thread gathers (and weights, with the
// table that carries T Lambda) all its k of one line into registers, the block
// finds each line's largest magnitude, and the values leave in fixed point.
// Bound by the FP64 multiplications of the weights and by the gathers (16-byte
// elements, one 32-byte sector each wherever the line and the contraction index
// both stride through the vertex): 110 us at N = 128 for 302 MB
// written and 15 M entries gathered, 11 us of it the line records (before them 99 us,
// and 159 us with the lines staged in shared memory between the gather and the
// conversion).  (The two operands as launches of their own, the right one beside the
// bubble weights: 130 us, the left one alone takes as long as both at N = 64.)
constexpr int PAN_LINES = 8;
// k per thread and range: eight on the larger grids (more gathers in flight: N =
// 128 99 against 111 us), four on the smaller ones (more warps: N = 64 18.0
// against 19.3 us; 16.8 with the weights' factor in the table).
static int panel_u(int maxN) { return maxN > 80 ? 8 : 4; }
// Elements along the contraction axis: one or two (direct channel) ranges of D
// padded to whole blocks.
__host__ __device__ inline int d16(int D) { return (D + KS - 1) / KS * KS; }
// Threads of a block: eight per k, and at most U k each (8 / U threads per k of the
// padded range, in whole warps).
static int panel_threads(int maxN) { return std::max(64, (d16(maxN) * (PAN_LINES / panel_u(maxN)) + 31) / 32 * 32); }

__device__ __forceinline__ unsigned mag(double2 v) {
  const unsigned a = (unsigned)__double2hiint(v.x) & 0x7fffffffu, b = (unsigned)__double2hiint(v.y) & 0x7fffffffu;
  return a > b ? a : b;
}
// Exponent of a line whose largest high word (sign cleared) is m: |x| < 0.993 2^e.
__device__ __forceinline__ int line_exp(unsigned m) {
  if (m == 0u) return 0;
  const int E = (int)(m >> 20);
  return (E ? E : 1) - 1022 + ((m & 0xfffffu) >= 0xfc000u ? 1 : 0);
}
// rint(x 2^(FIX - e)) + BIAS (ties away from zero), for |x| < 0.993 2^e, e >= -E_LIM.
// top: the upper word of the magnitude.
__device__ __forceinline__ unsigned long long to_fixed(double x, int e, unsigned &top) {
  const int h = __double2hiint(x);
  const int E = (h >> 20) & 0x7ff;
  // the 53-bit significand, eleven bits up, then right to one bit below the fixed
  // point (zero and denormals, whose implicit bit is set wrongly here, shift out)
  const unsigned long long m = (unsigned long long)((unsigned)h & 0xfffffu | 0x100000u) << 32 | (unsigned)__double2loint(x);
  const int sh = e + 1022 - E;
  const unsigned long long r = sh > 63 ? 0ull : (((m << 11) >> sh) + 1ull) >> 1;
  const unsigned long long s = (unsigned long long)(long long)(h >> 31);  // all ones for x < 0
  top = (unsigned)(r >> 32);
  return (r ^ s) + (BIAS - s);
}

// The vertex entries of one element: the pp and crossed operands and the direct
// channel's A and C (left) or B and D (right).
template <int CH, bool LEFT>
__device__ __forceinline__ void gather(const PointDesc &P, const double2 *__restrict__ V, const Geom &g, int line,
                                       int k, double2 &v, double2 &v2) {
  const int N = P.N, p = g.p_lo + k;
  auto at = [&](int i1, int i2, int i3) { return V[(i1 * N + i2) * N + i3]; };
  if (LEFT) {
    // every index is in the box for valid rows and k
    const int r = g.row_lo + line;
    if (CH == CH_PP) {
      v = at(r, g.x - r, p);
    } else if (CH == CH_DPH) {
      v = at(r, p, r + g.x);
      v2 = at(r, p, p - g.x);
    } else {
      v = at(p, r + g.x, r);
    }
  } else {
    const int c = line;
    const double2 U = make_double2(P.U, 0.0);
    if (CH == CH_PP) {
      v = inbox(N, g.x - c) ? at(p, g.x - p, c) : U;
    } else if (CH == CH_DPH) {
      // the fourth index of B and the third of D are both c - t
      const bool in = inbox(N, c - g.x);
      v = in ? at(p - g.x, c, p) : U;
      v2 = in ? at(p - g.x, c, c - g.x) : U;
    } else {
      v = inbox(N, c + g.x) ? at(c, p + g.x, p) : U;
    }
  }
}

template <int CH, bool LEFT, int U>
__device__ __forceinline__ void panel(const PointDesc &P, const RhsIO &o, const X64Pt &x, int m, int oct,
                                      double2 *sw, unsigned *smax, unsigned *ssum) {
  const int N = P.N;
  const Geom g = geom(CH, N, m);
  const int D = g.D, D16 = d16(D), nk = (CH == CH_DPH ? 2 : 1) * (D16 / KS);
  const int line0 = oct * PAN_LINES, nl = min(PAN_LINES, (LEFT ? D : N) - line0);
  if (nl <= 0) return;
  const int tid = threadIdx.x, line = tid & 7, kstep = blockDim.x >> 3;
  const double2 *__restrict__ V = static_cast<const double2 *>(o.gam);
  if (tid < PAN_LINES) {
    smax[tid] = 0u;
    ssum[tid] = 0u;
  }
  if (LEFT) {
    const double2 *L = CH == CH_PP ? P.LppS + (size_t)m * N : P.LphS + (size_t)(CH == CH_DPH ? 2 * N - 2 - m : m) * N;
    for (int k = tid; k < D; k += blockDim.x) sw[k] = L[g.p_lo + k];
  }
  double2 v[U], v2[U];
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const int k = (tid >> 3) + u * kstep;
    v[u] = v2[u] = make_double2(0.0, 0.0);
    if (k < D && line < nl) gather<CH, LEFT>(P, V, g, line0 + line, k, v[u], v2[u]);
  }
  const uint4 pr = x.prod[(size_t)CH * (2 * N - 1) + m];
  __syncthreads();
  unsigned um = 0u;
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const int k = (tid >> 3) + u * kstep;
    if (LEFT && k < D) {
      const double2 w = sw[k];
      if (CH == CH_DPH) {
        const double2 A = v[u], C = v2[u];
        v[u] = cmul(make_double2(fma(2.0, A.x, -C.x), fma(2.0, A.y, -C.y)), w);
        v2[u] = cmul(make_double2(-A.x, -A.y), w);
      } else {
        v[u] = cmul(make_double2(-v[u].x, -v[u].y), w);
      }
    }
    um = max(um, mag(v[u]));
    if (CH == CH_DPH) um = max(um, mag(v2[u]));
  }
  um = max(um, __shfl_xor_sync(0xffffffffu, um, 8));
  um = max(um, __shfl_xor_sync(0xffffffffu, um, 16));
  if ((tid & 31) < PAN_LINES) atomicMax(&smax[line], um);
  __syncthreads();
  const int tile = line0 / LINES, l0 = (line0 & (LINES - 1)) + line;
  const unsigned mx = smax[line];
  int e = line_exp(mx);
  const int bad = (mx >> 20) == 0x7ffu || e > E_LIM || e < -E_LIM ? UNSLICED : 0;
  e = max(-E_LIM, min(E_LIM, e));  // (an unsliced line's products are not used)
  ulonglong2 *dst = (LEFT ? x.L + (size_t)(pr.x + tile * nk) * BLK : x.R + (size_t)(pr.y + tile * nk) * BLK) + l0;
  unsigned sum = 0u;
  if (line < nl) {
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int k = (tid >> 3) + u * kstep;
      if (k >= D16) break;
      unsigned a, b;
      const unsigned long long re = to_fixed(v[u].x, e, a), im = to_fixed(v[u].y, e, b);
      dst[(size_t)k * LINES] = make_ulonglong2(re, im);
      if (k < D) sum += LEFT ? (a >> 22) + (b >> 22) + 2u : (a | b) >> (30 - EVEN) == 0u;
      if (CH == CH_DPH) {
        const unsigned long long re2 = to_fixed(v2[u].x, e, a), im2 = to_fixed(v2[u].y, e, b);
        dst[(size_t)(D16 + k) * LINES] = make_ulonglong2(re2, im2);
        if (k < D) sum += LEFT ? (a >> 22) + (b >> 22) + 2u : (a | b) >> (30 - EVEN) == 0u;
      }
    }
  }
  sum += __shfl_xor_sync(0xffffffffu, sum, 8);
  sum += __shfl_xor_sync(0xffffffffu, sum, 16);
  if ((tid & 31) < PAN_LINES) atomicAdd(&ssum[line], sum);
  __syncthreads();
  if (tid < nl) {
    const int n = (int)ssum[line];
    // (a row's sum is below 2^(its bits) / 2^9, and 1024 values below 0.993 stay below 2^10)
    if (LEFT)
      x.eL[(size_t)(pr.z + tile) * LINES + l0] = 4096 * e + 4 * min(SUM_MAX, max(0, 32 - __clz(n) - 9)) + bad;
    else
      x.eR[(size_t)(pr.w + tile) * LINES + l0] = 4096 * e + 4 * n + bad;
  }
}

// grid: (line octets of the left, then of the right operand; transfers;
// point x channel)
template <int U>
__global__ void __launch_bounds__(FRG_MAX_N *PAN_LINES / U, U == 8 ? 3 : 2)
    k_x64_panels(const PointDesc *__restrict__ pts, const RhsIO *__restrict__ io, const X64Pt *__restrict__ xp, int p0,
                 int chmask, int rev) {
  __shared__ double2 sw[FRG_MAX_N];
  __shared__ unsigned smax[PAN_LINES], ssum[PAN_LINES];
  chain_wait();
  // the direct channel's blocks first, and each channel's largest transfers (m =
  // N - 1 and outwards) first: the light blocks fill in at the end
  const int pi = p0 + blockIdx.z / 3, z = blockIdx.z % 3, ch = z == 0 ? CH_DPH : z == 1 ? CH_PP : CH_XPH;
  const RhsIO &o = io[pi];
  const X64Pt &x = xp[pi];
  if (!o.active || !x.prod || !(chmask >> ch & 1)) return;
  const PointDesc &P = pts[pi];
  const int half = gridDim.x / 2, y = blockIdx.y;
  if (y >= (rev ? P.N : 2 * P.N - 1)) return;
  const int m = rev ? P.N - 1 - y : P.N - 1 + (y & 1 ? (y + 1) / 2 : -(y / 2));
  const int b = blockIdx.x;
  if (b < half) {
    if (ch == CH_PP)
      panel<CH_PP, true, U>(P, o, x, m, b, sw, smax, ssum);
    else if (ch == CH_DPH)
      panel<CH_DPH, true, U>(P, o, x, m, b, sw, smax, ssum);
    else
      panel<CH_XPH, true, U>(P, o, x, m, b, sw, smax, ssum);
  } else {
    if (ch == CH_PP)
      panel<CH_PP, false, U>(P, o, x, m, b - half, sw, smax, ssum);
    else if (ch == CH_DPH)
      panel<CH_DPH, false, U>(P, o, x, m, b - half, sw, smax, ssum);
    else
      panel<CH_XPH, false, U>(P, o, x, m, b - half, sw, smax, ssum);
  }
}

// ------------------------------------------------------------ products ----
// A tile is 64 complex rows x 64 complex columns of one product, taken in chunks of
// CHUNK k-steps.  Real form of
// the complex product on the left operand: accumulator rows 0-63 hold Re,
// rows 64-127 Im of the product, from A = [Re a; Im a] against Re b and
// A = [-Im a; Re a] against Im b, so three planes of the left digits are kept.
// Accumulator g (digit weight 256^-g) takes the 64 columns from 64 g on (eight
// fill TMEM), and the B digits of one k-step lie one after the other, so that
// one instruction multiplies digit i of A with several consecutive digits of B:
// N up to 256.
// Roles: warps 0-15 epilogue, 16 MMA issue, 17 loader (bulk copies, two blocks
// per k-step), 18-25 transform (fixed-point values -> FP16 digit tiles).
// Bound by shared memory during the k-steps (3130 cycles each at N = 128: the tensor
// cores' operand reads alone are 243 KB, 1900 cycles at 128 B, beside 80 KB of digit
// tiles and 32 KB of blocks in and out; 2304 cycles of products) and by the drains between
// them (5000 cycles each, 4400 of them the additions of 16 warps, 16 columns each, which
// keep the sums in registers).  Rounding and storing run beside the next tile's products.
// N = 128 254 us, N = 64 34 us.
constexpr int EPI_W = 16, MMA_W = 16, LOAD_W = 17, XF_W0 = 18, N_XF = 8;
constexpr int THREADS = 32 * (XF_W0 + N_XF);
constexpr int NRAW = 3, NOP = 2;  // raw slots of one block; operand stages
static_assert(NRAW == 3, "the phases of the raw slots' barriers (k_x64_products)");
// Operand tiles, K-major without swizzle: core matrices of 8 lines x 16 bytes.
// A: [digit][k half][plane -Im, Re, Im][8 line groups][8 lines][16 B]
// B: [plane Re, Im][k half][digit][8 line groups][8 lines][16 B]
constexpr int PLANE = 1024;
constexpr int A_KC = 3 * PLANE, A_DIG = 2 * A_KC, A_BYTES = SL * A_DIG;
constexpr int B_KC = SL * PLANE, B_PL = 2 * B_KC, B_BYTES = 2 * B_PL;
constexpr int OP_STAGE = A_BYTES + B_BYTES;
constexpr int EPI_CPW = 64 / (EPI_W / 4);    // columns per epilogue warp
constexpr int EPI_COLS = 4;
constexpr int EPI_BUF = 32 * EPI_COLS * 16;  // one warp pair's 32 rows x 4 columns
constexpr int SMEM = 1024 + NOP * OP_STAGE + NRAW * BLK_BYTES + EPI_W / 2 * EPI_BUF + 256;
static_assert(2 * KS * LINES * 16 <= NOP * OP_STAGE && KS * LINES == 2 * 32 * EPI_W, "settle_tile");
static_assert(SMEM <= 232448, "shared memory budget");

// One tile, with what every role needs to start on it without a chain of
// dependent loads: its k-steps, where its operand blocks and line exponents start.
struct __align__(16) Work {
  int point;
  short m, ch, rt, ct;
  int nk;
  unsigned bl, br, el, er;  // first left and right block, left and right tile of exponents
};

// Shared-memory matrix descriptor, K-major, no swizzle: lbo between the two
// 16-byte columns of K, sbo between groups of eight lines.
__device__ __forceinline__ uint64_t desc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
  return (uint64_t)((addr & 0x3FFFFu) >> 4) | (uint64_t)(lbo >> 4) << 16 | (uint64_t)(sbo >> 4) << 32 | 1ull << 46;
}
// D f32, A and B f16, K-major, M = 128, N = n.
__host__ __device__ constexpr uint32_t idesc(int n) {
  return (1u << 4) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
}
__device__ __forceinline__ void bulk_copy(void *dst, const void *src, uint32_t bytes, uint64_t *bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   smem_u32(dst)),
               "l"(src), "r"(bytes), "r"(smem_u32(bar))
               : "memory");
}

// The epilogue warps' own barrier.
__device__ __forceinline__ void epi_sync() {
  asm volatile("bar.sync %0, %1;" ::"n"(1 + EPI_W / 2), "n"(32 * EPI_W) : "memory");
}
// Whether a predicate holds in both warps of an epilogue pair.
__device__ __forceinline__ bool pair_all(bool v, int pair) {
  uint32_t r;
  asm volatile(
      "{\n .reg .pred p, q;\n setp.ne.b32 p, %1, 0;\n bar.red.and.pred q, %2, 64, p;\n selp.b32 %0, 1, 0, q;\n}\n"
      : "=r"(r)
      : "r"((uint32_t)v), "r"(1 + pair)
      : "memory");
  return r != 0;
}

// What the roles read first on the CTA's next tiles, brought into the L1 cache one
// tile ahead by the loader's idle lanes (plain loads whose values nothing waits
// for).
__device__ __forceinline__ void touch(const void *p) {
  uint32_t v;
  asm volatile("ld.global.ca.u32 %0, [%1];" : "=r"(v) : "l"(p));
}
__device__ __forceinline__ void look_ahead(const PointDesc *__restrict__ pts, const RhsIO *__restrict__ io,
                                           const X64Pt *__restrict__ xp, const Work *__restrict__ work, int wi, int w1,
                                           int lane) {
  if (wi + 1 < w1) {
    const Work n = work[wi + 1];
    if (lane == 1) touch(&io[n.point].active);
    if (lane == 2) touch(&pts[n.point].N);
    if (lane == 3) touch(&xp[n.point].L);
    if (lane == 4) touch(&xp[n.point].PX);
  }
  if (wi + 2 < w1 && lane == 5) touch(work + wi + 2);
}

// Digit I of two values as a pair of FP16: 1024 + (digit + 128), less 1152.
__device__ __forceinline__ uint32_t sub2(uint32_t a, uint32_t b) {
  uint32_t r;
  asm("sub.rn.f16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
  return r;
}
constexpr uint32_t C1152 = 0x64806480u;  // (1152, 1152): 1024 + 128
template <int I>
__device__ __forceinline__ uint32_t biased(uint2 a, uint2 b) {
  constexpr uint32_t y = 3 - (I & 3);  // byte of the high (digits 0-3) or the low word
  const uint32_t p = I < 4 ? a.y : a.x, q = I < 4 ? b.y : b.x;
  return (__byte_perm(p, q, y | y << 4 | (4 + y) << 8 | (4 + y) << 12) & 0x00ff00ffu) | 0x64006400u;
}
// Digit I of the eight values of one line: Re, Im and (left operand) -Im.
template <int I, bool LEFT>
__device__ __forceinline__ void store_digit(uint8_t *dst, const uint4 (&v)[8]) {
  uint4 re, im, ni;
  uint32_t *r = &re.x, *i = &im.x, *n = &ni.x;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const uint4 a = v[2 * q], b = v[2 * q + 1];
    const uint32_t br = biased<I>(make_uint2(a.x, a.y), make_uint2(b.x, b.y));
    const uint32_t bi = biased<I>(make_uint2(a.z, a.w), make_uint2(b.z, b.w));
    r[q] = sub2(br, C1152);
    i[q] = sub2(bi, C1152);
    if (LEFT) n[q] = sub2(C1152, bi);
  }
  if (LEFT) {
    uint8_t *p = dst + I * A_DIG;
    *reinterpret_cast<uint4 *>(p) = ni;
    *reinterpret_cast<uint4 *>(p + PLANE) = re;
    *reinterpret_cast<uint4 *>(p + 2 * PLANE) = im;
  } else {
    uint8_t *p = dst + I * PLANE;
    *reinterpret_cast<uint4 *>(p) = re;
    *reinterpret_cast<uint4 *>(p + B_PL) = im;
  }
}
template <bool LEFT>
__device__ __forceinline__ void store_digits(uint8_t *dst, const uint4 (&v)[8]) {
  store_digit<0, LEFT>(dst, v);
  store_digit<1, LEFT>(dst, v);
  store_digit<2, LEFT>(dst, v);
  store_digit<3, LEFT>(dst, v);
  store_digit<4, LEFT>(dst, v);
  store_digit<5, LEFT>(dst, v);
  store_digit<6, LEFT>(dst, v);
  store_digit<7, LEFT>(dst, v);
}

// (Two columns at a time: four spill beside the sums, 453 against 405 us per rhs at N =
// 128; one at a time with the next one's loads ahead 410 us.)
__device__ __forceinline__ void tmem_ld2(uint32_t taddr, float (&v)[2]) {
  uint32_t r[2];
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x2.b32 {%0, %1}, [%2];" : "=r"(r[0]), "=r"(r[1]) : "r"(taddr));
  v[0] = __uint_as_float(r[0]);
  v[1] = __uint_as_float(r[1]);
}
// Adds the accumulators of one chunk (integers, accumulator g at most (g + 1) 2^21) to
// an entry's sum of the X_L X_R, in units of 2^(65 + l).  In FP32, whose additions run
// at one per issue slot here, where integer shifts and products take two and
// conversions eight (a join by conversions: 80 slots per entry, this one 42): the terms
// y_g = a_g 2^(49 - 8 g) go to three limbs, multiples of 2^(43 + l), of 2^(23 + l) and of
// 2^(2 + l).  Adding to m = 1.5 x 2^23 grids rounds to the grid, what is left over is exact
// (y_g has 24 bits) and goes to the next limb, and the bits of the sums are the limbs'
// integers, added modulo 2^64 (m's own bits leave with the initial value of s).
// The sums of a limb may reach a third of its m, 2^22 of its grid:
//  * upper: with the row's sum of |x| / 2^e below 2^l, |y_0| < 2^(64.01 + l) (a leading
//    digit is at most 2.01 x 128 |x|), and the chunk keeps |y_1| <= 2^63, |y_2| < 2^56 and
//    |y_3| <= 2^48: below 2^(64.6 + l), of 2^(65 + l);
//  * middle: four remainders of at most 2^(42 + l), y_4 to y_6 below 2^41 each, of 2^(45 +
//    l); the remainders of y_0 to y_2 are multiples of 2^33, on the grid for l <= 10;
//  * lower: four remainders of at most 2^(22 + l), of 2^(24 + l); rounded to the grid.
__host__ __device__ constexpr unsigned limb_bits(int grid) { return (unsigned)(127 + 23 + grid) << 23 | 0x400000u; }
struct Limbs {
  float t, u, z;
};
__device__ __forceinline__ Limbs limbs_of(int l) {
  return Limbs{__uint_as_float(limb_bits(43 + l)), __uint_as_float(limb_bits(23 + l)), __uint_as_float(limb_bits(2 + l))};
}
__device__ __forceinline__ unsigned long long limbs_sum(float t, float u, float z) {
  return ((unsigned long long)__float_as_uint(t) << 41) + ((unsigned long long)__float_as_uint(u) << 21) +
         __float_as_uint(z);
}
// Adds y to the limb's sum m and returns what is left over.
__device__ __forceinline__ float limb_add(float &m, float a, float w) {
  const float n = fmaf(a, w, m), r = fmaf(a, w, m - n);
  m = n;
  return r;
}
__device__ __forceinline__ void add_chunk(unsigned long long &s, const float (&d)[NACC][2], int c, const Limbs &m) {
  auto w = [](int e) { return e >= 0 ? (float)(1ll << e) : 1.f / (float)(1ll << -e); };
  float t = m.t, u = m.u;
  const float r0 = limb_add(t, d[0][c], w(49)), r1 = limb_add(t, d[1][c], w(41)), r2 = limb_add(t, d[2][c], w(33)),
              r3 = limb_add(t, d[3][c], w(25));
  u += r0;
  u += r1;
  u += r2;
  const float v3 = limb_add(u, r3, 1.f), v4 = limb_add(u, d[4][c], w(17)), v5 = limb_add(u, d[5][c], w(9)),
              v6 = limb_add(u, fmaf(d[7][c], w(-8), d[6][c]), w(1));
  const float z = m.z + v3 + v4 + v5 + v6;
  s += limbs_sum(t, u, z);
}
// s 2^e as FP64, rounded once, on the integer pipe (e within +-900: normal).
__device__ __forceinline__ double scaled(long long s, int e) {
  const unsigned sg = (unsigned)(s >> 32) & 0x80000000u;
  const unsigned long long a = s < 0 ? 0ull - (unsigned long long)s : (unsigned long long)s;
  unsigned h = (unsigned)(a >> 32), l = (unsigned)a;
  if (h == 0u) {  // a cancelled sum: bring its bits up, or an exact zero
    if (l == 0u) return 0.0;
    h = l;
    l = 0u;
    e -= 32;
  }
  const int lz = __clz((int)h);
  h = __funnelshift_l(l, h, lz);
  l <<= lz;
  // 53 leading bits, the implicit one included (it carries into the exponent)
  const unsigned long long mant = ((unsigned long long)(h >> 11) << 32 | __funnelshift_r(l, h, 11)) + (l >> 10 & 1u);
  return __hiloint2double((int)(((unsigned)(1023 + 63 - 1 + e - lz) << 20) + (unsigned)(mant >> 32) | sg),
                          (int)(unsigned)mant);
}

// ------------------------------------------- entries summed term by term ----
// What the elements' functions read of a point, in registers (the SM's storage is all
// shared memory here, so that every load goes to L2).
__device__ __forceinline__ PointDesc fields(const PointDesc &P) {
  PointDesc p;
  p.N = P.N;
  p.U = P.U;
  p.Lpp = P.Lpp;
  p.Lph = P.Lph;
  return p;
}
// Four consecutive columns of one row of a product in FP64, by one warp; lane q
// returns column c + q % 4.  Terms k and D - 1 - k are added first, so that a
// transfer and its mirror (frequency reversal) give conjugate sums bit for bit.
template <int CH>
__device__ __noinline__ double2 row_sums(const PointDesc &P, const RhsIO &o, int m, int row, int c, int lane) {
  const PointDesc p = fields(P);
  const void *gam = o.gam;
  const int N = p.N;
  const Geom g = geom(CH, N, m);
  double2 acc[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) acc[q] = make_double2(0.0, 0.0);
  for (int k0 = 0; k0 < g.K; k0 += g.D)  // (the direct channel's two ranges of D)
    for (int k = lane; 2 * k < g.D; k += 32) {
      const int j = g.D - 1 - k;
      const double2 a = left_elem<CH>(p, gam, g, row, k0 + k);
      const double2 b = j == k ? make_double2(0.0, 0.0) : left_elem<CH>(p, gam, g, row, k0 + j);
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        if (c + q >= N) break;
        double2 t = cmul(a, right_elem<CH>(p, gam, g, k0 + k, c + q));
        if (j != k) t = cadd(t, cmul(b, right_elem<CH>(p, gam, g, k0 + j, c + q)));
        acc[q] = cadd(acc[q], t);
      }
    }
  double2 z = acc[0];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    for (int off = 16; off > 0; off >>= 1) {
      acc[q].x += __shfl_xor_sync(0xffffffffu, acc[q].x, off);
      acc[q].y += __shfl_xor_sync(0xffffffffu, acc[q].y, off);
    }
    if ((lane & 3) == q) z = acc[q];
  }
  return cscale(z, (CH == CH_DPH ? 1.0 : -1.0) * P.T * (*o.lam));
}
// Row pointer of local row rr in the channel's own layout (pp: natural, dph: X,
// xph: W).
__device__ __forceinline__ double2 *out_row(int ch, double2 *kN, const X64Pt &x, int N, const Geom &g, int rr) {
  const int a = g.row_lo + rr;
  if (ch == CH_PP) return kN + ((size_t)a * N + (g.x - a)) * N;
  if (ch == CH_DPH) return x.PX + ((size_t)a * N + (a + g.x)) * N;
  return x.PW + ((size_t)(a + g.x) * N + a) * N;
}

// Whether the slices may not hold an entry z to FP64's own rounding (kl, kr: the records
// of its row and column).  Their error is some 2^-60 of B = 2^(eL + eR) and half a unit,
// 2^(-62 + v) B, per chunk; that of a chain of FP64 multiply-adds some 2^-53 of S = sum
// |L_k| |R_k|.  An entry stands that is large enough itself, or whose column's small
// values are too few to meet half of the row's sum (more than 2^(v - 1) 2^eL, each at most
// 2 2^eL): S is then above 2^-(EVEN + 2) 2^eR of that sum.
__device__ __forceinline__ bool unsettled(double2 z, int kl, int kr) {
  const int v = rec_val(kl), small = rec_val(kr);
  return ((kl | kr) & UNSLICED) ||
         (small && 8 * small > 1 << v && (int)(mag(z) >> 20) - 1023 < rec_exp(kl) + rec_exp(kr) + max(v - 9, -7));
}

// One tile in FP64 by the epilogue warps, 16 k at a time through the operand stages'
// shared memory (free by then): warp w the rows w, w + 16, ..., two columns per lane.
// Bound by the FP64 units (64 x 64 x 16 terms take 131000 cycles).
struct SettleSmem {
  double2 L[KS][LINES], R[KS][LINES];
};
template <int CH>
__device__ __noinline__ void settle_tile(const PointDesc &P, const RhsIO &o, const X64Pt &x, const Work &w,
                                            SettleSmem &sm, int t) {
  const PointDesc p = fields(P);
  const void *gam = o.gam;
  const int N = p.N, r0 = w.rt * LINES, c0 = w.ct * LINES, lane = t & 31, warp = t >> 5;
  const Geom g = geom(CH, N, w.m);
  const int nr = min(LINES, g.D - r0), nc = min(LINES, N - c0);
  double2 acc[4][2];
#pragma unroll
  for (int i = 0; i < 4; ++i) acc[i][0] = acc[i][1] = make_double2(0.0, 0.0);
  for (int k0 = 0; k0 < g.K; k0 += KS) {
    const int nk = min(KS, g.K - k0);
    const int q = t % LINES, k1 = t / LINES, k2 = k1 + 32 * EPI_W / LINES;
    const bool a = q < nr, b = q < nc;
    const double2 z = make_double2(0.0, 0.0);
    const double2 l1 = a && k1 < nk ? left_elem<CH>(p, gam, g, r0 + q, k0 + k1) : z,
                  l2 = a && k2 < nk ? left_elem<CH>(p, gam, g, r0 + q, k0 + k2) : z,
                  v1 = b && k1 < nk ? right_elem<CH>(p, gam, g, k0 + k1, c0 + q) : z,
                  v2 = b && k2 < nk ? right_elem<CH>(p, gam, g, k0 + k2, c0 + q) : z;
    sm.L[k1][q] = l1;
    sm.L[k2][q] = l2;
    sm.R[k1][q] = v1;
    sm.R[k2][q] = v2;
    epi_sync();
    for (int k = 0; k < nk; ++k)
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        if (warp + EPI_W * i >= nr) break;
        const double2 a = sm.L[k][warp + EPI_W * i];
        cfma(acc[i][0], a, sm.R[k][lane]);
        cfma(acc[i][1], a, sm.R[k][lane + 32]);
      }
    epi_sync();
  }
  const double sc = (CH == CH_DPH ? 1.0 : -1.0) * P.T * (*o.lam);
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int r = warp + EPI_W * i;
    if (r >= nr) break;
    double2 *out = out_row(CH, static_cast<double2 *>(o.dgam), x, N, g, r0 + r) + c0;
    if (lane < nc) out[lane] = cscale(acc[i][0], sc);
    if (lane + 32 < nc) out[lane + 32] = cscale(acc[i][1], sc);
  }
}

// The unsettled entries of a tile again in FP64 (all epilogue warps): each group of four
// columns of a row by one warp, or the whole tile at once where that is less work (a
// group takes the FP64 units some 25 K cycles, a tile 2 K for each of its entries: from a
// third of the groups on).  Call n counts its groups in cnt[n % 3]; before its barrier it
// zeroes the counter of call n + 1, which every warp has read (as that of call n - 2)
// before the barrier of call n - 1.
__device__ __noinline__ void settle(const PointDesc *__restrict__ pts, const RhsIO *__restrict__ io,
                                    const X64Pt *__restrict__ xp, const Work &w, SettleSmem &sm, int *cnt, int n,
                                    int t) {
  const PointDesc &P = pts[w.point];
  const RhsIO &o = io[w.point];
  const X64Pt &x = xp[w.point];
  const int N = P.N, r0 = w.rt * LINES, c0 = w.ct * LINES, lane = t & 31, warp = t >> 5;
  const Geom g = geom(w.ch, N, w.m);
  const int *eL = x.eL + (size_t)w.el * LINES, *eR = x.eR + (size_t)w.er * LINES;
  double2 *kN = static_cast<double2 *>(o.dgam);
  // eight rows at a time, four lanes each: warp w takes the columns 4 ((w + row) % 16) on
  // of a row, so that the groups of one row or one column lie in different warps
  auto col4 = [&](int row) { return 4 * ((warp + row) % (LINES / 4)); };
  unsigned mine = 0u;  // the lane's unsettled entries, a bit per eight rows
  int groups = 0;
  for (int b = 0; b < LINES / 8; ++b) {
    const int row = 8 * b + (lane >> 2), col = col4(row) + (lane & 3);
    const bool on = r0 + row < g.D && c0 + col < N &&
                    unsettled(out_row(w.ch, kN, x, N, g, r0 + row)[c0 + col], eL[row], eR[col]);
    mine |= (unsigned)on << b;
    const unsigned v = __ballot_sync(0xffffffffu, on);
    groups += __popc((v | v >> 1 | v >> 2 | v >> 3) & 0x11111111u);
  }
  if (lane == 0 && groups) atomicAdd(&cnt[n % 3], groups);
  if (t == 0) cnt[(n + 1) % 3] = 0;
  epi_sync();
  const int total = *const_cast<volatile int *>(cnt + n % 3);
  if (12 * total > min(LINES, g.D - r0) * min(LINES, N - c0)) {
    if (w.ch == CH_PP)
      settle_tile<CH_PP>(P, o, x, w, sm, t);
    else if (w.ch == CH_DPH)
      settle_tile<CH_DPH>(P, o, x, w, sm, t);
    else
      settle_tile<CH_XPH>(P, o, x, w, sm, t);
  } else if (groups) {
    for (int b = 0; b < LINES / 8; ++b)
      for (unsigned todo = __ballot_sync(0xffffffffu, mine >> b & 1u); todo;) {
        const int q = (__ffs(todo) - 1) >> 2, row = 8 * b + q, r = r0 + row, c = c0 + col4(row);
        const double2 s = w.ch == CH_PP    ? row_sums<CH_PP>(P, o, w.m, r, c, lane)
                          : w.ch == CH_DPH ? row_sums<CH_DPH>(P, o, w.m, r, c, lane)
                                           : row_sums<CH_XPH>(P, o, w.m, r, c, lane);
        if ((mine >> b & 1u) && lane >> 2 == q) out_row(w.ch, kN, x, N, g, r)[c + (lane & 3)] = s;
        todo &= ~(0xfu << (4 * q));
      }
  }
}

__global__ void __launch_bounds__(THREADS, 1)
    k_x64_products(const PointDesc *__restrict__ pts, const RhsIO *__restrict__ io, const X64Pt *__restrict__ xp,
                   const Work *__restrict__ work, const int *__restrict__ cta_start, unsigned *__restrict__ err) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t *smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  uint8_t *ops = smem, *raws = ops + NOP * OP_STAGE, *epi = raws + NRAW * BLK_BYTES;
  // raw barriers: [side][slot]
  uint64_t *raw_full = reinterpret_cast<uint64_t *>(epi + EPI_W / 2 * EPI_BUF), *raw_empty = raw_full + 2 * NRAW;
  uint64_t *op_full = raw_empty + 2 * NRAW, *op_empty = op_full + NOP, *tfull = op_empty + NOP, *tempty = tfull + 1;
  uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(tempty + 1);
  volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);
  int *again = reinterpret_cast<int *>(tmem_slot + 2);  // a second pass is wanted; a wait gave up; three counters
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (tid == 0) {
    for (int j = 0; j < 2 * NRAW; ++j) {
      mbar_init(&raw_full[j], 1);
      mbar_init(&raw_empty[j], N_XF / 2);
    }
    for (int s = 0; s < NOP; ++s) {
      mbar_init(&op_full[s], N_XF);
      mbar_init(&op_empty[s], 1);
    }
    mbar_init(tfull, 1);
    mbar_init(tempty, EPI_W);
    *abort_flag = 0;
    for (int j = 0; j < 5; ++j) again[j] = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == MMA_W) tmem_alloc(tmem_slot, 512);
  tc_before();
  __syncthreads();
  tc_after();
  const uint32_t tmem = *tmem_slot;
  const int w0 = cta_start[blockIdx.x], w1 = cta_start[blockIdx.x + 1];
  chain_wait();

  // Raw block b (left and right operand's in turn) lies in slot b % 3.  Each side has
  // barriers of its own for every slot, so that whoever waits on one takes part in each
  // of its phases: a side's n-th block is phase n / 3 of its slot's pair.
  if (warp == LOAD_W) {
    uint32_t b = 0;
    bool ok = true;
    for (int wi = w0; wi < w1 && ok; ++wi) {
      const Work w = work[wi];
      look_ahead(pts, io, xp, work, wi, w1, lane);
      if (!io[w.point].active) continue;
      const ulonglong2 *L = xp[w.point].L + (size_t)w.bl * BLK, *R = xp[w.point].R + (size_t)w.br * BLK;
      for (int kb = 0; kb < 2 * w.nk; ++kb, ++b) {
        const uint32_t j = b % NRAW, side = b & 1u;
        if (b >= NRAW) {  // the slot's previous block, the other side's
          const uint32_t p = b - NRAW;
          if (!(ok = wwait(&raw_empty[(p & 1u) * NRAW + j], ((p >> 1) / NRAW) & 1u, err, abort_flag))) break;
        }
        if (lane == 0) {
          uint64_t *bar = &raw_full[side * NRAW + j];
          arrive_expect_tx(bar, BLK_BYTES);
          bulk_copy(raws + j * BLK_BYTES, (side ? R : L) + (size_t)(kb >> 1) * BLK, BLK_BYTES, bar);
        }
        __syncwarp();
      }
    }
    // copies still in flight must land before the CTA leaves
    for (uint32_t k = b > (uint32_t)NRAW ? b - NRAW : 0u; k < b; ++k)
      wwait(&raw_full[(k & 1u) * NRAW + k % NRAW], ((k >> 1) / NRAW) & 1u, err, abort_flag);
  } else if (warp >= XF_W0) {
    // warps 0-3 of the role: left lines, 4-7: right lines; one line and eight
    // of the 16 k per thread
    const int xt = tid - 32 * XF_W0, side = xt >> 7, oct = (xt >> 6) & 1, line = xt & 63;
    const uint32_t src = (oct * 8 * LINES + line) * 16;
    const uint32_t at = (side ? A_BYTES + oct * B_KC : oct * A_KC) + line * 16;
    uint32_t it = 0;
    bool ok = true;
    for (int wi = w0; wi < w1 && ok; ++wi) {
      const Work w = work[wi];
      if (!io[w.point].active) continue;
      for (int kb = 0; kb < w.nk; ++kb, ++it) {
        const int j = (2 * it + side) % NRAW, s = it % NOP;
        if (!(ok = wwait(&raw_full[side * NRAW + j], (it / NRAW) & 1u, err, abort_flag))) break;
        const uint8_t *raw = raws + j * BLK_BYTES + src;
        uint4 v[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) v[q] = *reinterpret_cast<const uint4 *>(raw + q * LINES * 16);
        // the loader's next copy into this slot is an async-proxy write: order
        // the reads above before it
        fence_async_smem();
        __syncwarp();
        if (lane == 0) mbar_arrive(&raw_empty[side * NRAW + j]);
        if (!(ok = wwait(&op_empty[s], ((it / NOP) & 1u) ^ 1u, err, abort_flag))) break;
        uint8_t *dst = ops + s * OP_STAGE + at;
        if (side == 0)
          store_digits<true>(dst, v);
        else
          store_digits<false>(dst, v);
        fence_async_smem();
        __syncwarp();
        if (lane == 0) mbar_arrive(&op_full[s]);
      }
    }
  } else if (warp == MMA_W) {
    uint32_t it = 0, use = 0;
    bool ok = true;
    for (int wi = w0; wi < w1 && ok; ++wi) {
      const Work w = work[wi];
      if (!io[w.point].active) continue;
      for (int kb = 0; kb < w.nk; ++kb, ++it) {
        const int s = it % NOP;
        if (kb % CHUNK == 0) {
          if (!(ok = wwait(tempty, (use & 1u) ^ 1u, err, abort_flag))) break;
          ++use;
          tc_after();
        }
        if (!(ok = wwait(&op_full[s], (it / NOP) & 1u, err, abort_flag))) break;
        tc_after();
        if (lane == 0) {
          const uint32_t a0 = smem_u32(ops + s * OP_STAGE), b0 = a0 + A_BYTES;
#pragma unroll
          for (int q = 0; q < 2; ++q) {
            // q = 0: [Re; Im] (planes 1, 2) x Re b; q = 1: [-Im; Re] (planes 0, 1) x Im b
            const uint32_t aq = a0 + (q == 0 ? PLANE : 0), bq = b0 + q * B_PL;
#pragma unroll
            for (int i = 0; i < SL; ++i) {
              // (digit 0 starts every accumulator of the chunk's first k-step; 256 columns and the
              // rest, not two halves: 398 against 402 us per rhs at N = 128)
              const int cols = LINES * (NACC - i), n1 = cols > 256 ? 256 : cols;
              const uint64_t da = desc(aq + i * A_DIG, A_KC, 128);
              const uint32_t d = tmem + LINES * i, acc = (kb % CHUNK | q | i) ? 1u : 0u;
              mma_f16(d, da, desc(bq, B_KC, 128), idesc(n1), acc);
              if (cols > 256)  // the rest of the columns: 32 line groups further on
                mma_f16(d + n1, da, desc(bq + n1 / 8 * 128, B_KC, 128), idesc(cols - n1), acc);
            }
          }
          mma_commit(&op_empty[s]);
          if (kb % CHUNK == CHUNK - 1 || kb == w.nk - 1) mma_commit(tfull);
        }
        __syncwarp();
      }
    }
  } else {
    // warp w reads TMEM lanes 32 (w % 4) on (Re of the rows 0-31 and 32-63, then
    // their Im) and the columns 16 (w / 4) on.  The accumulators of all its entries
    // are added up in registers chunk by chunk, so that the next products can start;
    // after the tile's last chunk the entries are rounded and stored, four columns at
    // a time, through a buffer that warps w and w ^ 2 (Re and Im of the same rows) share.
    const int quarter = warp & 3, comp = quarter >> 1, pair = (quarter & 1) | (warp >> 2) << 1;
    const int cb = EPI_CPW * (warp >> 2);
    uint8_t *buf = epi + pair * EPI_BUF;
    const uint32_t tl = tmem + ((uint32_t)(quarter * 32) << 16) + cb;
    const int rl = 32 * (quarter & 1);  // first row of this warp's half
    uint32_t use = 0;
    bool ok = true, check = false;
    for (int wi = w0; wi < w1 && ok; ++wi) {
      const Work w = work[wi];
      if (!io[w.point].active) continue;
      const int N = pts[w.point].N, r0 = w.rt * LINES + rl, c0 = w.ct * LINES + cb;
      const Geom g = geom(w.ch, N, w.m);
      double2 *kN = static_cast<double2 *>(io[w.point].dgam);
      const X64Pt &x = xp[w.point];
      const int kl = r0 + lane < g.D ? x.eL[(size_t)w.el * LINES + rl + lane] : 0;
      const int kr = lane < EPI_CPW && c0 + lane < N ? x.eR[(size_t)w.er * LINES + cb + lane] : 0;
      check |= __any_sync(0xffffffffu, (kl & UNSLICED) || (kr & UNSLICED) || rec_val(kr));
      const Limbs limbs = limbs_of(rec_val(kl));
      unsigned long long s[EPI_CPW];
#pragma unroll
      for (int c = 0; c < EPI_CPW; ++c) s[c] = 0ull - (w.nk + CHUNK - 1) / CHUNK * limbs_sum(limbs.t, limbs.u, limbs.z);
      for (int kb = 0; kb < w.nk; kb += CHUNK) {
        // both warps of a pair leave together when a wait gave up
        if (!(ok = pair_all(wwait(tfull, use & 1u, err, abort_flag), pair))) break;
        ++use;
        tc_after();
#pragma unroll
        for (int c = 0; c < EPI_CPW; c += 2) {
          float a[NACC][2];
#pragma unroll
          for (int q = 0; q < NACC; ++q) tmem_ld2(tl + q * LINES + c, a[q]);
          tmem_wait_ld();
          add_chunk(s[c], a, 0, limbs);
          add_chunk(s[c + 1], a, 1, limbs);
        }
        tc_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(tempty);
      }
      if (!ok) break;
#pragma unroll
      for (int cc = 0; cc < EPI_CPW; cc += EPI_COLS) {
        if (c0 + cc >= N) break;  // (uniform over the pair)
#pragma unroll
        for (int c = 0; c < EPI_COLS; ++c)
          *reinterpret_cast<double *>(buf + lane * (EPI_COLS * 16) + ((c ^ ((lane >> 1) & 3)) << 4) + comp * 8) =
              scaled((long long)s[cc + c],
                     rec_exp(kl) + rec_exp(__shfl_sync(0xffffffffu, kr, cc + c)) + rec_val(kl) + 65 - 2 * FIX);
        asm volatile("bar.sync %0, 64;" ::"r"(1 + pair) : "memory");
        // each warp of the pair stores 16 of the 32 rows, 64 bytes a row
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const int row = comp * 16 + (lane >> 2) + 8 * i, c = lane & 3;
          const double2 z = *reinterpret_cast<const double2 *>(buf + row * (EPI_COLS * 16) + ((c ^ ((row >> 1) & 3)) << 4));
          const int col = c0 + cc + c;
          if (r0 + row < g.D && col < N) out_row(w.ch, kN, x, N, g, r0 + row)[col] = z;
        }
        asm volatile("bar.sync %0, 64;" ::"r"(1 + pair) : "memory");
      }
    }
    // a second pass (rare: kept out of the first one's registers) over the tiles, when
    // every warp's stores are done
    if (lane == 0 && check) again[0] = 1;
    if (lane == 0 && !ok) again[1] = 1;
    __threadfence_block();
    epi_sync();
    if (again[0] && !again[1]) {
      int n = 0;
      for (int wi = w0; wi < w1; ++wi)
        if (io[work[wi].point].active)
          settle(pts, io, xp, work[wi], *reinterpret_cast<SettleSmem *>(ops), again + 2, n++, tid);
    }
  }
  tc_before();
  __syncthreads();
  tc_after();
  if (warp == MMA_W) tmem_dealloc(tmem, 512);
}

// ------------------------------------------------------------- combine ----
// dGamma = (pp + direct) + crossed, the enabled channels, into the natural
// layout (the pp products are there already).  A thread takes IW consecutive
// i1 of one (i2, i3): 32 contiguous bytes of a W row; a warp covers 4 i2 (64
// bytes of each X row) x 8 i3 (128 bytes of each natural row).
// IW rows i1 per thread: two make a whole sector of the crossed output's layout, and
// enough blocks (flow N = 64 25.9 ms, against 26.8 with four and 25.7 with one; N = 128
// 320.8 us per rhs, against 322.5 and 324.4; with products of seven digits).
constexpr int IW = 2;
template <bool REV>
__global__ void __launch_bounds__(256, 6) k_x64_combine(const PointDesc *__restrict__ pts,
                                                     const RhsIO *__restrict__ io, const X64Pt *__restrict__ xp,
                                                     int p0, int nz, int chmask) {
  chain_wait();
  const int pi = p0 + blockIdx.z / nz;
  const RhsIO &o = io[pi];
  const X64Pt &x = xp[pi];
  if (!o.active || !x.prod) return;
  const PointDesc &P = pts[pi];
  // REV: the rows i1 < N / 2, each entry from its own transfer or, where that is
  // above N - 1, as the conjugate of its mirror's, and its mirror as the conjugate
  const int N = P.N, n1 = REV ? N / 2 : N, t = threadIdx.x;
  const size_t end = (size_t)N * N * N - 1;
  const int i1 = IW * (blockIdx.z % nz), b2 = 8 * blockIdx.y, b3 = 32 * blockIdx.x;
  if (i1 >= n1 || b2 >= N || b3 >= N) return;
  const int i2 = b2 + 4 * (t >> 7) + ((t >> 3) & 3), i3 = b3 + 8 * ((t >> 5) & 3) + (t & 7);
  double2 *out = static_cast<double2 *>(o.dgam);
  const double2 z = make_double2(0.0, 0.0);
  const bool on = i2 < N && i3 < N;
  double2 a[IW], b[IW], c[IW];
#pragma unroll
  for (int j = 0; j < IW; ++j) {
    const bool in = on && i1 + j < n1;
    const size_t ea = ((size_t)(i1 + j) * N + i2) * N + i3, eb = ((size_t)(i1 + j) * N + i3) * N + i2,
                 ec = ((size_t)i2 * N + i3) * N + i1 + j;
    const bool ma = REV && i1 + j + i2 > N - 1, mb = REV && i3 > i1 + j, mc = REV && i2 > i3;
    a[j] = in && (chmask & 1) ? out[ma ? end - ea : ea] : z;
    b[j] = in && (chmask & 2) ? x.PX[mb ? end - eb : eb] : z;
    c[j] = in && (chmask & 4) ? x.PW[mc ? end - ec : ec] : z;
    if (ma) a[j].y = -a[j].y;
    if (mb) b[j].y = -b[j].y;
    if (mc) c[j].y = -c[j].y;
  }
  if (!on) return;
#pragma unroll
  for (int j = 0; j < IW; ++j)
    if (i1 + j < n1) {
      const size_t e = ((size_t)(i1 + j) * N + i2) * N + i3;
      const double2 v = cadd(cadd(a[j], b[j]), c[j]);
      out[e] = v;
      if (REV) out[end - e] = make_double2(v.x, -v.y);
    }
}
}  // namespace x64

// ---------------------------------------------------------------- plan ----
struct X64Plan {
  using Sched = Schedule<x64::Work>;
  struct Group {
    int p0, p1, maxN;
    Sched all, half;  // half: the transfers m < N
  };
  std::vector<X64Pt> h;
  std::vector<int> N;          // per point, 0: not on this path
  std::vector<Sched> one;      // per point (a context of one point has its group's alone)
  std::vector<Group> groups;   // points whose operands share the workspace, one group after another
  X64Pt *d_x = nullptr;
  char *ws = nullptr;
  std::vector<void *> tables;
  unsigned *d_err = nullptr;
};

namespace {
// Operands of one group of points at most (a single point may need more: 2.9 GB
// at N = 256): a large batch reuses the workspace group by group, so that the
// path never takes more than a small part of the device's memory.
constexpr size_t X64_WS_CAP = (size_t)4 << 30;
constexpr int X64_GROUP = 256;  // points per group: the combine's grid.z, N / IW per point, stays below 65536
static_assert((FRG_MAX_N + x64::IW - 1) / x64::IW * X64_GROUP < 65536 && 3 * X64_GROUP < 65536, "grid.z");
size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }
thread_local bool t_withheld = false;  // frg_selftest_slices
}  // namespace

void x64_withhold(bool on) { t_withheld = on; }

int x64_create(X64Plan **out, const std::vector<PointDesc> &pts, int chmask, unsigned *d_err) {
  *out = nullptr;
  const int n = (int)pts.size();
  bool any = false;
  for (const PointDesc &P : pts) any = any || P.N >= X64_MIN_N;
  if (!any || !(chmask & 7) || t_withheld) return 0;
  int dev = 0, sms = 0, maj = 0, min_ = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&maj, cudaDevAttrComputeCapabilityMajor, dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&min_, cudaDevAttrComputeCapabilityMinor, dev) != cudaSuccess)
    return -3;
  if (maj != 10 || min_ != 3) return 0;
  X64Plan *p = new X64Plan();
  p->d_err = d_err;
  p->h.assign(n, X64Pt{});
  p->N.assign(n, 0);
  p->one.resize(n);
  // per point: product table, tiles, and the sizes of its operands
  struct Size {
    size_t blkL = 0, blkR = 0, tileL = 0, tileR = 0, n3 = 0;
  };
  std::vector<Size> size(n);
  std::vector<std::vector<uint4>> tab(n);
  std::vector<std::vector<std::pair<int, x64::Work>>> tiles(n);
  for (int i = 0; i < n; ++i) {
    const int N = pts[i].N;
    if (N < X64_MIN_N) continue;
    p->N[i] = N;
    Size &s = size[i];
    s.n3 = (size_t)N * N * N;
    tab[i].resize(3 * (2 * N - 1));
    const int nct = (N + x64::LINES - 1) / x64::LINES;
    for (int ch = 0; ch < 3; ++ch) {
      if (!(chmask >> ch & 1)) continue;
      for (int m = 0; m < 2 * N - 1; ++m) {
        const Geom g = geom(ch, N, m);
        const int nk = (ch == CH_DPH ? 2 : 1) * (x64::d16(g.D) / x64::KS);
        const int nrt = (g.D + x64::LINES - 1) / x64::LINES;
        const uint4 t = make_uint4((unsigned)s.blkL, (unsigned)s.blkR, (unsigned)s.tileL, (unsigned)s.tileR);
        tab[i][ch * (2 * N - 1) + m] = t;
        s.blkL += (size_t)nrt * nk;
        s.blkR += (size_t)nct * nk;
        s.tileL += nrt;
        s.tileR += nct;
        // the drain of a tile's accumulators costs about two k-steps
        for (int rt = 0; rt < nrt; ++rt)
          for (int ct = 0; ct < nct; ++ct)
            tiles[i].push_back({nk + 2, x64::Work{i, (short)m, (short)ch, (short)rt, (short)ct, nk, t.x + rt * nk,
                                                  t.y + ct * nk, t.z + rt, t.w + ct}});
      }
    }
  }
  auto bytes = [&](const Size &s) {
    return align256(s.blkL * x64::BLK_BYTES) + align256(s.blkR * x64::BLK_BYTES) + align256(s.tileL * x64::LINES * 4) +
           align256(s.tileR * x64::LINES * 4) + 2 * align256(s.n3 * sizeof(double2));
  };
  // consecutive points share the workspace up to its cap
  size_t ws = 0;
  std::vector<size_t> base(n, 0);
  for (int i = 0; i < n;) {
    size_t sum = 0;
    int j = i, maxN = 0;
    for (; j < n && j < i + X64_GROUP && (j == i || sum + bytes(size[j]) <= X64_WS_CAP); ++j) {
      base[j] = sum;
      sum += bytes(size[j]);
      maxN = std::max(maxN, p->N[j]);
    }
    if (maxN) p->groups.push_back({i, j, maxN, {}});
    ws = std::max(ws, sum);
    i = j;
  }
  bool ok = cudaMalloc(&p->ws, ws) == cudaSuccess &&
            cudaMalloc(&p->d_x, sizeof(X64Pt) * n) == cudaSuccess &&
            cudaFuncSetAttribute(x64::k_x64_products, cudaFuncAttributeMaxDynamicSharedMemorySize, x64::SMEM) ==
                cudaSuccess;
  for (int i = 0; i < n && ok; ++i) {
    if (!p->N[i]) continue;
    X64Pt &x = p->h[i];
    const Size &s = size[i];
    char *b = p->ws + base[i];
    x.L = reinterpret_cast<ulonglong2 *>(b);
    b += align256(s.blkL * x64::BLK_BYTES);
    x.R = reinterpret_cast<ulonglong2 *>(b);
    b += align256(s.blkR * x64::BLK_BYTES);
    x.eL = reinterpret_cast<int *>(b);
    b += align256(s.tileL * x64::LINES * 4);
    x.eR = reinterpret_cast<int *>(b);
    b += align256(s.tileR * x64::LINES * 4);
    x.PX = reinterpret_cast<double2 *>(b);
    b += align256(s.n3 * sizeof(double2));
    x.PW = reinterpret_cast<double2 *>(b);
    void *t = nullptr;
    ok = cudaMalloc(&t, sizeof(uint4) * tab[i].size()) == cudaSuccess;
    if (!ok) break;
    p->tables.push_back(t);
    x.prod = static_cast<const uint4 *>(t);
    ok = cudaMemcpy(t, tab[i].data(), sizeof(uint4) * tab[i].size(), cudaMemcpyHostToDevice) == cudaSuccess &&
         (n == 1 || upload_schedule(p->one[i], tiles[i], sms));
  }
  for (X64Plan::Group &g : p->groups) {
    if (!ok) break;
    std::vector<std::pair<int, x64::Work>> all;
    for (int i = g.p0; i < g.p1; ++i) all.insert(all.end(), tiles[i].begin(), tiles[i].end());
    std::vector<std::pair<int, x64::Work>> low;
    for (auto &t : all)
      if (t.second.m < pts[t.second.point].N) low.push_back(t);
    ok = upload_schedule(g.all, all, sms) && upload_schedule(g.half, low, sms);
  }
  ok = ok && cudaMemcpy(p->d_x, p->h.data(), sizeof(X64Pt) * n, cudaMemcpyHostToDevice) == cudaSuccess;
  if (!ok) {
    const bool room = cudaGetLastError() != cudaErrorMemoryAllocation;
    x64_destroy(p);
    return room ? -3 : 0;
  }
  *out = p;
  return 0;
}

void x64_destroy(X64Plan *p) {
  if (!p) return;
  for (auto &s : p->one) drop_schedule(s);
  for (auto &g : p->groups) {
    drop_schedule(g.all);
    drop_schedule(g.half);
  }
  for (void *t : p->tables) cudaFree(t);
  cudaFree(p->d_x);
  cudaFree(p->ws);
  delete p;
}

bool x64_has(const X64Plan *p, int point) { return p && p->N[point] > 0; }

int x64_run(X64Plan *p, const PointDesc *d_pts, const RhsIO *d_io, int point, int chmask, cudaStream_t st,
            bool chain, bool half) {
  for (size_t gi = 0; gi < p->groups.size(); ++gi) {
    X64Plan::Group &g = p->groups[gi];
    int p0 = g.p0, p1 = g.p1, maxN = g.maxN;
    const X64Plan::Sched *s = half ? &g.half : &g.all;
    if (point >= 0) {
      if (point < g.p0 || point >= g.p1) continue;
      p0 = point;
      p1 = point + 1;
      maxN = p->N[point];
      if (p->N.size() > 1) s = &p->one[point];
    }
    const int oct = (maxN + x64::PAN_LINES - 1) / x64::PAN_LINES, np = p1 - p0;
    const dim3 pg(2 * oct, half ? maxN : 2 * maxN - 1, 3 * np);
    const int nz = ((half ? maxN / 2 : maxN) + x64::IW - 1) / x64::IW, rev = half ? 1 : 0;
    // The combine is not chained: blocks that become resident beside the products' find
    // the SM's storage set up as shared memory and next to no L1, and so do the kernels
    // chained to them (N = 128 336 against 322 us per rhs, N = 64 62.0 against 59.8 us
    // and 37.8 against 35.8 ms per flow; nothing chained 327 and 65.0 us, 36.2 ms; all with
    // seven digits).
    if (launch_chained(x64::panel_u(maxN) == 8 ? x64::k_x64_panels<8> : x64::k_x64_panels<4>, pg,
                       x64::panel_threads(maxN), 0, st, chain, d_pts, d_io, p->d_x, p0, chmask, rev) != cudaSuccess ||
        launch_chained(x64::k_x64_products, s->grid, x64::THREADS, x64::SMEM, st, chain, d_pts, d_io, p->d_x, s->work,
                       s->start, p->d_err) != cudaSuccess ||
        launch_chained(half ? x64::k_x64_combine<true> : x64::k_x64_combine<false>,
                       dim3((maxN + 31) / 32, (maxN + 7) / 8, nz * np), 256, 0, st, false, d_pts, d_io, p->d_x, p0, nz,
                       chmask) != cudaSuccess)
      return -3;
    FRG_COUNT(3);
  }
  return cudaGetLastError() == cudaSuccess ? 0 : -3;
}

}  // namespace frg
