// frg_x64.cuh -- FP64 channel products on the tensor cores (plan and launch).
#pragma once
#include <vector>

#include "frg_common.cuh"

namespace frg {

// Smallest grid whose FP64 channel products take the sliced tensor-core path; the
// ones below take the one-launch rhs (frg_small.cu).  Measured per rhs: N = 24 32
// (sliced) against 25 us, N = 26 39 against 35 us, N = 28 37 against 40 us, N = 32 42
// against 47 us.
constexpr int X64_MIN_N = 28;

// Device-side operands of one point (frg_x64.cu).
struct X64Pt {
  const uint4 *prod;   // per ch * (2N - 1) + m: first left and right operand block, first left and right tile of
                       // exponents; null: not on this path
  ulonglong2 *L, *R;   // fixed-point operand blocks (re, im), 16 k x 64 lines each
  int *eL, *eR;        // line records (exponent and flags), 64 per tile
  double2 *PX, *PW;    // direct (layout X) and crossed (layout W) channel outputs
};

struct X64Plan;
// Plan for the points with N >= X64_MIN_N.  *out stays null when there is none
// or the device has no room for the operands (the caller then keeps those
// points on the CUDA-core path).  Returns 0, or -3 when a CUDA call failed.
int x64_create(X64Plan **out, const std::vector<PointDesc> &pts, int chmask, unsigned *d_err);
void x64_destroy(X64Plan *p);
// on: plans that the calling thread makes find no room (frg_selftest_slices).
void x64_withhold(bool on);
bool x64_has(const X64Plan *p, int point);
// Channel products of every point of the plan (point < 0) or of one point; chain:
// see launch_ex; half (every point): the inputs are reversal-symmetric, so the
// transfers m < N give the others (V(N-1-i1, N-1-i2, N-1-i3) = conj V(i1, i2, i3)
// takes transfer m of each channel to 2N - 2 - m).
int x64_run(X64Plan *p, const PointDesc *d_pts, const RhsIO *d_io, int point, int chmask, cudaStream_t st,
            bool chain, bool half);
}  // namespace frg
