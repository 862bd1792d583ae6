// frg_small.cuh -- FP64 right-hand sides of small grids in one launch.
#pragma once
#include "frg_common.cuh"

namespace frg {
constexpr int SMALL_MAX_N = 64;  // limited by the block's shared memory
// Vertex and self-energy rhs of every active point with N < n_below (<= 65).
// sig_in_place: a self-energy output overlaps its input (the self-energy rhs then
// takes a launch of one block per point, after every other block has read it).
// chain: see launch_ex.  half: the inputs are reversal-symmetric, so the entries
// with i1 < N / 2 give the others as conjugates.
int launch_rhs_small(const PointDesc *d_pts, const RhsIO *d_io, int n_points, int maxN, int n_below, int mask,
                     bool sig_in_place, cudaStream_t st, bool chain, bool half);
// The same for one point (N <= SMALL_MAX_N) given by value: no device memory.
int launch_rhs_small_value(const PointDesc &P, const RhsIO &o, double lam, int mask, bool sig_in_place,
                           cudaStream_t st);
// Before a stand-alone one-launch rhs: whether its self-energy output overlaps the input;
// an input that the vertex output overlaps is moved into the self-energy output first.
int small_sigma(RhsIO &o, int N, cudaStream_t st, bool *in_place);
}  // namespace frg
