// frg_integrator.cuh -- launchers of the device-resident Dormand-Prince pair.
#pragma once
#include "frg_common.cuh"

namespace frg {

int upload_tableau();
// Embedded error weights E_j = b_j - bstar_j of the Dormand-Prince pair (FP64)
// and E_7 as a float pair, for the split paths' scatter-add of k7, which
// completes the step's error estimate.
struct ErrWeights {
  double E[7];
  float e7h, e7l;
};
ErrWeights host_error_weights();
void host_tableau(double *c, double *a, double *bstar);
int launch_init(const PointDesc *d_pts, Ctl *d_ctl, int maxN, int n, cudaStream_t st);
int launch_set_ctl(const PointDesc *d_pts, Ctl *d_ctl, int pi, double t, double h, cudaStream_t st);
int launch_set_stage_io(const PointDesc *d_pts, Ctl *d_ctl, RhsIO *d_io, int stage, int split, int n,
                        cudaStream_t st);
int launch_finish_k1(Ctl *d_ctl, const RhsIO *d_io, int n, cudaStream_t st);
int launch_prepare(const PointDesc *d_pts, Ctl *d_ctl, int n, cudaStream_t st);
// FP64 path: stage sum s (1..6) of every point; the first block of each point
// also writes the stage's rhs IO record (as launch_set_stage_io), and the seventh
// stage leaves the partial error sum in the place of k2.  rev (here and in
// launch_error): the flow keeps the reversal reduction.
int launch_stage_fp64(const PointDesc *d_pts, Ctl *d_ctl, int s, RhsIO *d_io, cudaStream_t st, int n_points, int maxN,
                      bool rev);
// Split paths: stage sum s of every point, the vertex part only, on a grid of
// lb_grid x n_points layout blocks (frg_lblock.cuh; lb_grid = the largest
// point's vertex blocks), also writing the W / X / Z copies in `want`;
// launch_sigma_stage does the self-energy part and the IO record.
int launch_stage(const PointDesc *d_pts, Ctl *d_ctl, int s, cudaStream_t st, int lb_grid, int n_points, int want);
// Split flows: the scatter-add of the rhs of stage s - 1 (channel bits and
// FRG_TAILS of mask) fused with the vertex part of stage sum s (s = 2..6; rev:
// the reversal reduction's canonical half and mirrored reads; vmax: keep the
// stage input's bound for the BF16x3 slicing), on the stage kernels' grid.
int launch_combine_stage(const PointDesc *d_pts, Ctl *d_ctl, int s, bool rev, bool vmax, int mask, cudaStream_t st,
                         int lb_grid, int n_points, int want);
// Split paths: the self-energy part of stage s and the stage's rhs IO record
// (one block per point).  Independent of the vertex part, so it may run on
// another stream beside launch_stage's kernel.
int launch_sigma_stage(const PointDesc *d_pts, Ctl *d_ctl, RhsIO *d_io, int s, int n_points, cudaStream_t st,
                       int mask);
// Dynamic shared-memory limits of the split stage kernels (once per set-up).
int stage_split_init();
// FP64 path's error norm of the step (after the seventh rhs).
int launch_error(const PointDesc *d_pts, Ctl *d_ctl, cudaStream_t st, int n_points, int maxN, bool rev);
int launch_controller(const PointDesc *d_pts, Ctl *d_ctl, int n, cudaStream_t st);

}  // namespace frg
