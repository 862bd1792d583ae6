// frg_layout.cuh -- launchers of the vertex relayout and channel-combine kernels.
#pragma once
#include "frg_common.cuh"

namespace frg {
// Dynamic shared-memory limits of the layout kernels (once per context set-up).
int layout_init();
// The FP32 operand copies of one point from a natural FP64 vertex: Y32 and the
// layouts in want (LAY_* bits), with vmax also the bound of its entries.
int launch_relayout(const PointDesc *d_pt, const double2 *gam, int N, int want, bool vmax, cudaStream_t st,
                    bool chain);
// The constant (bare U) entries of every point's Z layout, once at set-up.
int launch_fill_z(const PointDesc *d_pts, int n_points, cudaStream_t st);
// io.dgam (natural; it holds the pp output when mask bit 0, unless FRG_REVERSAL
// in mask: then PN holds it) += PX, PW; with err (the seventh rhs of a flow
// step) also the step's error estimate (io.ctl).  canon_half: every active
// point's io.canon is set (only the rows i1 < N/2 are formed), so the grid
// covers those alone.  out64: the sum goes to io.out64 in FP64 instead.
// chain (launch_relayout; the combine with out64): see launch_ex.
int launch_combine(const PointDesc *d_pts, const RhsIO *d_io, int n_points, int maxN, int mask, cudaStream_t st,
                   bool err = false, bool canon_half = false, bool out64 = false, bool chain = false);
}  // namespace frg
