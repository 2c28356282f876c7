// Host side of the fixed-point colour passes (fixed_sweeps.cu).
#pragma once
#include "ps_common.cuh"

namespace ps {

enum { FC_SWEEP = 0, FC_LAG = 1, FC_RESID = 2, FC_NORM = 3, FC_OPEN = 4 };

// High words of the largest |phi| as last tracked, of the boundary data and of
// the largest |fs| (device); track (FC_LAG, FC_NORM; optional) takes the largest interior
// |phi| read.
struct FcBounds {
  const unsigned *phi, *boundary, *fs;
  unsigned* track;
};

// Sweeps between two trackings for which the bounds hold (7-point 3, 13-point 2).
inline bool fx_sweeps_fit(int order, int nu) { return nu >= 1 && nu <= (order == 2 ? 3 : 2); }

// Partials that any pass over a level may write.
int fc_partials(const Dims& d);

// Levels that take these passes: fixed.cuh's fx_level, 13-point with equal spacings.
bool fc_level(const Dims& d, int order, const double h[3]);

// One pass over an FP64 level in the library's layout.  mode FC_SWEEP: colour
// `colour`, omega = 1, in place; FC_LAG: colour 0, out = the saved old values
// (skipped once st->done); FC_OPEN: colour 0, skipped once st->done, marks
// st->lag_pending; FC_RESID: out = delta; FC_NORM.  FC_LAG and FC_NORM
// write *nblocks partials {sum of delta^2, 0}.
cudaError_t launch_fc_pass(const Dims& d, int order, const double h[3], int mode, int colour, double* phi,
                           const double* fs, double* out, DevState* st, const FcBounds& b, double* partials, int* nblocks,
                           cudaStream_t s);

}  // namespace ps
