// Host side of the staged colour passes of FP32 and BF16 levels (staged_sweeps.cu).
#pragma once
#include "ps_common.cuh"

namespace ps {

constexpr long long SS_MIN_NODES = 1000000;

// Levels that take the passes: 13-point, rows at 16-byte multiples (TMA), enough tiles.
bool colour_staged_level(const Dims& d, int order, int dt);

// One colour pass, omega = 1, in place: the bits of launch_sweep_colour's.  phi and
// fs 16-byte aligned; *fault is set when a copy did not land in time.
cudaError_t launch_colour_staged(const Dims& d, int order, const double h[3], int dt, int colour, void* phi,
                                 const void* fs, int* fault, cudaStream_t s);

}  // namespace ps
