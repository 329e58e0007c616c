// Instantiates the one-pass k-space part of 3-D problems with an arbitrary mask (dc_brick.cuh) for one group of readout
// lengths (compile with -DGLEAM_GROUP=<g>).
#include "dc_brick.cuh"

namespace gleam {
#define GLEAM_SIZE(N, A0, A1, B0, B1, B2, LC) \
    extern const BrickLaunch brick_##N = &BrickImpl<Plan<N, A0, A1>>::launch;
#include "sizes.def"
#undef GLEAM_SIZE
}  // namespace gleam
