// Instantiates the readout pass of 3-D problems with an arbitrary mask (dc_axis.cuh) for one group of lengths (compile
// with -DGLEAM_GROUP=<g>).
#include "dc_axis.cuh"

namespace gleam {
#define GLEAM_SIZE(N, A0, A1, B0, B1, B2, LC) \
    extern const AxisOps axis_ops_##N = {N, &AxisImpl<Plan<N, A0, A1>>::launch};
#include "sizes.def"
#undef GLEAM_SIZE
}  // namespace gleam
