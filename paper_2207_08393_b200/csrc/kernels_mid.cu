// Instantiates the middle pass of the row-tile scheme (dc_mid.cuh) for one group of ky lengths (compile with
// -DGLEAM_GROUP=<g>): two-stage lengths split as their row plan, the others have a single row per block of passes 1, 3.
#include "dc_mid.cuh"

namespace gleam {
#define GLEAM_SIZE(N, A0, A1, B0, B1, B2, LC) \
    extern const MidOps mid_ops_##N = {N, A1 > 1 ? A0 : 1, A1 > 1 ? A1 : A0, &MidImpl<(A1 > 1 ? A0 : 1), (A1 > 1 ? A1 : A0)>::launch};
#include "sizes.def"
#undef GLEAM_SIZE
}  // namespace gleam
