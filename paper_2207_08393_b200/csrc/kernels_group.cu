// Instantiates the kernels of one group of transform lengths (compile with -DGLEAM_GROUP=<g>).
#include "size_ops.cuh"

namespace gleam {
#define GLEAM_SIZE(N, A0, A1, B0, B1, B2, LC) \
    extern const SizeOps size_ops_##N = {N, ZPlan<Plan<N, A0, A1>>::BFL, &SizeImpl<Plan<N, A0, A1>, Plan<N, B0, B1, B2>, LC>::row, \
                                         &SizeImpl<Plan<N, A0, A1>, Plan<N, B0, B1, B2>, LC>::col_z};
#include "sizes.def"
#undef GLEAM_SIZE
}  // namespace gleam
