// Instantiates passes 1 and 3 of the row-tile scheme (dc_tile.cuh) for one number RY of rows per block and every
// kz length (compile with -DGLEAM_TILE_RY=<RY>).
#include "dc_mid.cuh"

#ifndef GLEAM_TILE_RY
#error "compile with -DGLEAM_TILE_RY=<RY>"
#endif
#define GLEAM_CAT2(a, b) a##b
#define GLEAM_CAT(a, b) GLEAM_CAT2(a, b)

namespace gleam {

const TileOps* GLEAM_CAT(find_tile_, GLEAM_TILE_RY)(int n2) {
    switch (n2) {
#define GLEAM_SIZE(N, A0, A1, B0, B1, B2, LC)                                                              \
        case N: {                                                                                                  \
            static const TileOps ops = {GLEAM_TILE_RY, N, &TileImpl<Plan<N, A0, A1>, GLEAM_TILE_RY>::fwd,      \
                                        &TileImpl<Plan<N, A0, A1>, GLEAM_TILE_RY>::inv};                       \
            return &ops;                                                                                           \
        }
#include "sizes.def"
#undef GLEAM_SIZE
        default: return nullptr;
    }
}

}  // namespace gleam
