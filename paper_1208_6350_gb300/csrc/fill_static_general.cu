// The allocation-free forward fill for general alphabets (fill_static.cuh).
#include "fill_static.cuh"

namespace gsw {

StaticGeom static_geom_general(int alphabet) { return static_geom<false>(alphabet); }

cudaError_t static_setup_general() { return static_setup<false>(); }

void static_launch_general(bool rest, const BatchView &b, const Scoring &sc, uint8_t *scratch, const StaticGeom &g, int grid,
                       cudaStream_t st) {
    static_launch<false>(rest, b, sc, scratch, g, grid, st);
}

}  // namespace gsw
