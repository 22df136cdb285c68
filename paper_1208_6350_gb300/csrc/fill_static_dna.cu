// The allocation-free forward fill for 4-letter alphabets (fill_static.cuh).
#include "fill_static.cuh"

namespace gsw {

StaticGeom static_geom_dna(int alphabet) { return static_geom<true>(alphabet); }

cudaError_t static_setup_dna() { return static_setup<true>(); }

void static_launch_dna(bool rest, const BatchView &b, const Scoring &sc, uint8_t *scratch, const StaticGeom &g, int grid,
                       cudaStream_t st) {
    static_launch<true>(rest, b, sc, scratch, g, grid, st);
}

}  // namespace gsw
