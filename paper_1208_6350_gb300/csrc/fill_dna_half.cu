// The fill kernels of 4-letter alphabets, half-precision clamp (a translation unit of its own: the
// instantiations compile in parallel).
#include "fill.cuh"

namespace gsw {

ClassGeom fill_geom_dna_half(int c, const FillLaunch &fl, int sms) { return tu_geom<true, true>(c, fl, sms); }

cudaError_t fill_launch_dna_half(int c, const FillLaunch &fl, const ClassGeom &g, cudaStream_t st) {
    return tu_launch<true, true>(c, fl, g, st);
}

}  // namespace gsw
