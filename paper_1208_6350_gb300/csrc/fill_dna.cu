// The fill kernels of 4-letter alphabets (a translation unit of its own: the
// instantiations compile in parallel).
#include "fill.cuh"

namespace gsw {

ClassGeom fill_geom_dna(int c, const FillLaunch &fl, int sms) { return tu_geom<true, false>(c, fl, sms); }

cudaError_t fill_launch_dna(int c, const FillLaunch &fl, const ClassGeom &g, cudaStream_t st) {
    return tu_launch<true, false>(c, fl, g, st);
}

}  // namespace gsw
