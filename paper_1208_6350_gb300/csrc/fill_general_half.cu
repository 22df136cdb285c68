// The fill kernels of other alphabets, half-precision clamp (a translation unit of its own: the
// instantiations compile in parallel).
#include "fill.cuh"

namespace gsw {

ClassGeom fill_geom_general_half(int c, const FillLaunch &fl, int sms) { return tu_geom<false, true>(c, fl, sms); }

cudaError_t fill_launch_general_half(int c, const FillLaunch &fl, const ClassGeom &g, cudaStream_t st) {
    return tu_launch<false, true>(c, fl, g, st);
}

}  // namespace gsw
