// The fill kernels of other alphabets (a translation unit of its own: the
// instantiations compile in parallel).
#include "fill.cuh"

namespace gsw {

cudaError_t launch_fill_general(const FillLaunch &fl, int sms, int max_blocks, cudaStream_t st) {
    return launch_all<false>(fl, sms, max_blocks, st);
}

int fill_slots_general(int A, int sms) { return max_slots<false>(A, sms); }

}  // namespace gsw
