// The fill kernels of 4-letter alphabets (a translation unit of its own: the
// instantiations compile in parallel).
#include "fill.cuh"

namespace gsw {

cudaError_t launch_fill_dna(const FillLaunch &fl, int sms, int max_blocks, cudaStream_t st) {
    return launch_all<true>(fl, sms, max_blocks, st);
}

int fill_slots_dna(int A, int sms) { return max_slots<true>(A, sms); }

}  // namespace gsw
