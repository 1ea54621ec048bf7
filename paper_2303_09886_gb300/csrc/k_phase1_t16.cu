// Phase-1 kernels for T = 16 taps (one translation unit per tap count so the
// instantiations compile in parallel).
#include "k_phase1.cuh"

namespace fe {
template cudaError_t launch_phase1_n1<16, 1>(int, int, const GroupArgs<Phase1Params, 1> *, cudaStream_t, bool);
template cudaError_t launch_phase1_n1<16, kMaxGroup>(int, int, const Phase1Group *, cudaStream_t, bool);
}  // namespace fe
