// Pruned scale-search kernels, instantiated for fp32 input.
#include "mxq_pruned.cuh"

namespace mxq {
cudaError_t launch_brute_pruned_f32(const QuantArgs& a, int B, int fmt, cudaStream_t s) {
    return launch_pruned_dt<kF32>(a, B, fmt, s);
}
}  // namespace mxq
