// Pruned scale-search kernels, instantiated for bf16 input.
#include "mxq_pruned.cuh"

namespace mxq {
cudaError_t launch_brute_pruned_bf16(const QuantArgs& a, int B, int fmt, cudaStream_t s) {
    return launch_pruned_dt<kBF16>(a, B, fmt, s);
}
}  // namespace mxq
