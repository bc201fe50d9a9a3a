// Instances of the register-streaming adjoint step: F16 states.
#include "bte_adjoint_stream.cuh"

namespace bte {
namespace adjs {
cudaError_t launch_f16(const StepArgs &a, const AdjStreamArgs &g, int limiter, cudaStream_t s) {
    return launch_storage<kStoreF16>(a, g, limiter, s);
}
}  // namespace adjs
}  // namespace bte
